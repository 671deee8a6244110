// Chunkwise HGRN2 forward on the Blackwell tensor cores (tcgen05 + TMEM + TMA), bf16 I/O, fp32
// state, d_k = d_v = 128, chunk length C = 64.  A CTA walks the chunks of a (batch, head) unit, or of a segment of one,
// in order with the running state resident in tensor memory (frame and formulas: tc_chunk.cuh); where those are many
// and short it then takes another one without draining its pipelines (work items: tc_chunk.cuh).
//
// Warp roles (none of them ever waits on a CTA-wide barrier inside the chunk loop; every stretch of
// work between two hand-offs is latency-bound, so the roles are many and narrow rather than few and
// wide, and their loops stay rolled to keep the instruction footprint small):
//   T   transform warps (4 per group): raw o, f tiles -> Qs, Ks in place, running ahead of the rest
//       by up to two chunks (three TMA stages);
//   E1  8 state warps: rescale the accumulator once per chunk (the critical chain) and publish its
//       bf16 copy S' for Y = Qs S' and for the saved-state store;
//   E2  4 output warps: causal mask of A into an operand slab, Y into a staging tile;
//   L   1 warp: TMA loads of o, f, i;
//   MS  1 warp: tcgen05.mma issue of A = Qs Ks^T and of the state update S' += Ks^T V, then the TMA store of
//       S' (the saved chunk state) straight from the operand copy;
//   MY  1 warp: tcgen05.mma issue of Y = Qs S', Y += tril(A) V;
//   ST  1 warp: TMA stores of the Y tiles.
// Hand-offs are mbarriers; every wait is bounded (tc_common.cuh).
//
// Tensor-memory plan (512 columns): S' at [0,128) (lane = key dim, column = value dim); Y, double
// buffered, at [128,384) and A, double buffered, at [384,512) in the M = 64 accumulator layout
// (row r -> lane 32 * (r / 16) + r % 16).
#include <atomic>

#include "chunk_alu.cuh"
#include "tc_chunk.cuh"

namespace hgrn2 {

namespace {

using namespace tc;

constexpr int kTGroups = 1, kTWarps = 4 * kTGroups;
constexpr int kE1Warps = 8, kE2Warps = 4;
constexpr int kE1Threads = kE1Warps * 32, kE2Threads = kE2Warps * 32;
constexpr int kWarpE1 = kTWarps, kWarpE2 = kWarpE1 + kE1Warps;
constexpr int kWarpLoad = kWarpE2 + kE2Warps, kWarpMmaS = kWarpLoad + 1, kWarpMmaY = kWarpLoad + 2,
              kWarpStore = kWarpLoad + 3;
constexpr int kThreads = (kWarpStore + 1) * 32;
static_assert(kWarpE1 % 4 == 0 && kWarpE2 % 4 == 0, "epilogue warps must start on a TMEM lane-quarter boundary");

constexpr int kStages = 3;
constexpr uint32_t kStageBytes = 3 * kTile;                       // q, f, v
constexpr uint32_t kOffS = kStages * kStageBytes;                 // bf16 copy of S'
constexpr uint32_t kOffP = kOffS + kStateTile;                    // bf16 tril(A): two slabs (double buffer)
constexpr uint32_t kOffY = kOffP + 2 * kSlab;                     // Y staging tile for the TMA store
constexpr uint32_t kOffPm = kOffY + kTile;                        // float pm[4][128]
constexpr uint32_t kOffE = kOffPm + 4 * 128 * 4;                  // float ee[4][128]
constexpr uint32_t kOffCtl = kOffE + 4 * 128 * 4;
constexpr uint32_t kSmemBytes = kOffCtl + 768 + 1024;             // + alignment slack

constexpr uint32_t kColS = 0, kColY = 128, kColA = 384;

struct Ctl {
    uint64_t fullqf[kStages];    // TMA (o, f tiles) -> T
    uint64_t full[kStages];      // TMA (i tile) -> MS, MY
    uint64_t emptyqf[kStages];   // tcgen05.commit (MS and MY) -> L: every MMA reading Qs, Ks of the stage has completed
    uint64_t emptyv[kStages];    // tcgen05.commit (MS and MY) -> L: every MMA reading V of the stage has completed
    uint64_t t_done[kStages];    // T -> MS, MY, E1 (Pm, E of the chunk)
    uint64_t m_tmem;             // E1 -> MS: the accumulator holds S' of the chunk
    uint64_t m_done;             // E1 -> MY: the bf16 copy of S' is in shared memory
    uint64_t barS;               // tcgen05.commit -> E1: state update complete
    uint64_t barS2;              // tcgen05.commit (MY) + MS -> E1: Y = Qs S' complete, S' stored: copy reusable
    uint64_t barA[2];            // tcgen05.commit -> E2: A is complete
    uint64_t p_ready[2];         // E2 -> MY: tril(A) is in shared memory
    uint64_t barY[2];            // tcgen05.commit -> E2: Y is complete
    uint64_t y_tfree[2];         // E2 -> MY: the Y accumulator has been read out
    uint64_t y_staged;           // E2 -> ST
    uint64_t y_sfree;            // ST -> E2: the staging tile may be overwritten
    uint64_t drain;              // tcgen05.commit (MS and MY, after their loops): every product issued has completed
    alignas(16) ItemRing ring;
    int abort_flag;              // set by the first wait that runs out: every later wait returns at once
    uint32_t tmem_base;
    int exact_flag;              // E1: a decay of this CTA's tokens left the range of the rescaled operands
    int l_qf, l_v;               // L: chunks whose o, f tiles (i tile) have been asked for, for the abort epilogue
    int claimed;                 // redo_claim's answer
};
static_assert(sizeof(Ctl) <= 768, "control block");
static_assert(kSmemBytes <= 232448, "shared memory budget");

constexpr int kExactC = 32;      // chunk length of the exact fp32 routines at d = 128 (their shared-memory budget)
static_assert(alu::fwd_smem_floats(kD, kD, kExactC) * sizeof(float) <= kSmemBytes - 1024, "exact path fits the CTA's shared memory");

constexpr int kRingWarps = kTWarps + kE1Warps + kE2Warps + 3;    // readers of the item ring: T, E1, E2, MS, MY, ST

// kRagged: sequences need not be whole chunks (a partial chunk is padded with neutral tokens), and a packed batch is one.
// kEnc: the f tensor holds k = 1 - f (see transform_half).  kPersist: several items per CTA (tc_chunk.cuh).
template <bool kRagged, bool kEnc, bool kPersist>
__global__ void __launch_bounds__(kThreads, 1)
tc_fwd_kernel(const __grid_constant__ CUtensorMap map_o, const __grid_constant__ CUtensorMap map_f,
              const __grid_constant__ CUtensorMap map_i, const __grid_constant__ CUtensorMap map_y,
              const __grid_constant__ CUtensorMap map_saved, const float *S0, const float *chain,
              int *__restrict__ redo, float *__restrict__ SN, float *__restrict__ totals, int want_y, int want_saved,
              const __grid_constant__ WorkArgs wk, StatusBlock *status, int clear_status, const ExactArgs ex,
              int start_aborted)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *sbuf = smem + kOffS;
    uint8_t *pbuf = smem + kOffP;
    uint8_t *ybuf = smem + kOffY;
    float *pm = reinterpret_cast<float *>(smem + kOffPm);
    float *ee = reinterpret_cast<float *>(smem + kOffE);
    Ctl *ctl = reinterpret_cast<Ctl *>(smem + kOffCtl);
    volatile int *abort_flag = &ctl->abort_flag;

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&ctl->fullqf[s], 1);
            mbar_init(&ctl->full[s], 1);
            mbar_init(&ctl->emptyqf[s], 2);
            mbar_init(&ctl->emptyv[s], 2);
            mbar_init(&ctl->t_done[s], kTransformThreads);
        }
        mbar_init(&ctl->m_tmem, kE1Threads);
        mbar_init(&ctl->m_done, kE1Threads);
        mbar_init(&ctl->barS, 1);
        mbar_init(&ctl->barS2, 2);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&ctl->barA[b], 1);
            mbar_init(&ctl->p_ready[b], kE2Threads);
            mbar_init(&ctl->barY[b], 1);
            mbar_init(&ctl->y_tfree[b], kE2Threads);
        }
        mbar_init(&ctl->y_staged, kE2Threads);
        mbar_init(&ctl->y_sfree, 1);
        mbar_init(&ctl->drain, 2);
        ctl->abort_flag = start_aborted;
        ctl->exact_flag = 0;
        ctl->l_qf = 0;
        ctl->l_v = 0;
        ring_init(ctl->ring, kRingWarps);
        fence_barrier_init();
        tma_prefetch_desc(&map_o);
        tma_prefetch_desc(&map_f);
        tma_prefetch_desc(&map_i);
        tma_prefetch_desc(&map_y);
        tma_prefetch_desc(&map_saved);
    }
    if (warp == 0) tmem_alloc(&ctl->tmem_base, kTmemCols);
    chain_wait();
    if (clear_status && blockIdx.x == 0) begin_call(status, kRagged ? wk.cu : nullptr, wk.B, wk.N);
    const Item first = warp_uniform(work_item<kRagged>(wk, blockIdx.x));
    if (kPersist && tid == 0) {
        ctl->ring.item[0] = first;
        if (first.chain >= 0) ctl->ring.cuts[ctl->ring.n_cuts++] = first.id;
        mbar_arrive(&ctl->ring.full[0]);
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = ctl->tmem_base;
    const int sub = warp & 3;                                        // TMEM lane quarter of this warp
    const uint32_t lane_base = static_cast<uint32_t>(32 * sub) << 16;

    if (warp < kTWarps) {
        // ================= T: transform =================
        PT_DECL
        const int tt = tid & (kTransformThreads - 1);
        int g = 0;                                                   // chunks so far, over all items
        Item it;
        for (int k = 0; next_item<kPersist>(&ctl->ring, k, abort_flag, first, it); ++k) {
            float *tg = totals ? totals + (size_t)it.slot0 * 2 * kD : nullptr;   // Pm, E of every chunk for the backward
            for (int left = it.n; left > 0; left -= kC, ++g) {
                const int s = g % kStages;
                uint8_t *qbuf = smem + s * kStageBytes;
                mbar_wait(&ctl->fullqf[s], (g / kStages) & 1, abort_flag);
                PT_MARK(0)
                if (kRagged && left < kC) neutral_rows<kEnc>(qbuf, qbuf + kTile, left, tt);
                transform_stream<kEnc>(qbuf, qbuf + kTile, pm + (g & 3) * 128, ee + (g & 3) * 128, tg, tg ? tg + kD : nullptr, tt);
                if (tg) tg += 2 * kD;
                fence_proxy_async_smem();
                mbar_arrive(&ctl->t_done[s]);
                PT_MARK(1)
            }
        }
        PT_DUMP(status, 0, 2, tid == 0)
    } else if (warp < kWarpE2) {
        // ================= E1: state warps =================
        const int half = (warp - kWarpE1) >> 2;                      // column half [64 * half, 64 * half + 64)
        const int krow = 32 * sub + lane;
        const int v0 = 64 * half;
        int g = 0;
        PT_DECL
        Item it;
        for (int k = 0; next_item<kPersist>(&ctl->ring, k, abort_flag, first, it); ++k) {
            const int n = it.n;
            const size_t row = ((size_t)it.unit * kD + krow) * kD + v0;
            float e_prev = 1.f;
            // the accumulator starts as the initial state, so the loop over the chunks has no first-chunk case of its own
            if (n > 0) {
                const float *init = it.chain >= 0 ? chain + ((size_t)it.chain * kD + krow) * kD + v0 : (S0 ? S0 + row : nullptr);
#pragma unroll 1
                for (int part = 0; part < 2; ++part) {
                    uint32_t r[32];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float4 x = init ? reinterpret_cast<const float4 *>(init + 32 * part)[j] : make_float4(0.f, 0.f, 0.f, 0.f);
                        r[4 * j + 0] = __float_as_uint(x.x); r[4 * j + 1] = __float_as_uint(x.y);
                        r[4 * j + 2] = __float_as_uint(x.z); r[4 * j + 3] = __float_as_uint(x.w);
                    }
                    tmem_st32(tmem + lane_base + kColS + v0 + 32 * part, r);
                }
                tmem_wait_st();
            }
            for (int left = n; left > 0; left -= kC, ++g) {
                // S' = (E_prev Pm) S'' (S'' = the accumulator) back into TMEM
                mbar_wait(&ctl->t_done[g % kStages], (g / kStages) & 1, abort_flag);
                PT_MARK(0)
                const float pm_c = pm[(g & 3) * 128 + krow];
                const float e_old = e_prev;
                const float factor = e_prev * pm_c;
                e_prev = ee[(g & 3) * 128 + krow];
                // a total on the floor: the decay across that half chunk is more than the rescaled operands can carry
                if (fminf(pm_c, e_prev) <= kProdFloor) {
                    ctl->exact_flag = 1;
                    if (kPersist) ctl->ring.flagged[k & 7] = it.id + 1;
                }
                uint32_t r[64];
                if (g > 0) mbar_wait(&ctl->barS, (g - 1) & 1, abort_flag);
                PT_MARK(1)
                tc_fence_after_sync();
                tmem_ld32(tmem + lane_base + kColS + v0, *reinterpret_cast<uint32_t(*)[32]>(r));
                tmem_ld32(tmem + lane_base + kColS + v0 + 32, *reinterpret_cast<uint32_t(*)[32]>(r + 32));
                tmem_wait_ld();
                // Each of the two decays is above the floor, but their product can leave fp32's range although the
                // accumulator, which sits in the previous chunk's frame, is as large as that decay is small: then the
                // two are applied one after the other (key dimensions whose decay over those 64 tokens is below
                // 2^-120: rare).  One loop for both cases: the roles' code together is about what the instruction
                // cache holds, and a second unrolled copy here cost up to 5 % (the first one alone: 73 -> 72 us).
                const bool safe = factor >= kFactorSafe;
                float f1 = safe ? factor : e_old;
#pragma unroll 1
                for (int more = safe ? 0 : 1; more >= 0; --more, f1 = pm_c)
#pragma unroll
                    for (int j = 0; j < 64; j += 2) scale2(r[j], r[j + 1], f1);
                tmem_st32(tmem + lane_base + kColS + v0, *reinterpret_cast<uint32_t(*)[32]>(r));
                tmem_st32(tmem + lane_base + kColS + v0 + 32, *reinterpret_cast<uint32_t(*)[32]>(r + 32));
                uint4 sw[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) sw[j] = pack8(r + 8 * j);
                tmem_wait_st();
                tc_fence_before_sync();
                mbar_arrive(&ctl->m_tmem);
                PT_MARK(2)
                // its bf16 copy, once Y = Qs S' of the previous chunk no longer reads the old one
                if (g >= 1) mbar_wait(&ctl->barS2, (g - 1) & 1, abort_flag);
                PT_MARK(3)
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    *reinterpret_cast<uint4 *>(sbuf + half * kStateSlab + slab_chunk_off(krow, j)) = sw[j];
                fence_proxy_async_smem();
                mbar_arrive(&ctl->m_done);
                PT_MARK(4)
            }
            // S_N = Diag(E_last) S''; without tokens the state passes through.  The accumulator is free for the next item
            // behind this in any case.
            if (n > 0) {
                mbar_wait(&ctl->barS, (g - 1) & 1, abort_flag);
                tc_fence_after_sync();
            }
            if (SN != nullptr && it.last) {
#pragma unroll 1
                for (int part = 0; part < 2; ++part) {
                    uint32_t r[32];
                    float4 *dst = reinterpret_cast<float4 *>(SN + row + 32 * part);
                    if (n > 0) {
                        tmem_ld32(tmem + lane_base + kColS + v0 + 32 * part, r);
                        tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            dst[j] = make_float4(__uint_as_float(r[4 * j + 0]) * e_prev, __uint_as_float(r[4 * j + 1]) * e_prev,
                                                 __uint_as_float(r[4 * j + 2]) * e_prev, __uint_as_float(r[4 * j + 3]) * e_prev);
                    } else {
#pragma unroll 1
                        for (int j = 0; j < 8; ++j)
                            dst[j] = S0 ? reinterpret_cast<const float4 *>(S0 + row + 32 * part)[j] : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
            }
        }
        PT_DUMP(status, 2, 5, tid == kWarpE1 * 32)
    } else if (warp < kWarpLoad) {
        // ================= E2: output warps =================
        const int t = 16 * sub + lane;                               // accumulator row of lanes 0..15
        PT_DECL
        // A step: tril(A(g)) -> operand slab | Y(g-1) -> staging tile.  Y(g-1) is not held back over an item without tokens:
        // the store warp cannot give its item up before it has the tile, and no item kRing further on is published before
        // it has, so this role would wait for an item that waits for this role.
        int left = 0;
        bool more = true, held = false;                              // held: Y(g-1) is still to be staged
        for (int g = 0, k = 0; more;) {
            if (left == 0) {
                Item it;
                more = next_item<kPersist>(&ctl->ring, k++, abort_flag, first, it);
                left = more && want_y ? (it.n + kC - 1) / kC : 0;
            }
            const bool chunk = left > 0;
            if (chunk) {
                const int b = g & 1;
                mbar_wait(&ctl->barA[b], (g >> 1) & 1, abort_flag);
                PT_MARK(0)
                tc_fence_after_sync();
#pragma unroll 1
                for (int h = 0; h < 2; ++h)
                    tril_to_slab(tmem + lane_base + kColA + 64 * b + 32 * h, pbuf + b * kSlab, sub, h, lane);
                fence_proxy_async_smem();
                tc_fence_before_sync();
                mbar_arrive(&ctl->p_ready[b]);
                PT_MARK(1)
            }
            if (held) {
                const int b = (g - 1) & 1;
                mbar_wait(&ctl->barY[b], ((g - 1) >> 1) & 1, abort_flag);
                PT_MARK(2)
                tc_fence_after_sync();
                if (g >= 2) mbar_wait(&ctl->y_sfree, (g - 2) & 1, abort_flag);
                PT_MARK(3)
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
                    uint32_t r[64];
                    const uint32_t ta = tmem + lane_base + kColY + 128 * b + 64 * h;
                    tmem_ld32(ta, *reinterpret_cast<uint32_t(*)[32]>(r));
                    tmem_ld32(ta + 32, *reinterpret_cast<uint32_t(*)[32]>(r + 32));
                    tmem_wait_ld();
                    if (lane < 16) {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            *reinterpret_cast<uint4 *>(ybuf + h * kSlab + slab_chunk_off(t, j)) = pack8(r + 8 * j);
                    }
                }
                tc_fence_before_sync();
                mbar_arrive(&ctl->y_tfree[b]);
                fence_proxy_async_smem();
                mbar_arrive(&ctl->y_staged);
                PT_MARK(4)
            }
            held = chunk;
            if (chunk) {
                ++g;
                --left;
            }
        }
        PT_DUMP(status, 7, 5, tid == kWarpE2 * 32)
    } else if (warp == kWarpLoad) {
        // ================= L: TMA loads =================
        int g = 0;                                               // chunks whose tiles have been asked for
        // A barrier must never be armed twice within one phase.  Normally the stage's previous fill has long
        // been consumed when its empty barrier completes; on the time-out exit that wait returns at once, so
        // the previous fill is waited for explicitly (one poll that succeeds at once in normal running;
        // stopping this lane on the wait's return value instead cost 8 %).
        Item it = first;
        for (int k = 0; it.id >= 0; ++k) {
            const int nc = (it.n + kC - 1) / kC, plane = it.plane;
            int row = it.row0;
            bool asked = false;
            for (int c = 0; c < nc; ++c, ++g, row += kC) {
                const int s = g % kStages;
                uint8_t *st = smem + s * kStageBytes;
                // o and f have barriers of their own in both directions: the transform, which paces the kernel,
                // needs only them, and their tiles are free as soon as Y = Qs S' of the chunk three back is done,
                // well before its last product Y += P V has read V
                if (g >= kStages) {
                    mbar_wait(&ctl->emptyqf[s], ((g / kStages) - 1) & 1, abort_flag);
                    mbar_wait_drain(&ctl->fullqf[s], ((g / kStages) - 1) & 1, 20000000ull);
                }
                // the next chunk's o, f tiles are asked into L2 now: their load can be issued only when their stage
                // frees, one chunk from now, and then finds them there (measured on the fwd + bwd step: -1 %; two
                // chunks ahead, or including the v tile, gave nothing)
                if (c + 1 < nc)
                    for (int b = 0; b < 2; ++b) {
                        tma_prefetch_3d(&map_o, 64 * b, row + kC, plane);
                        tma_prefetch_3d(&map_f, 64 * b, row + kC, plane);
                    }
                mbar_arrive_expect_tx(&ctl->fullqf[s], 2 * kTile);
                for (int b = 0; b < 2; ++b) {
                    tma_load_3d(st + b * kSlab, &map_o, &ctl->fullqf[s], 64 * b, row, plane);
                    tma_load_3d(st + kTile + b * kSlab, &map_f, &ctl->fullqf[s], 64 * b, row, plane);
                }
                ctl->l_qf = g + 1;
                // the next item is asked for as this one's last tiles are: the answer takes about a microsecond
                if (kPersist && (c + 2 == nc || nc == 1)) asked = ring_ask(&ctl->ring, k + 1, &ctl->exact_flag, abort_flag);
                if (g >= kStages) {
                    mbar_wait(&ctl->emptyv[s], ((g / kStages) - 1) & 1, abort_flag);
                    mbar_wait_drain(&ctl->full[s], ((g / kStages) - 1) & 1, 20000000ull);
                }
                mbar_arrive_expect_tx(&ctl->full[s], kTile);
                for (int b = 0; b < 2; ++b)
                    tma_load_3d(st + 2 * kTile + b * kSlab, &map_i, &ctl->full[s], 64 * b, row, plane);
                ctl->l_v = g + 1;
            }
            if (!kPersist) break;
            if (nc == 0) asked = ring_ask(&ctl->ring, k + 1, &ctl->exact_flag, abort_flag);
            it = warp_uniform(*ring_take<kRagged>(&ctl->ring, k + 1, asked, wk, abort_flag));
        }
    } else if (warp == kWarpMmaS) {
        // ================= MS: state update =================
        constexpr uint32_t idescS = idesc_bf16(128, 128, 1, 1);    // Ks^T (MN-major) x V (MN-major)
        // Descriptors are formed once; a K step or a stage change only adds to the 14-bit
        // start-address field (addresses are in 16-byte units and stay below 2^14).
        const uint64_t dfm0 = smem_desc_sw128(smem_u32(smem) + kTile, kSlab, 1024);      // Ks, MN-major
        const uint64_t dvm0 = smem_desc_sw128(smem_u32(smem) + 2 * kTile, kSlab, 1024);  // V, MN-major
        constexpr uint32_t idescA = idesc_bf16(64, 64, 0, 0);      // Qs (K-major) x Ks (K-major)
        const uint64_t dq0 = smem_desc_sw128(smem_u32(smem), 16, 1024);                  // Qs, K-major
        const uint64_t dfk0 = smem_desc_sw128(smem_u32(smem) + kTile, 16, 1024);         // Ks, K-major
        auto kmaj = [](int kk) { return (uint64_t)(((kk >> 2) * kSlab + (kk & 3) * 32) >> 4); };
        PT_DECL
        int g = 0;
        Item it;
        for (int k = 0; next_item<kPersist>(&ctl->ring, k, abort_flag, first, it); ++k) {
            int slot = it.slot0;
            for (int left = it.n; left > 0; left -= kC, ++g, ++slot) {
                const int s = g % kStages;
                const uint64_t so = (uint64_t)s * (kStageBytes >> 4);
                mbar_wait(&ctl->full[s], (g / kStages) & 1, abort_flag);
                mbar_wait(&ctl->t_done[s], (g / kStages) & 1, abort_flag);
                PT_MARK(0)
                // A = Qs Ks^T is issued here, not by the lane of the other output products: this lane has nothing
                // to do until the state is rescaled, and every tcgen05.mma also costs the issuing lane's scheduler
                // (shared with a transform warp) issue time, so the products are spread over two schedulers
                if (want_y) {
                    const int b = g & 1;
                    if (g >= 2) {                                    // tril(A) of chunk g - 2 has left this buffer
                        mbar_wait(&ctl->p_ready[b], ((g - 2) >> 1) & 1, abort_flag);
                        tc_fence_after_sync();
                    }
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        mma_bf16_ss(tmem + kColA + 64 * b, dq0 + so + kmaj(kk), dfk0 + so + kmaj(kk), idescA, kk > 0);
                    mma_commit(&ctl->barA[b]);
                }
                mbar_wait(&ctl->m_tmem, g & 1, abort_flag);
                PT_MARK(1)
                tc_fence_after_sync();
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)              // S' += Ks^T V
                    mma_bf16_ss(tmem + kColS, dfm0 + so + (uint64_t)(kk * 128), dvm0 + so + (uint64_t)(kk * 128),
                                idescS, 1);
                mma_commit(&ctl->barS);
                mma_commit(&ctl->emptyqf[s]);
                mma_commit(&ctl->emptyv[s]);
                PT_MARK(2)
                // the saved chunk state, straight from the operand copy of S' (this lane is idle until the next
                // chunk's state is ready; in the lane that issues the outputs' products the wait for the store
                // to have read 32 KB would hold those up)
                mbar_wait(&ctl->m_done, g & 1, abort_flag);
                if (lane == 0) {
                    if (want_saved) {
                        tma_store_3d(&map_saved, sbuf, 0, 0, slot);
                        tma_store_3d(&map_saved, sbuf + kStateSlab, 64, 0, slot);
                        tma_store_commit();
                        tma_store_wait_read();
                    }
                    mbar_arrive(&ctl->barS2);                   // second arrival: the tcgen05.commit of Y = Qs S'
                }
                __syncwarp();
            }
        }
        PT_DUMP(status, 12, 3, true)
        if (want_saved && lane == 0) tma_store_wait_all();
        mma_commit(&ctl->drain);
    } else if (warp == kWarpMmaY) {
        // ================= MY: outputs (+ saved-state stores) =================
        constexpr uint32_t idescY = idesc_bf16(64, 128, 0, 1);     // Qs or P (K-major) x S' or V (MN-major)
        const uint64_t dq0 = smem_desc_sw128(smem_u32(smem), 16, 1024);                  // Qs, K-major
        const uint64_t dvm0 = smem_desc_sw128(smem_u32(smem) + 2 * kTile, kSlab, 1024);  // V, MN-major
        const uint64_t dsm = smem_desc_sw128(smem_u32(sbuf), kStateSlab, 1024);          // S', MN-major
        const uint64_t dp0 = smem_desc_sw128(smem_u32(pbuf), 16, 1024);                  // tril(A), K-major
        auto kmaj = [](int kk) { return (uint64_t)(((kk >> 2) * kSlab + (kk & 3) * 32) >> 4); };
        PT_DECL
        int g = 0;
        Item it;
        for (int k = 0; next_item<kPersist>(&ctl->ring, k, abort_flag, first, it); ++k) {
            for (int left = it.n; left > 0; left -= kC, ++g) {
                const int s = g % kStages, b = g & 1;
                const uint64_t so = (uint64_t)s * (kStageBytes >> 4);
                const uint64_t dq = dq0 + so, dvm = dvm0 + so;
                const uint64_t dp = dp0 + (uint64_t)b * (kSlab >> 4);
                const uint32_t ty = tmem + kColY + 128 * b;
                mbar_wait(&ctl->full[s], (g / kStages) & 1, abort_flag);
                mbar_wait(&ctl->t_done[s], (g / kStages) & 1, abort_flag);
                PT_MARK(0)
                mbar_wait(&ctl->m_done, g & 1, abort_flag);
                PT_MARK(1)
                if (want_y) {
                    if (g >= 2) {
                        mbar_wait(&ctl->y_tfree[b], ((g - 2) >> 1) & 1, abort_flag);
                        tc_fence_after_sync();
                    }
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)          // Y = Qs S'
                        mma_bf16_ss(ty, dq + kmaj(kk), dsm + (uint64_t)(kk * 128), idescY, kk > 0);
                }
                PT_MARK(2)
                mma_commit(&ctl->barS2);
                mma_commit(&ctl->emptyqf[s]);               // A and Y = Qs S' were the last readers of Qs, Ks here
                if (want_y) {
                    mbar_wait(&ctl->p_ready[b], (g >> 1) & 1, abort_flag);
                    PT_MARK(3)
                    tc_fence_after_sync();
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)          // Y += P V
                        mma_bf16_ss(ty, dp + (uint64_t)(kk * 2), dvm + (uint64_t)(kk * 128), idescY, 1);
                    mma_commit(&ctl->barY[b]);
                }
                mma_commit(&ctl->emptyv[s]);
                PT_MARK(4)
            }
        }
        PT_DUMP(status, 15, 5, true)
        mma_commit(&ctl->drain);
    } else {
        // ================= ST: Y stores =================
        // In a packed batch the rows after a sequence's last token belong to the next sequence (a tile store
        // would overwrite them; past the end of an ordinary tensor it simply drops them), so the partial last
        // chunk of a packed sequence is stored row by row, by the whole warp.
        int g = 0;
        Item it;
        for (int k = 0; next_item<kPersist>(&ctl->ring, k, abort_flag, first, it); ++k) {
            int row = it.row0;
            for (int left = want_y ? it.n : 0; left > 0; left -= kC, ++g, row += kC) {
                mbar_wait(&ctl->y_staged, g & 1, abort_flag);
                if (!kRagged || wk.cu == nullptr || left >= kC) {
                    if (lane == 0) {
                        tma_store_3d(&map_y, ybuf, 0, row, it.plane);
                        tma_store_3d(&map_y, ybuf + kSlab, 64, row, it.plane);
                        tma_store_commit();
                        tma_store_wait_read();
                    }
                } else {
                    uint4 *dst = reinterpret_cast<uint4 *>(ex.y + ((size_t)it.plane * wk.N + row) * kD);
                    for (int x = lane; x < left * 16; x += 32) {             // 16-byte pieces: row, slab, chunk
                        const int r = x >> 4, h = (x >> 3) & 1, j = x & 7;
                        dst[(size_t)r * 16 + h * 8 + j] = *reinterpret_cast<const uint4 *>(ybuf + h * kSlab + slab_chunk_off(r, j));
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&ctl->y_sfree);
            }
        }
        if (lane == 0) tma_store_wait_all();
    }
    tc_fence_before_sync();
    __syncthreads();
    if (tid == 0) {
        // Nothing may be in flight when the CTA gives up its tensor and shared memory.  The two issuing lanes
        // committed once more after their loops: that barrier completes when every product they issued has.
        mbar_wait_drain(&ctl->drain, 0, 20000000ull);
        if (*abort_flag) {
            report_error(status, HGRN2_ERR_TIMEOUT, 1);
            if (kPersist && ctl->ring.asked > 0) mbar_wait_drain(&ctl->ring.answered, (ctl->ring.asked - 1) & 1, 20000000ull);
            // tiles asked for but never consumed may still be on their way into this CTA's shared memory
            for (int s = 0; s < kStages; ++s) {
                const int nq = ctl->l_qf, nv = ctl->l_v;
                if (nq > s) mbar_wait_drain(&ctl->fullqf[s], (((nq - 1 - s) / kStages)) & 1, 20000000ull);
                if (nv > s) mbar_wait_drain(&ctl->full[s], (((nv - 1 - s) / kStages)) & 1, 20000000ull);
            }
        }
    }
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);

    // ---- exact path: the sweep met a decay its operands cannot represent, so the item - or, for segments of whole chunks,
    // the unit (redo_claim) - is redone, from its inputs and the state it started from, by the pairwise-safe fp32
    // routine (every output of it is overwritten)
    if (ex.o == nullptr || *abort_flag) return;
    const bool units = !kRagged && redo != nullptr;                  // there are segments of whole chunks
    const int listed = kPersist ? 8 : 1, cuts = !units ? 0 : kPersist ? ctl->ring.n_cuts : first.chain >= 0 ? 1 : 0;
    for (int j = ctl->exact_flag ? 0 : listed; j < listed + cuts; ++j) {
        const bool claim = j >= listed;                              // flagged items, then the claims
        const int id = kPersist ? (claim ? ctl->ring.cuts[j - listed] : ctl->ring.flagged[j] - 1) : first.id;
        bool go = id >= 0 && !(units && id >= wk.main);
        if (claim) {
            if (tid == 0)
                ctl->claimed = redo_claim(redo + 2 * ((id - wk.main) % wk.tail),
                                          kPersist ? ring_flagged(ctl->ring, id) : ctl->exact_flag != 0, wk.G);
            __syncthreads();
            go = ctl->claimed != 0;
        }
        if (go) {
            if (tid == 0) atomicAdd(&status->exact_units, 1);
            const Item it = claim ? cut_unit(wk, id, 0) : work_item<kRagged>(wk, id);
            const size_t seq = ((size_t)it.plane * wk.N + it.row0) * kD, st = (size_t)it.unit * kD * kD;
            alu::fwd_unit<__nv_bfloat16, __nv_bfloat16, kEnc ? alu::kGateEnc : alu::kGateIsF>(
                reinterpret_cast<float *>(smem), ex.o + seq, ex.f + seq, ex.i + seq,
                it.chain >= 0 ? chain + (size_t)it.chain * kD * kD : (S0 ? S0 + st : nullptr), ex.y ? ex.y + seq : nullptr,
                SN != nullptr && it.last ? SN + st : nullptr, ex.states ? ex.states + (size_t)it.slot0 * kD * kD : nullptr,
                kC / kExactC, it.n, kD, kD, kExactC, (it.n + kExactC - 1) / kExactC);
        }
        __syncthreads();                                             // the routine's shared memory, and the answer, are free
    }
}

}  // namespace

bool tc_supported(const hgrn2_desc *d)
{
    return d->io == HGRN2_BF16 && d->dk == kD && d->dv == kD;
}
int  tc_default_chunk() { return kC; }
bool tc_chunk_supported(int C) { return C == kC; }

// ---- sequences cut into segments -------------------------------------------------------------------------
// One work item per unit leaves most SMs idle when there are few units (a 16K-token batch of two sequences has
// 32).  The recurrence is linear in the state, so a sequence can be cut into G segments that run side by side: (1)
// every segment runs state-only from a zero state (chunk_tc_state.cu), giving its local end state and its
// total decay Lambda = prod f; (2) a small kernel chains them in place, S <- Diag(Lambda[r]) S + S_local[r], and leaves
// S_N behind the last one; (3) every segment runs in full from its start state.  The same for units beyond the last full
// wave of whole units, which would keep a few SMs busy for a whole sequence while the rest idle.
// S_N is the chain's and not the last segment's own final state although that would save the state-only pass over the last
// segment: the state-only pass rounds a token's decay from the segment's end, where it is 1, the full pass in the
// mid-chunk frame, and the recent tokens weigh most.  Against fp64 S_N is off by 1.5e-3 and not 1.64e-3 (16 units of
// 5000 tokens, f >= 0.9), 1.6e-3 and not 2.4e-3 (6 of 9000, f >= 0.5); dS_0 likewise (2.24 and 2.40e-3, 2.06 and 2.3e-3).
int sm_count()
{
    // asked for several times per call (plans and sizes), so kept per device
    static std::atomic<int> known[64];
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (dev >= 0 && dev < 64 && (n = known[dev].load(std::memory_order_relaxed)) > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (dev >= 0 && dev < 64) known[dev].store(n, std::memory_order_relaxed);
    return n;
}

// How an ordinary batch of U units of NC chunks is cut.  The unit of the estimates is one chunk of the full pass (2 us
// forward, 4 us backward): a whole sequence takes NC + 4 (start-up and pipeline fill); segments take
// waves * (Lc + 4) for the full pass, 6 for the two extra launches with their start-up and 0.4 per chunk and pair of CTAs per
// SM for the state-only pass (measured: 55 us of state-only pass against 140 us of full pass at 64 chunks per CTA).
// At least 6 chunks per segment, at most 16 segments.  `gain` = the cut is expected to pay; the size queries make room for
// the best cut even where it does not.
SegPlan tc_plan(uint64_t U, int NC)
{
    SegPlan p{(int)U, 0, 1, 0, false};
    const int sms = sm_count();
    if (U == 0 || sms == 0 || U > 0x3fffffff) return p;
    const int cut = U <= (uint64_t)sms ? (int)U : (int)(U % sms);
    double best = 0.;
    for (int g = 2; cut > 0 && g <= 16; ++g) {
        const int Lc = (NC + g - 1) / g < 6 ? 6 : (NC + g - 1) / g, G = (NC + Lc - 1) / Lc;
        if (G < 2) continue;
        const int waves = (cut * G + sms - 1) / sms, pairs = (cut * G + 2 * sms - 1) / (2 * sms);
        const double cost = waves * (Lc + 4.0) + 6.0 + 0.4 * Lc * pairs;
        if (p.tail == 0 || cost < best) {
            best = cost;
            p = SegPlan{(int)U - cut, cut, G, Lc, cost < NC + 4.0};
        }
    }
    return p;
}

// Segments per sequence of a packed batch of T rows per head: as many as fill the SMs when the units alone fill at
// most half of them; none when no sequence can be longer than one segment (8 chunks).
int tc_packed_segments(uint64_t U, int T)
{
    const int sms = sm_count();
    if (U == 0 || sms == 0 || 2 * U > (uint64_t)sms || T <= 8 * kC) return 1;
    const int G = sms / (int)U;
    return G > 8 ? 8 : G;
}

namespace {

bool no_cut(const hgrn2_desc *d) { return (d->flags & kFlagNoSegments) != 0; }
SegPlan plan_of(const hgrn2_desc *d)
{
    const uint64_t U = (uint64_t)d->B * d->H;
    return no_cut(d) ? SegPlan{(int)U, 0, 1, 0, false} : tc_plan(U, (d->N + kC - 1) / kC);
}
int packed_segments_of(const hgrn2_desc *d) { return no_cut(d) ? 1 : tc_packed_segments((uint64_t)d->B * d->H, d->N); }
size_t chain_bytes(size_t units, int G) { return units * G * (kD * kD + kD) * sizeof(float) + ((units * 2 * sizeof(int) + 15) & ~(size_t)15); }

}  // namespace

size_t tc_saved_bytes(const hgrn2_desc *d, int C)
{
    const size_t NC = ((size_t)d->N + C - 1) / C;
    const uint64_t U = (uint64_t)d->B * d->H;
    size_t slots = (size_t)U * NC;
    if (d->N % C != 0) {
        const SegPlan p = plan_of(d);              // spare slots of cut units that are not whole chunks
        slots += (size_t)p.tail * (d->N / C + p.G + 1 - NC);
    }
    return slots * (kSavedStateBytes + kSavedTotalsBytes);
}

// Chain slots of the cut units, their segments' decays and what redo_claim counts.
size_t tc_segment_scratch_bytes(const hgrn2_desc *d, int C)
{
    const SegPlan p = plan_of(d);
    return p.tail ? chain_bytes(p.tail, p.G) : 0;
}

// One float matrix per work item for the exact path of the backward (chunk_alu.cuh, bwd_unit).
size_t tc_exact_scratch_bytes(const hgrn2_desc *d, bool packed)
{
    if (packed) return (size_t)d->B * d->H * packed_segments_of(d) * kD * kD * sizeof(float);
    const SegPlan p = plan_of(d);
    return ((size_t)p.main + (size_t)p.tail * p.G) * kD * kD * sizeof(float);
}

size_t tc_saved_bytes_packed(const hgrn2_desc *d)
{
    return (size_t)d->H * ((size_t)d->N / kC + (size_t)d->B * packed_segments_of(d) + 1) * (kSavedStateBytes + kSavedTotalsBytes);
}

size_t tc_segment_scratch_bytes_packed(const hgrn2_desc *d)
{
    const int G = packed_segments_of(d);
    // room for two matrices per segment
    return G <= 1 ? 0 : (size_t)d->B * d->H * G * (2 * kD * kD + kD) * sizeof(float);
}

// The work items of a call, the planes and chunk-state slots its tensors have, and where the decay totals sit.
TcWork tc_work(SeqArgs &a)
{
    TcWork t;
    const uint64_t U = (uint64_t)a.B * a.H;
    t.wk.N = a.N;
    t.wk.NC = a.NC;
    if (a.cu) {
        t.wk.cu = a.cu;
        t.wk.B = a.B;
        t.wk.H = a.H;
        t.wk.G = a.seg_scratch ? tc_packed_segments(U, a.N) : 1;
        t.wk.spp = a.N / kC + a.B * t.wk.G + 1;
        t.planes = a.H;
        t.slots = (uint64_t)a.H * t.wk.spp;
        t.cut = U;
        t.items = U * t.wk.G;
    } else {
        SegPlan p{(int)U, 0, 1, 0, false};
        if (a.seg_scratch) p = tc_plan(U, a.NC);
        if (!p.gain) p = SegPlan{(int)U, 0, 1, 0, false};
        t.wk.main = p.main;
        t.wk.tail = p.tail;
        t.wk.G = p.G;
        t.wk.Lc = p.Lc;
        t.planes = U;
        t.slots = U * a.NC;
        t.cut = p.tail;
        t.items = p.main + (uint64_t)p.tail * p.G;
    }
    if (t.wk.G > 1) {
        t.chain = static_cast<float *>(a.seg_scratch);
        t.lam = t.chain + t.cut * t.wk.G * kD * kD;
        if (!a.cu && a.N % kC == 0) t.redo = reinterpret_cast<int *>(t.lam + t.cut * t.wk.G * kD);
    }
    t.chunks = a.cu ? ((uint64_t)a.N / kC * a.H + t.items / 2) / (t.items ? t.items : 1) : (uint64_t)a.NC;
    if (a.states)
        a.totals = reinterpret_cast<float *>(reinterpret_cast<char *>(a.states) + t.slots * kSavedStateBytes);
    return t;
}

// Chains every cut unit's slots in place: on entry slot r holds what segment r adds to the state (backward: to the
// gradient), on exit the state at the start of segment r (the gradient at its end); `fin` (nullable) takes what is behind
// the last one of the chain.  A thread owns four neighbouring elements and has all its slots' loads in flight: the kernel is
// the latency of one round trip (16 units of 9 segments: 4.0 us, four slots at a time 9.4).
constexpr int kChainAhead = 16;
template <bool kBwd>
__global__ void __launch_bounds__(128)
seg_chain_kernel(const float *init, float *fin, float *chain, const float *lam, int *redo, const WorkArgs w)
{
    chain_wait();
    const size_t t = blockIdx.y, unit = w.main + t;
    const int e = (blockIdx.x * 128 + threadIdx.x) * 4, k = e / kD, G = w.G;
    if (redo != nullptr && blockIdx.x == 0 && threadIdx.x < 2) redo[2 * t + threadIdx.x] = 0;
    if (w.cu != nullptr && packed_malformed(w, (int)t / w.H)) fin = nullptr;      // such a unit writes nothing
    float S[4] = {0.f, 0.f, 0.f, 0.f};
    if (init) load4(init + unit * kD * kD + e, S);
    float *slots = chain + t * G * kD * kD + e;
    const float *lams = lam + t * G * kD + k;
    const int n = fin ? G : G - 1;                                   // without fin nobody has filled the chain's last slot
    for (int n0 = 0; n0 < G; n0 += kChainAhead) {
        float x[kChainAhead][4], l[kChainAhead];
#pragma unroll
        for (int j = 0; j < kChainAhead; ++j)
            if (n0 + j < n) {
                const int r = kBwd ? G - 1 - n0 - j : n0 + j;
                load4(slots + (size_t)r * kD * kD, x[j]);
                l[j] = lams[r * kD];
            }
#pragma unroll
        for (int j = 0; j < kChainAhead; ++j)
            if (n0 + j < G) {
                const int r = kBwd ? G - 1 - n0 - j : n0 + j;
                *reinterpret_cast<float4 *>(slots + (size_t)r * kD * kD) = make_float4(S[0], S[1], S[2], S[3]);
                if (n0 + j < n)
#pragma unroll
                    for (int i = 0; i < 4; ++i) S[i] = fmaf(l[j], S[i], x[j][i]);
            }
    }
    if (fin) *reinterpret_cast<float4 *>(fin + unit * kD * kD + e) = make_float4(S[0], S[1], S[2], S[3]);
}

cudaError_t launch_seg_chain(bool bwd, const TcWork &t, const float *init, float *fin, cudaStream_t stream)
{
    const dim3 grid(kD * kD / 512, (unsigned)t.cut);
    return launch_chained(bwd ? seg_chain_kernel<true> : seg_chain_kernel<false>, grid, 128, 0, stream, init, fin, t.chain, t.lam, t.redo, t.wk);
}

// More items than SMs: a CTA takes several (kPersist).  Against one CTA per item on 148 SMs: 4736 units of 64 tokens 193
// instead of 294 us, 1184 of 256 107 / 136, 592 of 512 92 / 104, 296 of 1024 86 / 89, 592 of 2048 320 / 325.  With one item
// per CTA that instantiation gains nothing and costs about a microsecond.
cudaError_t launch_tc_fwd(const SeqArgs &a0)
{
    SeqArgs a = a0;
    const TcWork t = tc_work(a);
    if (t.items > 0x7fffffffull) return cudaErrorInvalidConfiguration;
    const bool want_y = a.y != nullptr, want_saved = a.states != nullptr;
    cudaError_t err;
    if (t.wk.G > 1) {
        // the state-only pass holds for every f: it needs no exact path of its own
        err = launch_tc_state(false, nullptr, a.f, a.i, t, a.SN != nullptr, a.gate_enc, a.status, a.clear_status, a.start_aborted, a.stream);
        if (err != cudaSuccess) return err;
        if ((err = launch_seg_chain(false, t, a.S0, a.SN, a.stream)) != cudaSuccess) return err;
        a.clear_status = false;
    }
    CUtensorMap mo, mf, mi, my, ms;
    // tensor maps need a valid base even for outputs that are not wanted: point those at an input
    if (!make_map(&mo, a.o, t.planes, a.N, kC) || !make_map(&mf, a.f, t.planes, a.N, kC) || !make_map(&mi, a.i, t.planes, a.N, kC) ||
        !make_map(&my, want_y ? a.y : a.i, t.planes, a.N, kC) ||
        !make_map(&ms, want_saved ? static_cast<const void *>(a.states) : a.i, want_saved ? t.slots : t.planes,
                  want_saved ? (uint64_t)kD : (uint64_t)a.N, want_saved ? kD : kC))
        return cudaErrorInvalidValue;
    const bool ragged = a.N % kC != 0 || a.cu != nullptr, persist = t.items > (uint64_t)sm_count();
    auto kernel = a.gate_enc ? (ragged ? (persist ? tc_fwd_kernel<true, true, true> : tc_fwd_kernel<true, true, false>)
                                       : (persist ? tc_fwd_kernel<false, true, true> : tc_fwd_kernel<false, true, false>))
                             : (ragged ? (persist ? tc_fwd_kernel<true, false, true> : tc_fwd_kernel<true, false, false>)
                                       : (persist ? tc_fwd_kernel<false, false, true> : tc_fwd_kernel<false, false, false>));
    if ((err = ensure_dynamic_smem(reinterpret_cast<const void *>(kernel), kSmemBytes)) != cudaSuccess) return err;
    ExactArgs ex;
    ex.o = static_cast<const __nv_bfloat16 *>(a.o);
    ex.f = static_cast<const __nv_bfloat16 *>(a.f);
    ex.i = static_cast<const __nv_bfloat16 *>(a.i);
    ex.y = static_cast<__nv_bfloat16 *>(a.y);
    ex.states = reinterpret_cast<__nv_bfloat16 *>(a.states);
    return launch_chained(kernel, dim3((unsigned)t.items), kThreads, kSmemBytes, a.stream, mo, mf, mi, my, ms, a.S0, t.chain, t.redo, a.SN, want_saved ? a.totals : nullptr, want_y, want_saved, t.wk, a.status, a.clear_status ? 1 : 0, ex, a.start_aborted);
}

}  // namespace hgrn2
