// Chunkwise HGRN2 backward on the Blackwell tensor cores (tcgen05 + TMEM + TMA), bf16 I/O, fp32
// state gradient, d_k = d_v = 128, chunk length C = 64 (frame and notation: tc_chunk.cuh).
//
// Reverse sweep over the chunks with the state gradient resident in tensor memory.  In the mid frame,
// with dS'' = Diag(E) dS_out and S' the saved forward state of the chunk:
//
//   A  = tril(Qs Ks^T)          dA = tril(dY V^T)
//   dQs^T       = Ks^T dA^T + S' dY^T            (accumulator [key dim][t])
//   dKs_intra^T = Qs^T dA                        (accumulator [key dim][s])
//   dKs_inter^T = dS'' V^T                       (accumulator [key dim][s])
//   dV^T        = dY^T A + dS''^T Ks^T           (accumulator [value dim][s])
//   dS'         = dS'' + Qs^T dY,   dS_in = Diag(Pm) dS'
//   a = Qs*dQs - Ks*dKs_intra,  e = Ks*dKs_inter,  R_k = sum_v dS''[k,v] S'[k,v]
//   dg_t = sum_{j>=t} a_j + sum_{s<t} e_s + R            (gradient w.r.t. log f_t)
//   d_o = dQs * exp(b_t - b_m),  dk = (dKs_intra + dKs_inter) * exp(b_m - b_s),  d_f = dg / f - dk
//
// Every accumulator that feeds an output puts one key (or value) dimension in each TMEM lane, so the
// thread that owns the lane sees a whole column of the chunk: the scans along time stay in registers
// and each output store of a warp covers 64 contiguous bytes of one token row.
//
// Warp roles (hand-offs are mbarriers, every wait is bounded; loops stay rolled to keep the
// instruction footprint of the concurrently running roles small):
//   T   4 warps: raw o, f tiles -> Qs, Ks in place, one chunk ahead (two TMA stages);
//   E1  4 warps: rescale the dS accumulator and publish its bf16 copy dS'' (the chain between chunks), R;
//   E3  8 warps: d_o and d_f from dQs^T, dKs_intra^T, dKs_inter^T.  A thread owns (key dim, half of the chunk)
//       and walks its 32 steps outwards from the middle, carrying the decay product and one running sum;
//       what is still missing then is one constant per key dimension (R plus the two halves' sums), so the
//       almost finished d_f and 1/f are parked in the TMEM columns just read, and once all eight warps are
//       through each thread completes its own 32 rows.  It works from a second, unswizzled copy of raw o and f
//       and recomputes Qs, Ks with the transform's roundings, so the operand stage is free as soon as the
//       chunk's products are done;
//   O   4 warps: the causal masks of A and dA into operand slabs (32 rows per warp), and d_i from dV^T;
//   L   1 warp: TMA loads (o, f, dy stage; v; saved S'; raw o, f), each refilled when its last reader is done;
//   MX, MY1, MY2  1 warp each: tcgen05.mma issue of the groups below (one lane issuing all 56
//       products of a chunk is itself a bottleneck: its instruction stream is long and serial).
// Per chunk the tensor pipe runs, each group as soon as what it overwrites has been read out
//   X  (MX) : A | dA, then dS' += Qs^T dY   (overlap the outputs of the previous chunk)
//   Y1a (MY1): dV^T = dS''^T Ks^T           (needs the previous chunk's d_i out: early)
//   Y1b (MY1): dKs_inter^T                  (needs the previous chunk's output walk finished)
//   Y2a (MY2): dV^T += dY^T A               (needs tril(A), and Y1a complete)
//   Y2b (MY2): dQs^T | dKs_intra^T          (needs tril(dA), S', and the previous chunk's parked values consumed)
// Event stamps of one CTA put the chunk period at: output walk (3.7 k cycles) -> completion of d_f (1.3 k) ->
// Y2b (1.1 k) -> next walk; with a single Y1 group behind the walk and the masks and the completion pass in the
// other roles' hands the same stamps showed a second, equally long chain through Y1 and Y2.
//
// Tensor-memory plan (512 columns, no spare): dS [0,128); A [128,192) in lanes 0..63 and dA [192,256) in
// lanes 64..127 (products of the stacked operand (Qs; dY), M = 128); dQs^T [256,320); dKs_intra^T [320,384);
// dKs_inter^T [384,448); dV^T [448,512).
#include "chunk_alu.cuh"
#include "tc_chunk.cuh"

namespace hgrn2 {

namespace {

using namespace tc;

constexpr int kTWarps = 4, kE1Warps = 4, kE3Warps = 8, kOWarps = 4;
constexpr int kE1Threads = kE1Warps * 32, kE3Threads = kE3Warps * 32, kOThreads = kOWarps * 32;
constexpr int kWarpE1 = kTWarps, kWarpE3 = kWarpE1 + kE1Warps, kWarpO = kWarpE3 + kE3Warps;
constexpr int kWarpLoad = kWarpO + kOWarps, kWarpMmaX = kWarpLoad + 1, kWarpMmaY1 = kWarpLoad + 2,
              kWarpMmaY2 = kWarpLoad + 3;
constexpr int kThreads = (kWarpMmaY2 + 1) * 32;
constexpr int kRingWarps = kTWarps + kE1Warps + kE3Warps + kOWarps + 3;   // readers of the item ring

constexpr int kStages = 2;
constexpr uint32_t kStageBytes = 3 * kTile;                       // q, dy, f: free again when the chunk's products are done
// Stage layout: [q slab 0][dy slab 0][q slab 1][dy slab 1][f slab 0][f slab 1].  With the slabs of q and dy
// interleaved, (Qs; dY) also reads as ONE 128-row K-major operand whose slabs are 16 KB apart.
constexpr uint32_t kSS = 2 * kSlab;                               // distance between the two slabs of the q and dy tiles
constexpr uint32_t kOffQ = 0, kOffG = kSlab, kOffK = 2 * kTile;
constexpr uint32_t kOffV = kStages * kStageBytes;                 // v: one buffer, free when X and Y1 of the chunk are done
constexpr uint32_t kOffS = kOffV + kTile;                         // S' (bf16, from the forward)
constexpr uint32_t kOffDS = kOffS + kStateTile;                   // bf16 copy of dS''
constexpr uint32_t kOffP = kOffDS + kStateTile;                   // bf16 tril(A)
constexpr uint32_t kOffDP = kOffP + kSlab;                        // bf16 tril(dA)
constexpr uint32_t kOffRawO = kOffDP + kSlab;                     // raw o and f of the chunk, plain [64][128] bf16, for
constexpr uint32_t kOffRawF = kOffRawO + kTile;                   // the output warps (the stage holds Qs, Ks by then)
constexpr uint32_t kOffR = kOffRawF + kTile;                      // float rr[2][128]
constexpr uint32_t kOffX = kOffR + 2 * 128 * 4;                   // float xa[128], xe[128]
constexpr uint32_t kOffCtl = kOffX + 2 * 128 * 4;
constexpr uint32_t kSmemBytes = kOffCtl + 768;                    // no slack: the base must be 1024-byte aligned

constexpr uint32_t kColDS = 0, kColA = 128, kColDA = 192, kColDQ = 256, kColDKi = 320, kColDKx = 384, kColDV = 448;

struct Ctl {
    uint64_t full[kStages];       // TMA (o, f, dy tiles) -> T, M
    uint64_t vfull;               // TMA (v tile) -> M
    uint64_t rawfull;             // TMA (second, unswizzled copy of o and f) -> E3
    uint64_t raw_read;            // E3 -> L: the raw copies have been read for the last time
    uint64_t t_done[kStages];     // T -> M, E1
    uint64_t sfull;               // TMA (saved S') -> E1, M
    uint64_t m_done;              // E1 -> M: dS'' is in TMEM and in shared memory
    uint64_t barA;                // tcgen05.commit -> O: A, dA complete
    uint64_t barX;                // tcgen05.commit -> E1, L: the dS' update complete as well
    uint64_t pd_ready;            // O -> M: tril(A), tril(dA) are in shared memory
    uint64_t barY1a;              // tcgen05.commit -> MY2: dV^T = dS''^T Ks^T complete
    uint64_t barY1;               // tcgen05.commit -> E1, L, MY2: both products of dS'' complete (its copy and v no longer read)
    uint64_t barY2;               // tcgen05.commit -> E3, O, L: every product of the chunk complete
    uint64_t r_ready[2];          // E1 -> E3, L: R of the chunk is in shared memory, S' no longer read by threads
                                  // (two barriers: the slower of the two waiters must not be lapped)
    uint64_t acc_free1;           // E3 -> M: dKs_inter^T has been read out
    uint64_t acc_freeV;           // O -> M: dV^T has been read out
    uint64_t parked;              // E3 -> E3: every thread's parked values and the halves' sums are in place
    uint64_t acc_free2;           // E3 -> M: dQs^T and dKs_intra^T columns are free again
    uint64_t drain;               // tcgen05.commit (MX, MY1, MY2, after their loops): every product issued has completed
    alignas(16) ItemRing ring;
    int abort_flag;               // set by the first wait that runs out: every later wait returns at once
    uint32_t tmem_base;
    int exact_flag;               // E1: a decay of this CTA's tokens left the range of the rescaled operands
    int l_stage, l_v, l_state, l_raw;   // L: fills asked for so far, per buffer, for the abort epilogue
    int claimed;                  // redo_claim's answer
};
static_assert(sizeof(Ctl) <= 768, "control block");
static_assert(kSmemBytes <= 232448, "shared memory budget");

constexpr int kExactC = 32;       // chunk length of the exact fp32 routines at d = 128 (their shared-memory budget)
static_assert(alu::bwd_smem_floats(kD, kD, kExactC) * sizeof(float) <= kSmemBytes, "exact path fits the CTA's shared memory");

// d_o and the nearly finished d_f of one thread: key dimension k, local times [32 * kUp, 32 * kUp + 32),
// walked outwards from the middle of the chunk in blocks of four rows (a short loop body: the role shares its
// scheduler's instruction stream with four others).  Returns this half's sums of a and e.
// do_g points at element (row 0 of the chunk, column k) of d_o in global memory.  oraw, fraw: the chunk's raw
// o and f as plain [64][128] bf16 tiles (rows beyond the end of the sequence hold the neutral f = 1, o = 0).
// Qs and Ks are recomputed from them with the transform's own roundings, so the operand stage does not have to be held until the outputs
// are done.  The role is bound by its instruction count: per element one reciprocal (1/f is the ratio of two
// consecutive products), fused packed multiply-adds, and a single running sum.  kPartial: a sequence's last, partial
// chunk.  Such chunks have an instance of their own, and so have their d_f and d_i below: a test per row, or per block
// of rows, on the stores of every chunk made the ragged backward 5 to 11 % slower than the other (160 us instead of
// 142 for 128 units of 2047 and 2048 tokens; 146 now).
template <bool kUp, bool kPartial, bool kEnc>
__device__ __forceinline__ void phase_main(uint32_t tmem_lane, const unsigned short *oraw, const unsigned short *fraw,
                                           int k, __nv_bfloat16 *do_g, int n_valid, float &asum, float &esum)
{
    float cp = 1.f, ci = 1.f;       // running product of f between the middle and the current row, and its reciprocal
    float W = 0.f;                  // running sum of a - e over the rows visited so far
    float2 Gp = make_float2(0.f, 0.f);   // sum of a over the rows visited so far, even and odd rows apart
#pragma unroll 1
    for (int b = 0; b < 8; ++b) {
        const int t0 = kUp ? 32 + 4 * b : 28 - 4 * b;          // lowest row of the block (a multiple of 4)
        uint32_t x[4], y[4], z[4];
        tmem_ld4(tmem_lane + kColDQ + t0, x);
        tmem_ld4(tmem_lane + kColDKi + t0, y);
        tmem_ld4(tmem_lane + kColDKx + t0, z);
        uint32_t fw[4], qw[4];         // raw bf16 bits
        float fv[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int t = t0 + j;
            fw[j] = fraw[t * kD + k];
            qw[j] = oraw[t * kD + k];
            if (kEnc) {                       // fw[j] becomes the bf16 bits of k, as the transform formed them
                float kv;
                gate_decode(fw[j], fv[j], kv);
                fw[j] = pack_bf16(kv, 0.f) & 0xFFFFu;        // rounded to bf16 exactly as the transform rounds it
            } else {
                fv[j] = __uint_as_float(fw[j] << 16);
            }
        }
        tmem_wait_ld();
        // Scale factors along the walk (sequential in the running product) and 1/f.  No floor here: a product
        // that would need one has put the unit on the exact path already (the totals the state warps test are
        // never larger than any product formed here), and what this pass writes for such a unit is overwritten.
        // 1/f is the ratio of two consecutive products, so one reciprocal per element serves both.
        float sq[4], sk[4], rf[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int j = kUp ? i : 3 - i;                      // visiting order: away from the middle
            const float c0 = cp, i0 = ci;
            cp *= fv[j];
            ci = rcp_fast(cp);
            sq[j] = kUp ? cp : i0;
            sk[j] = kUp ? ci : c0;
            rf[j] = kEnc ? rcp_fast(fmaxf(fv[j], kFDivMinK)) : c0 * ci;
        }
        // element-wise part, two rows per instruction (packed fp32)
        float w[4], dk[4];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int j = 2 * p;
            const float2 X = make_float2(__uint_as_float(x[j]), __uint_as_float(x[j + 1]));
            const float2 Y = make_float2(__uint_as_float(y[j]), __uint_as_float(y[j + 1]));
            const float2 Z = make_float2(__uint_as_float(z[j]), __uint_as_float(z[j + 1]));
            // Qs and -Ks of the two rows exactly as the transform warps rounded them for the products: the terms
            // of a cancel in pairs along the chunk only if both sides use the same operand values
            const uint32_t sqp = pack_bf16(sq[j], sq[j + 1]), skp = pack_bf16(sk[j], sk[j + 1]);
            const uint32_t qsp = mul_bf16x2(qw[j] | (qw[j + 1] << 16), sqp);
            const uint32_t ksn = kEnc ? mul_bf16x2(fw[j] | (fw[j + 1] << 16), skp ^ 0x80008000u)
                                      : fma_bf16x2(fw[j] | (fw[j + 1] << 16), skp, skp ^ 0x80008000u);
            const float2 QS = make_float2(bf16_lo(qsp), bf16_hi(qsp)), KSn = make_float2(bf16_lo(ksn), bf16_hi(ksn));
            const float2 dox = mul2(X, make_float2(sq[j], sq[j + 1]));
            const float2 a2 = fma2(KSn, Y, mul2(QS, X));
            const float2 w2 = fma2(KSn, Z, a2);                 // a - e
            Gp = add2(Gp, a2);
            const float2 dk2 = mul2(add2(Y, Z), make_float2(sk[j], sk[j + 1]));
            if (!kPartial || t0 + j < n_valid) do_g[(size_t)(t0 + j) * kD] = __float2bfloat16_rn(dox.x);
            if (!kPartial || t0 + j + 1 < n_valid) do_g[(size_t)(t0 + j + 1) * kD] = __float2bfloat16_rn(dox.y);
            w[j] = w2.x; w[j + 1] = w2.y;
            dk[j] = dk2.x; dk[j + 1] = dk2.y;
        }
        // With K = R + (sum of a over the second half) + (sum of e over the first half), which the final pass
        // adds, dg_t = K - sum_{32 <= s < t} (a_s - e_s) after the middle and K + sum_{t <= j < 32} (a_j - e_j)
        // before it: one running sum along the walk
        float u[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int j = kUp ? i : 3 - i;
            if (kUp) {
                u[j] = fmaf(-W, rf[j], -dk[j]);
                W += w[j];
            } else {
                W += w[j];
                u[j] = fmaf(W, rf[j], -dk[j]);
            }
        }
        // park u and 1/f in the columns just read
        tmem_st4(tmem_lane + kColDQ + t0, u);
        tmem_st4(tmem_lane + kColDKi + t0, rf);
    }
    asum = Gp.x + Gp.y;
    esum = asum - W;
}

// kRagged: sequences need not be whole chunks (a partial chunk is padded with neutral tokens), and a packed batch is one.
// kEnc: the f tensor holds the signed gate encoding (see transform_half); d_f stays the gradient with respect to f.
// kPersist: several items per CTA (tc_chunk.cuh).
template <bool kRagged, bool kEnc, bool kPersist>
__global__ void __launch_bounds__(kThreads, 1)
tc_bwd_kernel(const __grid_constant__ CUtensorMap map_o, const __grid_constant__ CUtensorMap map_f,
              const __grid_constant__ CUtensorMap map_i, const __grid_constant__ CUtensorMap map_dy,
              const __grid_constant__ CUtensorMap map_saved, const __grid_constant__ CUtensorMap map_o_raw,
              const __grid_constant__ CUtensorMap map_f_raw, const float *totals,
              const float *dSN, const float *chain, int *__restrict__ redo, __nv_bfloat16 *__restrict__ d_o,
              __nv_bfloat16 *__restrict__ d_f, __nv_bfloat16 *__restrict__ d_i, float *__restrict__ dS0,
              const __grid_constant__ WorkArgs wk, StatusBlock *status, int clear_status, const ExactArgs ex,
              int start_aborted)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    if (smem_u32(smem) & 1023u) {          // every byte is spoken for: the swizzled tiles need the base aligned
        chain_wait();
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            if (clear_status) clear_block(status);
            report_error(status, HGRN2_ERR_CUDA, 3);
        }
        return;
    }
    uint8_t *sbuf = smem + kOffS;
    uint8_t *dsbuf = smem + kOffDS;
    uint8_t *pbuf = smem + kOffP;
    uint8_t *dpbuf = smem + kOffDP;
    unsigned short *oraw = reinterpret_cast<unsigned short *>(smem + kOffRawO);          // bf16 bits
    unsigned short *fraw = reinterpret_cast<unsigned short *>(smem + kOffRawF);
    uint8_t *vbuf = smem + kOffV;
    float *rr = reinterpret_cast<float *>(smem + kOffR);
    float *xa = reinterpret_cast<float *>(smem + kOffX);
    float *xe = xa + 128;
    Ctl *ctl = reinterpret_cast<Ctl *>(smem + kOffCtl);
    volatile int *abort_flag = &ctl->abort_flag;

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&ctl->full[s], 1);
            mbar_init(&ctl->t_done[s], kTransformThreads);
        }
        mbar_init(&ctl->vfull, 1);
        mbar_init(&ctl->rawfull, 1);
        mbar_init(&ctl->raw_read, kE3Threads);
        mbar_init(&ctl->sfull, 1);
        mbar_init(&ctl->m_done, kE1Threads);
        mbar_init(&ctl->barA, 1);
        mbar_init(&ctl->barX, 1);
        mbar_init(&ctl->pd_ready, kOThreads);
        mbar_init(&ctl->barY1a, 1);
        mbar_init(&ctl->barY1, 1);
        mbar_init(&ctl->barY2, 1);
        mbar_init(&ctl->r_ready[0], kE1Threads);
        mbar_init(&ctl->r_ready[1], kE1Threads);
        mbar_init(&ctl->acc_free1, kE3Threads);
        mbar_init(&ctl->acc_freeV, kOThreads);
        mbar_init(&ctl->parked, kE3Threads);
        mbar_init(&ctl->acc_free2, kE3Threads);
        mbar_init(&ctl->drain, 3);
        ctl->abort_flag = start_aborted;
        ctl->exact_flag = 0;
        ctl->l_stage = ctl->l_v = ctl->l_state = ctl->l_raw = 0;
        ring_init(ctl->ring, kRingWarps);
        fence_barrier_init();
        tma_prefetch_desc(&map_o);
        tma_prefetch_desc(&map_f);
        tma_prefetch_desc(&map_i);
        tma_prefetch_desc(&map_dy);
        tma_prefetch_desc(&map_saved);
        tma_prefetch_desc(&map_o_raw);
        tma_prefetch_desc(&map_f_raw);
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
    const int krow = 32 * sub + lane;                                // TMEM lane of this thread

    // it = 0, 1, ... counts the chunks over all of the CTA's items; an item's chunks are visited from its last to its first
    if (warp < kTWarps) {
        // ================= T: transform =================
        PT_DECL
        int it = 0;
        Item im;
        for (int k = 0; next_item<kPersist>(&ctl->ring, k, abort_flag, first, im); ++k) {
            for (int c = (im.n + kC - 1) / kC - 1; c >= 0; --c, ++it) {
                const int s = it % kStages;
                uint8_t *qbuf = smem + s * kStageBytes;
                mbar_wait(&ctl->full[s], (it / kStages) & 1, abort_flag);
                // No pacing: the transform of chunk `it` may run alongside the output walk of chunk it - 2.  (While A and
                // dA waited for the state gradient, holding it back until that walk was over was 2 % faster; since they
                // do not, it is 1 % slower: 128 units of 2048 tokens forward + backward 212 against 206 us, 592 of 512 256 against 252.)
                PT_MARK(0)
                PT_STAMP(status, 1, tid == 0 && it == 16) PT_STAMP(status, 20, tid == 0 && it == 18)
                // Pm and E of the chunk are not kept: the backward takes them from what the forward saved
                if (kRagged && im.n - c * kC < kC) neutral_rows<kEnc, kSS, kSlab>(qbuf + kOffQ, qbuf + kOffK, im.n - c * kC, tid);
                transform_stream<kEnc, kSS, kSlab>(qbuf + kOffQ, qbuf + kOffK, nullptr, nullptr, nullptr, nullptr, tid);
                fence_proxy_async_smem();
                mbar_arrive(&ctl->t_done[s]);
                PT_MARK(1)
                PT_STAMP(status, 2, tid == 0 && it == 16)
            }
        }
        PT_DUMP(status, 0, 2, tid == 0)
    } else if (warp < kWarpE3) {
        // ================= E1: state-gradient warps =================
        // Pm, E of every chunk come from the forward's saved totals, so this chain does not wait for T
        PT_DECL
        int it = 0;
        Item im;
        for (int k = 0; next_item<kPersist>(&ctl->ring, k, abort_flag, first, im); ++k) {
            const int nc = (im.n + kC - 1) / kC;
            const size_t row = ((size_t)im.unit * kD + krow) * kD;
            float pm_prev = 1.f, pm_c = 1.f, ee_c = 1.f;
            const float *tot_u = totals + (size_t)im.slot0 * 2 * kD + krow;
            // the accumulator starts as the gradient that comes in, so the loop over the chunks has no first-chunk case (the
            // previous item's last update of it is done behind barX)
            if (nc > 0) {
                const float *init = im.chain >= 0 ? chain + ((size_t)im.chain * kD + krow) * kD : (dSN ? dSN + row : nullptr);
                pm_c = tot_u[(size_t)(nc - 1) * 2 * kD];
                ee_c = tot_u[(size_t)(nc - 1) * 2 * kD + kD];
                if (it > 0) mbar_wait(&ctl->barX, (it - 1) & 1, abort_flag);
                tc_fence_after_sync();
#pragma unroll 1
                for (int part = 0; part < 4; ++part) {
                    uint32_t r[32];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float4 v4 = init ? reinterpret_cast<const float4 *>(init + 32 * part)[j] : make_float4(0.f, 0.f, 0.f, 0.f);
                        r[4 * j + 0] = __float_as_uint(v4.x); r[4 * j + 1] = __float_as_uint(v4.y);
                        r[4 * j + 2] = __float_as_uint(v4.z); r[4 * j + 3] = __float_as_uint(v4.w);
                    }
                    tmem_st32(tmem + lane_base + kColDS + 32 * part, r);
                }
                tmem_wait_st();
            }
            for (int c = nc - 1; c >= 0; --c, ++it) {
                // ---- dS'' = (Pm_prev E) dS' (the accumulator) -> TMEM, bf16 copy -> dsbuf
                PT_MARK(0)
                // a total on the floor: the decay across that half chunk is more than the rescaled operands can carry
                if (fminf(pm_c, ee_c) <= kProdFloor) {
                    ctl->exact_flag = 1;
                    if (kPersist) ctl->ring.flagged[k & 7] = im.id + 1;
                }
                const float pm_old = pm_prev, ee_old = ee_c;
                const float factor = pm_prev * ee_c;
                pm_prev = pm_c;
                const bool safe = factor >= kFactorSafe;
                if (c > 0) {
                    pm_c = tot_u[(size_t)(c - 1) * 2 * kD];
                    ee_c = tot_u[(size_t)(c - 1) * 2 * kD + kD];
                }
                if (it > 0) {
                    mbar_wait(&ctl->barX, (it - 1) & 1, abort_flag);   // dS' of the previous chunk is complete
                    mbar_wait(&ctl->barY1, (it - 1) & 1, abort_flag);    // its dS'' copy is no longer read
                    tc_fence_after_sync();
                }
                PT_MARK(1)
                PT_STAMP(status, 5, tid == kWarpE1 * 32 && it == 16)
#pragma unroll 1
                for (int part = 0; part < 4; ++part) {
                    uint32_t r[32];
                    tmem_ld32(tmem + lane_base + kColDS + 32 * part, r);
                    tmem_wait_ld();
                    float f1 = safe ? factor : pm_old;               // see the forward kernel: or the two decays one after the other
#pragma unroll 1
                    for (int more = safe ? 0 : 1; more >= 0; --more, f1 = ee_old)
#pragma unroll
                        for (int j = 0; j < 32; j += 2) scale2(r[j], r[j + 1], f1);
                    tmem_st32(tmem + lane_base + kColDS + 32 * part, r);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        *reinterpret_cast<uint4 *>(dsbuf + (part >> 1) * kStateSlab + slab_chunk_off(krow, 4 * (part & 1) + j)) =
                            pack8(r + 8 * j);
                }
                tmem_wait_st();
                tc_fence_before_sync();
                fence_proxy_async_smem();
                mbar_arrive(&ctl->m_done);
                PT_MARK(2)
                PT_STAMP(status, 6, tid == kWarpE1 * 32 && it == 16)

                // ---- R_k = sum_v dS''[k,v] S'[k,v] from the two bf16 copies
                mbar_wait(&ctl->sfull, it & 1, abort_flag);
                PT_MARK(3)
                float2 racc2 = make_float2(0.f, 0.f);
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
#pragma unroll 2
                    for (int j = 0; j < 8; ++j) {
                        const uint32_t off = h * kStateSlab + slab_chunk_off(krow, j);
                        const uint4 dw = *reinterpret_cast<const uint4 *>(dsbuf + off);
                        const uint4 sw = *reinterpret_cast<const uint4 *>(sbuf + off);
                        racc2 = fma2(make_float2(bf16_lo(dw.x), bf16_hi(dw.x)), make_float2(bf16_lo(sw.x), bf16_hi(sw.x)), racc2);
                        racc2 = fma2(make_float2(bf16_lo(dw.y), bf16_hi(dw.y)), make_float2(bf16_lo(sw.y), bf16_hi(sw.y)), racc2);
                        racc2 = fma2(make_float2(bf16_lo(dw.z), bf16_hi(dw.z)), make_float2(bf16_lo(sw.z), bf16_hi(sw.z)), racc2);
                        racc2 = fma2(make_float2(bf16_lo(dw.w), bf16_hi(dw.w)), make_float2(bf16_lo(sw.w), bf16_hi(sw.w)), racc2);
                    }
                }
                const float racc = racc2.x + racc2.y;
                rr[(it & 1) * 128 + krow] = racc;
                mbar_arrive(&ctl->r_ready[it & 1]);
                PT_MARK(4)
                PT_STAMP(status, 9, tid == kWarpE1 * 32 && it == 16)
            }
            // dS_0 = Diag(Pm of chunk 0) dS'; without tokens the gradient passes through
            if (dS0 != nullptr && im.last) {
                if (nc > 0) {
                    mbar_wait(&ctl->barX, (it - 1) & 1, abort_flag);
                    tc_fence_after_sync();
                }
#pragma unroll 1
                for (int part = 0; part < 4; ++part) {
                    uint32_t r[32];
                    float4 *dst = reinterpret_cast<float4 *>(dS0 + row + 32 * part);
                    if (nc > 0) {
                        tmem_ld32(tmem + lane_base + kColDS + 32 * part, r);
                        tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            dst[j] = make_float4(__uint_as_float(r[4 * j + 0]) * pm_prev, __uint_as_float(r[4 * j + 1]) * pm_prev,
                                                 __uint_as_float(r[4 * j + 2]) * pm_prev, __uint_as_float(r[4 * j + 3]) * pm_prev);
                    } else {
#pragma unroll 1
                        for (int j = 0; j < 8; ++j)
                            dst[j] = dSN ? reinterpret_cast<const float4 *>(dSN + row + 32 * part)[j] : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
            }
        }
        PT_DUMP(status, 2, 5, tid == kWarpE1 * 32)
    } else if (warp < kWarpO) {
        // ================= E3: d_o and d_f =================
        const int half = (warp - kWarpE3) >> 2;                      // half of the chunk: local times [32 * half, +32)
        const uint32_t tl = tmem + lane_base;
        PT_DECL
        int it = 0;
        Item im;
        for (int k = 0; next_item<kPersist>(&ctl->ring, k, abort_flag, first, im); ++k) {
            const size_t grow0 = (size_t)im.plane * wk.N + im.row0;     // first row of the item in the [planes * rows][128] view
            for (int c = (im.n + kC - 1) / kC - 1; c >= 0; --c, ++it) {
                const int n_valid = kRagged ? min(kC, im.n - c * kC) : kC;
                const size_t crow0 = grow0 + c * kC;
                // ---- outputs
                mbar_wait(&ctl->rawfull, it & 1, abort_flag);
                mbar_wait(&ctl->barY2, it & 1, abort_flag);
                PT_MARK(2)
                tc_fence_after_sync();
                float asum, esum;
                PT_STAMP(status, 14, tid == kWarpE3 * 32 && it == 16)
                __nv_bfloat16 *do_g = d_o + crow0 * kD + krow;
                if (kRagged && n_valid < kC) {
                    // rows beyond the end: see neutral_rows (this thread's column of its half)
#pragma unroll 1
                    for (int r = max(n_valid, 32 * half); r < 32 * half + 32; ++r) {
                        oraw[r * kD + krow] = 0u;
                        fraw[r * kD + krow] = kEnc ? 0x8000u : 0x3F80u;
                    }
                    if (half) phase_main<true, true, kEnc>(tl, oraw, fraw, krow, do_g, n_valid, asum, esum);
                    else      phase_main<false, true, kEnc>(tl, oraw, fraw, krow, do_g, n_valid, asum, esum);
                    fence_proxy_async_smem();                        // the rows written here, before the tiles' next load
                } else {
                    if (half) phase_main<true, false, kEnc>(tl, oraw, fraw, krow, do_g, n_valid, asum, esum);
                    else      phase_main<false, false, kEnc>(tl, oraw, fraw, krow, do_g, n_valid, asum, esum);
                }
                mbar_arrive(&ctl->raw_read);
                if (half) xa[krow] = asum; else xe[krow] = esum;
                tmem_wait_st();
                tc_fence_before_sync();
                mbar_arrive(&ctl->acc_free1);
                mbar_arrive(&ctl->parked);
                PT_MARK(3)
                PT_STAMP(status, 15, tid == kWarpE3 * 32 && it == 16)
                // ---- d_f completed from the parked values, each thread its own 32 rows, once both halves' sums and R
                // of the chunk are there
                mbar_wait(&ctl->r_ready[it & 1], (it >> 1) & 1, abort_flag);
                mbar_wait(&ctl->parked, it & 1, abort_flag);
                tc_fence_after_sync();
                {
                    const float K = rr[(it & 1) * 128 + krow] + xa[krow] + xe[krow];
                    __nv_bfloat16 *df_g = d_f + crow0 * kD + krow;
                    // the thread's 64 parked values in two reads (the pass is on the chunk's critical chain)
                    if (!kRagged || n_valid == kC) {
                        uint32_t uu[32], rf[32];
                        tmem_ld32(tl + kColDQ + 32 * half, uu);
                        tmem_ld32(tl + kColDKi + 32 * half, rf);
                        tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            df_g[(size_t)(32 * half + j) * kD] =
                                __float2bfloat16_rn(fmaf(K, __uint_as_float(rf[j]), __uint_as_float(uu[j])));
                    } else {
#pragma unroll 1
                        for (int t0 = 32 * half; t0 < 32 * half + 32; t0 += 4) {
                            uint32_t uu[4], rf[4];
                            tmem_ld4(tl + kColDQ + t0, uu);
                            tmem_ld4(tl + kColDKi + t0, rf);
                            tmem_wait_ld();
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                if (t0 + j < n_valid)
                                    df_g[(size_t)(t0 + j) * kD] =
                                        __float2bfloat16_rn(fmaf(K, __uint_as_float(rf[j]), __uint_as_float(uu[j])));
                        }
                    }
                }
                tc_fence_before_sync();
                mbar_arrive(&ctl->acc_free2);
                PT_MARK(4)
            }
        }
        PT_DUMP(status, 7, 5, tid == kWarpE3 * 32)
    } else if (warp < kWarpLoad) {
        // ================= O: causal masks, d_i =================
        const uint32_t tl = tmem + lane_base;
        PT_DECL
        int it = 0;
        Item im;
        for (int k = 0; next_item<kPersist>(&ctl->ring, k, abort_flag, first, im); ++k) {
            const size_t grow0 = (size_t)im.plane * wk.N + im.row0;     // first row of the item in the [planes * rows][128] view
            for (int c = (im.n + kC - 1) / kC - 1; c >= 0; --c, ++it) {
                const int n_valid = kRagged ? min(kC, im.n - c * kC) : kC;
                const size_t crow0 = grow0 + c * kC;
                // ---- tril(A), tril(dA) -> operand slabs: rows of A sit in lanes 0..63, rows of dA in lanes 64..127, a
                // warp converts its 32 rows.  The previous chunk's products have read the slabs: this role waited for
                // them before that chunk's d_i.
                mbar_wait(&ctl->barA, it & 1, abort_flag);
                tc_fence_after_sync();
#pragma unroll 1
                for (int hh = 0; hh < 2; ++hh)
                    tril_row_block(tl + (sub < 2 ? kColA : kColDA) + 32 * hh, sub < 2 ? pbuf : dpbuf, krow & 63, hh);
                fence_proxy_async_smem();
                tc_fence_before_sync();
                mbar_arrive(&ctl->pd_ready);
                mbar_wait(&ctl->barY2, it & 1, abort_flag);
                PT_MARK(0)
                PT_STAMP(status, 16, tid == kWarpO * 32 && it == 16)
                tc_fence_after_sync();
                // d_i = dV: lane = value dimension, columns = local times
                __nv_bfloat16 *di_g = d_i + crow0 * kD + krow;
                if (!kRagged || n_valid == kC) {
#pragma unroll 1
                    for (int b = 0; b < 8; ++b) {
                        uint32_t r[8];
                        tmem_ld8(tl + kColDV + 8 * b, r);
                        tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < 8; ++j) di_g[(size_t)(8 * b + j) * kD] = __float2bfloat16_rn(__uint_as_float(r[j]));
                    }
                } else {
#pragma unroll 1
                    for (int b = 0; b < 8; ++b) {
                        uint32_t r[8];
                        tmem_ld8(tl + kColDV + 8 * b, r);
                        tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (8 * b + j < n_valid) di_g[(size_t)(8 * b + j) * kD] = __float2bfloat16_rn(__uint_as_float(r[j]));
                    }
                }
                tc_fence_before_sync();
                mbar_arrive(&ctl->acc_freeV);
                PT_MARK(1)
                PT_STAMP(status, 17, tid == kWarpO * 32 && it == 16)
            }
        }
        PT_DUMP(status, 11, 4, tid == kWarpO * 32)
    } else if (warp == kWarpLoad) {
        // ================= L: TMA loads =================
        int n_stage = 0, n_v = 0, n_state = 0, n_raw = 0;       // fills asked for so far, per buffer
        struct Pos { int plane, row, slot; bool ok; };          // a chunk
        // The stage loads lead: they walk the items, take the next one as they get to the end of the current one, and
        // the other buffers' loads follow a chunk behind.
        Item im = first;
        int k = 0, c = (im.n + kC - 1) / kC;
        bool asked = false, ask_done = false;
        // The next chunk, of this item or the one behind it; not ok: that one is empty, or (im.id < 0) there is none.
        auto advance = [&]() -> Pos {
            for (int step = 0; step < 2 && im.id >= 0; ++step) {
                if (kPersist && c <= 2 && !ask_done) {          // two chunks ahead: the answer takes about a microsecond
                    asked = ring_ask(&ctl->ring, k + 1, &ctl->exact_flag, abort_flag);
                    ask_done = true;
                }
                if (c > 0) {
                    --c;
                    return Pos{im.plane, im.row0 + c * kC, im.slot0 + c, true};
                }
                if (!kPersist || step > 0) break;
                im = warp_uniform(*ring_take<kRagged>(&ctl->ring, ++k, asked, wk, abort_flag));
                c = (im.n + kC - 1) / kC;
                asked = ask_done = false;
            }
            return Pos{0, 0, 0, false};
        };
        // Any further: only with nothing of a chunk left to be asked for.  The roles cannot finish that chunk's item without
        // it, and an item kRing further on cannot be asked for before they have (tc_chunk.cuh).
        auto over_empty = [&](Pos p) -> Pos {
            while (kPersist && !p.ok && im.id >= 0) p = advance();
            return p;
        };
        auto issue_stage = [&](const Pos &p) {
            const int s = n_stage++ % kStages;
            uint8_t *st = smem + s * kStageBytes;
            mbar_arrive_expect_tx(&ctl->full[s], kStageBytes);
            for (int b = 0; b < 2; ++b) {
                tma_load_3d(st + kOffQ + b * kSS, &map_o, &ctl->full[s], 64 * b, p.row, p.plane);
                tma_load_3d(st + kOffK + b * kSlab, &map_f, &ctl->full[s], 64 * b, p.row, p.plane);
            }
            for (int b = 0; b < 2; ++b)
                tma_load_3d(st + kOffG + b * kSS, &map_dy, &ctl->full[s], 64 * b, p.row, p.plane);
        };
        auto issue_v = [&](const Pos &p) {
            ++n_v;
            mbar_arrive_expect_tx(&ctl->vfull, kTile);
            for (int b = 0; b < 2; ++b) tma_load_3d(vbuf + b * kSlab, &map_i, &ctl->vfull, 64 * b, p.row, p.plane);
        };
        auto issue_raw = [&](const Pos &p) {
            ++n_raw;
            mbar_arrive_expect_tx(&ctl->rawfull, 2 * kTile);
            tma_load_3d(smem + kOffRawO, &map_o_raw, &ctl->rawfull, 0, p.row, p.plane);
            tma_load_3d(smem + kOffRawF, &map_f_raw, &ctl->rawfull, 0, p.row, p.plane);
        };
        auto issue_state = [&](const Pos &p) {
            ++n_state;
            mbar_arrive_expect_tx(&ctl->sfull, kStateTile);
            for (int b = 0; b < 2; ++b)
                tma_load_3d(sbuf + b * kStateSlab, &map_saved, &ctl->sfull, 64 * b, 0, p.slot);
        };
        // Every buffer is refilled as soon as its last reader of the previous chunk is done; the waits below are in
        // the order in which those readers finish.  Pass `it` loads v, S' and the raw tiles of chunk `it`, and the stage of
        // chunk it + 1 (pass 0 also its own stage).
        // A barrier must never be armed twice within one phase.  Normally a buffer's previous fill has long been
        // consumed when its readers report; on the time-out exit those waits return at once, so before every
        // refill the previous fill is waited for explicitly (one poll that succeeds at once in normal running).
        Pos next = over_empty(advance());
        if (next.ok) issue_stage(next);
        for (int it = 0; next.ok; ++it) {
            if (it > 0) {
                mbar_wait(&ctl->barX, (it - 1) & 1, abort_flag);     // dA = dY V^T ...
                mbar_wait(&ctl->barY1, (it - 1) & 1, abort_flag);    // ... and dKs_inter^T = dS'' V^T have read v
                mbar_wait_drain(&ctl->vfull, (it - 1) & 1, 20000000ull);
            }
            issue_v(next);
            Pos after = advance();
            if (it > 0) {
                mbar_wait(&ctl->r_ready[(it - 1) & 1], ((it - 1) >> 1) & 1, abort_flag);   // R has read S' ...
                mbar_wait(&ctl->barY2, (it - 1) & 1, abort_flag);    // ... and so have the chunk's products;
                mbar_wait_drain(&ctl->sfull, (it - 1) & 1, 20000000ull);
            }
            issue_state(next);
            if (after.ok) {                                          // o, f, dy of the stage are free as well
                if (it > 0) mbar_wait_drain(&ctl->full[(it - 1) % kStages], ((it - 1) / kStages) & 1, 20000000ull);
                issue_stage(after);
            }
            if (it > 0) {
                mbar_wait(&ctl->raw_read, (it - 1) & 1, abort_flag); // the output warps are done with raw o, f
                mbar_wait_drain(&ctl->rawfull, (it - 1) & 1, 20000000ull);
            }
            issue_raw(next);
            if (kPersist && !after.ok) {
                after = over_empty(after);
                if (after.ok) {
                    if (it > 0) mbar_wait_drain(&ctl->full[(it - 1) % kStages], ((it - 1) / kStages) & 1, 20000000ull);
                    issue_stage(after);
                }
            }
            next = after;
        }
        ctl->l_stage = n_stage; ctl->l_v = n_v; ctl->l_state = n_state; ctl->l_raw = n_raw;
    } else {
        // ================= MX, MY1, MY2: MMA issue =================
        constexpr uint32_t idDS = idesc_bf16(128, 128, 1, 1);     // Qs^T (MN-major) x dY (MN-major)
        constexpr uint32_t idKK = idesc_bf16(128, 64, 0, 0);      // dS'' x V^T, S' x dY^T (all K-major)
        constexpr uint32_t idMK = idesc_bf16(128, 64, 1, 0);      // dS''^T (MN) x Ks^T (K);  Ks^T (MN) x dP^T (K)
        constexpr uint32_t idMM = idesc_bf16(128, 64, 1, 1);      // Qs^T (MN) x dP (MN);  dY^T (MN) x P (MN)
        // descriptors once; K steps and stage changes only add to the 14-bit start-address field
        const uint32_t sm0 = smem_u32(smem);
        const uint64_t dqk0 = smem_desc_sw128(sm0 + kOffQ, 16, 1024), dqm0 = smem_desc_sw128(sm0 + kOffQ, kSS, 1024);
        const uint64_t dfk0 = smem_desc_sw128(sm0 + kOffK, 16, 1024), dfm0 = smem_desc_sw128(sm0 + kOffK, kSlab, 1024);
        const uint64_t dvk = smem_desc_sw128(smem_u32(vbuf), 16, 1024);
        const uint64_t dgk0 = smem_desc_sw128(sm0 + kOffG, 16, 1024), dgm0 = smem_desc_sw128(sm0 + kOffG, kSS, 1024);
        const uint64_t dsk = smem_desc_sw128(smem_u32(sbuf), 16, 1024);
        const uint64_t ddsk = smem_desc_sw128(smem_u32(dsbuf), 16, 1024), ddsm = smem_desc_sw128(smem_u32(dsbuf), kStateSlab, 1024);
        const uint64_t dpm = smem_desc_sw128(smem_u32(pbuf), kSlab, 1024);
        const uint64_t ddpk = smem_desc_sw128(smem_u32(dpbuf), 16, 1024), ddpm = smem_desc_sw128(smem_u32(dpbuf), kSlab, 1024);
        auto kmaj = [](int kk) { return (uint64_t)(((kk >> 2) * kSlab + (kk & 3) * 32) >> 4); };          // [64][128] tile
        auto kmaj_i = [](int kk) { return (uint64_t)(((kk >> 2) * kSS + (kk & 3) * 32) >> 4); };          // interleaved q / dy tile
        auto kmaj_s = [](int kk) { return (uint64_t)(((kk >> 2) * kStateSlab + (kk & 3) * 32) >> 4); };   // [128][128] tile
        PT_DECL
        if (warp == kWarpMmaX) {
            int it = 0;
            Item im;
            for (int k = 0; next_item<kPersist>(&ctl->ring, k, abort_flag, first, im); ++k) {
                for (int left = im.n; left > 0; left -= kC, ++it) {
                    const int s = it % kStages;
                    const uint64_t so = (uint64_t)s * (kStageBytes >> 4);
                    const uint64_t dqk = dqk0 + so, dqm = dqm0 + so, dfk = dfk0 + so, dgm = dgm0 + so;
                    mbar_wait(&ctl->full[s], (it / kStages) & 1, abort_flag);
                    mbar_wait(&ctl->t_done[s], (it / kStages) & 1, abort_flag);
                    PT_MARK(0)
                    if (it > 0) mbar_wait(&ctl->pd_ready, (it - 1) & 1, abort_flag);   // A, dA of the previous chunk read out
                    mbar_wait(&ctl->vfull, it & 1, abort_flag);
                    tc_fence_after_sync();
                    // A and dA first: they need the chunk's tiles but not dS'', and the masks and the products behind
                    // them do not have to wait for the rescaling of the state gradient (the other way round, with
                    // one barrier for all three: forward + backward of 128 units of 2048 tokens 206 instead of 203 us,
                    // 592 of 512 253 instead of 249).
                    // (Qs; dY) as one 128-row operand: (Qs; dY) Ks^T has A in lanes 0..63 and (Qs; dY) V^T has dA
                    // in lanes 64..127 (the other halves are not used), so every lane carries a row to mask
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        mma_bf16_ss(tmem + kColA, dqk + kmaj_i(kk), dfk + kmaj(kk), idKK, kk > 0);
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        mma_bf16_ss(tmem + kColDA, dqk + kmaj_i(kk), dvk + kmaj(kk), idKK, kk > 0);
                    mma_commit(&ctl->barA);
                    mbar_wait(&ctl->m_done, it & 1, abort_flag);          // dS'' in TMEM
                    PT_MARK(1)
                    PT_STAMP(status, 3, it == 16)
                    tc_fence_after_sync();
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)              // dS' = dS'' + Qs^T dY
                        mma_bf16_ss(tmem + kColDS, dqm + (uint64_t)(kk * 128), dgm + (uint64_t)(kk * 128), idDS, 1);
                    mma_commit(&ctl->barX);
                    PT_MARK(2)
                    PT_STAMP(status, 4, it == 16)
                }
            }
            PT_DUMP(status, 15, 3, true)
        } else if (warp == kWarpMmaY1) {
            int it = 0;
            Item im;
            for (int k = 0; next_item<kPersist>(&ctl->ring, k, abort_flag, first, im); ++k) {
                for (int left = im.n; left > 0; left -= kC, ++it) {
                    const int s = it % kStages;
                    const uint64_t so = (uint64_t)s * (kStageBytes >> 4);
                    const uint64_t dfk = dfk0 + so;
                    mbar_wait(&ctl->full[s], (it / kStages) & 1, abort_flag);
                    mbar_wait(&ctl->t_done[s], (it / kStages) & 1, abort_flag);
                    mbar_wait(&ctl->m_done, it & 1, abort_flag);          // bf16 dS'' in shared memory
                    PT_MARK(0)
                    // dV^T first: its accumulator is free as soon as d_i of the previous chunk is out, long before the
                    // output warps have finished with dKs_inter^T
                    if (it > 0) mbar_wait(&ctl->acc_freeV, (it - 1) & 1, abort_flag);
                    tc_fence_after_sync();
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)              // dV^T = dS''^T Ks^T
                        mma_bf16_ss(tmem + kColDV, ddsm + (uint64_t)(kk * 128), dfk + kmaj(kk), idMK, kk > 0);
                    mma_commit(&ctl->barY1a);
                    mbar_wait(&ctl->vfull, it & 1, abort_flag);
                    if (it > 0) mbar_wait(&ctl->acc_free1, (it - 1) & 1, abort_flag);
                    PT_MARK(1)
                    PT_STAMP(status, 10, it == 16)
                    tc_fence_after_sync();
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)              // dKs_inter^T = dS'' V^T
                        mma_bf16_ss(tmem + kColDKx, ddsk + kmaj_s(kk), dvk + kmaj(kk), idKK, kk > 0);
                    mma_commit(&ctl->barY1);
                    PT_MARK(2)
                }
            }
            PT_DUMP(status, 18, 3, true)
        } else {
            int it = 0;
            Item im;
            for (int k = 0; next_item<kPersist>(&ctl->ring, k, abort_flag, first, im); ++k) {
                for (int left = im.n; left > 0; left -= kC, ++it) {
                    const int s = it % kStages;
                    const uint64_t so = (uint64_t)s * (kStageBytes >> 4);
                    const uint64_t dqm = dqm0 + so, dfm = dfm0 + so, dgk = dgk0 + so, dgm = dgm0 + so;
                    mbar_wait(&ctl->pd_ready, it & 1, abort_flag);   // tril(A), tril(dA); implies X and T of the chunk
                    mbar_wait(&ctl->barY1a, it & 1, abort_flag);          // dV^T += ... must follow dV^T = ...
                    PT_MARK(0)
                    PT_STAMP(status, 11, it == 16)
                    tc_fence_after_sync();
                    // dV^T first: it does not touch the columns that still hold the previous chunk's parked values
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)              // dV^T += dY^T A
                        mma_bf16_ss(tmem + kColDV, dgm + (uint64_t)(kk * 128), dpm + (uint64_t)(kk * 128), idMM, 1);
                    mbar_wait(&ctl->sfull, it & 1, abort_flag);
                    if (it > 0) mbar_wait(&ctl->acc_free2, (it - 1) & 1, abort_flag);
                    PT_MARK(1)
                    PT_STAMP(status, 12, it == 16)
                    tc_fence_after_sync();
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)              // dQs^T = Ks^T dA^T
                        mma_bf16_ss(tmem + kColDQ, dfm + (uint64_t)(kk * 128), ddpk + (uint64_t)(kk * 2), idMK, kk > 0);
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)              //        + S' dY^T
                        mma_bf16_ss(tmem + kColDQ, dsk + kmaj_s(kk), dgk + kmaj_i(kk), idKK, 1);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)              // dKs_intra^T = Qs^T dA
                        mma_bf16_ss(tmem + kColDKi, dqm + (uint64_t)(kk * 128), ddpm + (uint64_t)(kk * 128), idMM, kk > 0);
                    // barY2 stands for every product of the chunk: dKs_inter^T is another lane's, so wait for it first
                    // (it was issued when the output warps finished the previous chunk, well before this point)
                    mbar_wait(&ctl->barY1, it & 1, abort_flag);
                    mma_commit(&ctl->barY2);
                    PT_MARK(2)
                    PT_STAMP(status, 13, it == 16)
                }
            }
            PT_DUMP(status, 21, 3, true)
        }
        mma_commit(&ctl->drain);          // each of the three issuing lanes, after its loop
    }
    tc_fence_before_sync();
    __syncthreads();
    if (tid == 0) {
        // Nothing may be in flight when the CTA gives up its tensor and shared memory.  The three issuing lanes
        // committed once more after their loops: that barrier completes when every product they issued has.
        mbar_wait_drain(&ctl->drain, 0, 20000000ull);
        if (*abort_flag) {
            report_error(status, HGRN2_ERR_TIMEOUT, 2);
            if (kPersist && ctl->ring.asked > 0) mbar_wait_drain(&ctl->ring.answered, (ctl->ring.asked - 1) & 1, 20000000ull);
            // tiles asked for but never consumed may still be on their way into this CTA's shared memory
            const int ns = ctl->l_stage, nv = ctl->l_v, nst = ctl->l_state, nr = ctl->l_raw;
            for (int s = 0; s < kStages; ++s)
                if (ns > s) mbar_wait_drain(&ctl->full[s], ((ns - 1 - s) / kStages) & 1, 20000000ull);
            if (nv > 0) mbar_wait_drain(&ctl->vfull, (nv - 1) & 1, 20000000ull);
            if (nst > 0) mbar_wait_drain(&ctl->sfull, (nst - 1) & 1, 20000000ull);
            if (nr > 0) mbar_wait_drain(&ctl->rawfull, (nr - 1) & 1, 20000000ull);
        }
    }
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);

    // ---- exact path (see the forward kernel): flagged items, or their units, are redone from their inputs, their saved
    // chunk states and the gradient they started from by the pairwise-safe fp32 routine
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
            const Item im = claim ? cut_unit(wk, id, wk.G - 1) : work_item<kRagged>(wk, id);
            const size_t seq = ((size_t)im.plane * wk.N + im.row0) * kD, st = (size_t)im.unit * kD * kD;
            alu::bwd_unit<__nv_bfloat16, __nv_bfloat16, kEnc ? alu::kGateEnc : alu::kGateIsF>(
                reinterpret_cast<float *>(smem), ex.o + seq, ex.f + seq, ex.i + seq, ex.dy + seq,
                im.chain >= 0 ? chain + (size_t)im.chain * kD * kD : (dSN ? dSN + st : nullptr),
                ex.states + (size_t)im.slot0 * kD * kD, kC / kExactC, ex.scratch + (size_t)id * kD * kD, ex.d_o + seq,
                ex.d_f + seq, ex.d_i + seq, dS0 != nullptr && im.last ? dS0 + st : nullptr, im.n, kD, kD, kExactC,
                (im.n + kExactC - 1) / kExactC);
        }
        __syncthreads();                                             // the routine's shared memory, and the answer, are free
    }
}

}  // namespace

// Several items per CTA (kPersist) where they are short: 4736 units of 64 tokens 247 instead of 341 us, 2368 of 128 211 / 246,
// 1184 of 256 182 / 189, 789 of 384 182 / 186, but 592 of 512 171 / 162 and 296 of 1024 164 / 146: that instantiation's
// larger code takes up to a tenth more per chunk.
constexpr uint64_t kPersistChunks = 6;

cudaError_t launch_tc_bwd(const SeqArgs &a0)
{
    SeqArgs a = a0;
    const TcWork t = tc_work(a);
    if (t.items > 0x7fffffffull) return cudaErrorInvalidConfiguration;
    cudaError_t err;
    if (t.wk.G > 1) {
        // sequences cut into segments (chunk_tc_fwd.cu), mirrored: what every segment adds to the state gradient (it
        // holds for every f), chained in reverse
        err = launch_tc_state(true, a.o, a.f, a.dy, t, a.dS0 != nullptr, a.gate_enc, a.status, a.clear_status, a.start_aborted, a.stream);
        if (err != cudaSuccess) return err;
        if ((err = launch_seg_chain(true, t, a.dSN, a.dS0, a.stream)) != cudaSuccess) return err;
        a.clear_status = false;
    }
    CUtensorMap mo, mf, mi, mg, ms, mor, mfr;
    if (!make_map(&mo, a.o, t.planes, a.N, kC) || !make_map(&mf, a.f, t.planes, a.N, kC) || !make_map(&mi, a.i, t.planes, a.N, kC) ||
        !make_map(&mg, a.dy, t.planes, a.N, kC) || !make_map(&ms, a.states, t.slots, kD, kD) ||
        !make_map_plain(&mor, a.o, t.planes, a.N, kC) || !make_map_plain(&mfr, a.f, t.planes, a.N, kC))
        return cudaErrorInvalidValue;
    const bool ragged = a.N % kC != 0 || a.cu != nullptr, persist = t.items > (uint64_t)sm_count() && t.chunks <= kPersistChunks;
    auto kernel = a.gate_enc ? (ragged ? (persist ? tc_bwd_kernel<true, true, true> : tc_bwd_kernel<true, true, false>)
                                       : (persist ? tc_bwd_kernel<false, true, true> : tc_bwd_kernel<false, true, false>))
                             : (ragged ? (persist ? tc_bwd_kernel<true, false, true> : tc_bwd_kernel<true, false, false>)
                                       : (persist ? tc_bwd_kernel<false, false, true> : tc_bwd_kernel<false, false, false>));
    if ((err = ensure_dynamic_smem(reinterpret_cast<const void *>(kernel), kSmemBytes)) != cudaSuccess) return err;
    ExactArgs ex;
    ex.o = static_cast<const __nv_bfloat16 *>(a.o);
    ex.f = static_cast<const __nv_bfloat16 *>(a.f);
    ex.i = static_cast<const __nv_bfloat16 *>(a.i);
    ex.dy = static_cast<const __nv_bfloat16 *>(a.dy);
    ex.d_o = static_cast<__nv_bfloat16 *>(a.d_o);
    ex.d_f = static_cast<__nv_bfloat16 *>(a.d_f);
    ex.d_i = static_cast<__nv_bfloat16 *>(a.d_i);
    ex.states = reinterpret_cast<__nv_bfloat16 *>(a.states);
    ex.scratch = a.exact_scratch;
    return launch_chained(kernel, dim3((unsigned)t.items), kThreads, kSmemBytes, a.stream, mo, mf, mi, mg, ms, mor, mfr, a.totals, a.dSN, t.chain, t.redo, static_cast<__nv_bfloat16 *>(a.d_o), static_cast<__nv_bfloat16 *>(a.d_f), static_cast<__nv_bfloat16 *>(a.d_i), a.dS0, t.wk, a.status, a.clear_status ? 1 : 0, ex, a.start_aborted);
}

}  // namespace hgrn2
