// Pieces shared by the tensor-core forward and backward kernels: tile geometry, the in-place
// operand transform of one chunk, accumulator-to-operand conversions and the TMA tensor maps.
//
// Mid-chunk reference frame.  Within a chunk of C = 64 steps let b_j = sum_{r<=j} log f_r (per key
// dimension) and let m be the middle of the chunk (after local row 31).  Only two rescaled operands
// are formed:
//
//     Qs_t = q_t * exp(b_t - b_m)          Ks_s = k_s * exp(b_m - b_s)          (q = o, k = 1 - f)
//
// so that Qs_t . Ks_s = q_t k_s exp(b_t - b_s) for every pair, and with Pm = exp(b_m),
// E = exp(b_C - b_m) (per key dimension):
//
//     A  = tril(Qs Ks^T)                       S' = Diag(Pm) S_in      (state in the mid frame)
//     Y  = A V + Qs S'                         S_out = Diag(E) (S' + Ks^T V)
//
// The factors exp(b_t - b_m) are in-chunk cumulative PRODUCTS of f taken outward from the middle
// (the linear-space image of the log-space cumulative sum): rows after m multiply by prod f, rows
// before m divide by it.  The two factors of a pair can be represented only while the decay across each
// half of the chunk stays above 2^-100 per key dimension.  The totals Pm and E are floored there; a half whose
// total sits on the floor has left the range, which the state warps of both kernels see when they pick the
// totals up: they raise the CTA's exact-path flag and the kernels then redo the whole unit with the
// pairwise-safe fp32 routines of chunk_alu.cuh, which hold on all of [0, 1].  The running products inside a
// half are NOT floored (every one of them is at least as large as the half's total, so inside the range none
// needs it, and two instructions per element pair in the role that paces the forward are worth 5 % of it):
// outside the range they may reach zero and the operands Inf or NaN, which stay inside that unit's own
// accumulators and outputs, all of which the exact path then rewrites.
#pragma once

#include "tc_common.cuh"

namespace hgrn2 {
namespace tc {

constexpr int kC = 64;                          // chunk length
constexpr int kD = 128;                         // d_k = d_v
constexpr uint32_t kSlab = kC * 128;            // bytes of one slab of a [64][128] bf16 tile
constexpr uint32_t kTile = 2 * kSlab;           // one [64][128] bf16 tile
constexpr uint32_t kStateSlab = kD * 128;       // bytes of one slab of a [128][128] bf16 state copy
constexpr uint32_t kStateTile = 2 * kStateSlab;
constexpr float kProdFloor = 7.888609052210118e-31f;   // 2^-100
constexpr float kFactorSafe = 7.52316384526264e-37f;    // 2^-120: below it the product of two decay totals is applied in two steps
constexpr uint32_t kTmemCols = 512;
constexpr int kTransformThreads = 128;          // threads that run transform_stream together
// Saved-for-backward buffer of the tensor-core path, per (unit, chunk): the bf16 state S' in the mid
// frame ([128][128]), then, after all states, the decay totals Pm[128], E[128] (float) of every chunk.
constexpr size_t kSavedStateBytes = (size_t)kD * kD * 2;
constexpr size_t kSavedTotalsBytes = 2 * kD * sizeof(float);

// Optional per-role cycle counters of CTA 0 (development aid; compiled out unless HGRN2_PHASE_TIMING
// is defined).  Totals land in the padding words of the status block.
#ifdef HGRN2_PHASE_TIMING
#define PT_DECL long long pt_t0 = clock64(); long long pt_acc[12] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
#define PT_MARK(i) { const long long pt_t = clock64(); pt_acc[i] += pt_t - pt_t0; pt_t0 = pt_t; }
#define PT_DUMP(st, base, n, cond) if ((cond) && blockIdx.x == 0 && (st) != nullptr) { for (int pt_i = 0; pt_i < (n); ++pt_i) (st)->pad[(base) + pt_i] = (int)(pt_acc[pt_i] >> 4); }
#define PT_STAMP(st, idx, cond) if (blockIdx.x == 0 && (cond) && (st) != nullptr) (st)->pad[30 + (idx)] = (int)(clock64() & 0x3fffffff);
#else
#define PT_STAMP(st, idx, cond)
#define PT_DECL
#define PT_MARK(i)
#define PT_DUMP(st, base, n, cond)
#endif

// Signed gate encoding (kEnc): bits of one bf16 value in the low half of w -> f and k = 1 - f.  Sign clear: the
// magnitude is f; sign set: the magnitude is k (so the neutral token f = 1, k = 0 is 0x8000).
__device__ __forceinline__ void gate_decode(uint32_t w, float &f, float &k)
{
    const float m = __uint_as_float((w & 0x7FFFu) << 16);
    const bool is_k = (w & 0x8000u) != 0u;
    f = is_k ? 1.0f - m : m;
    k = is_k ? m : 1.0f - m;
}

__device__ __forceinline__ float rcp_fast(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ uint4 pack8(const uint32_t *r)
{
    uint4 w;
    w.x = pack_bf16(__uint_as_float(r[0]), __uint_as_float(r[1]));
    w.y = pack_bf16(__uint_as_float(r[2]), __uint_as_float(r[3]));
    w.z = pack_bf16(__uint_as_float(r[4]), __uint_as_float(r[5]));
    w.w = pack_bf16(__uint_as_float(r[6]), __uint_as_float(r[7]));
    return w;
}

// In-place rescaling of the raw o and f tiles of one chunk into Qs and Ks (see the file header).
// Run by 128 threads with no synchronisation among them: thread = one column pair x one half of the
// chunk.  The half before the middle walks its rows downwards from row 31, the half after it walks
// upwards from row 32, each carrying the running product of f, so only a few rows are live.  Rows are
// handled in batches of eight, and the loads of the next batch are issued before the stores of the
// current one (the tiles are rewritten in place, so the compiler would otherwise serialise every
// load behind the previous row's stores).  Pm (product over rows 0..31) and E (product over rows
// 32..63) of the chunk are left in pm[128] and ee[128] (shared memory) and / or pm_g[128], ee_g[128]
// (global memory); either pair may be null.  kEnc: the gate tile holds the SMALLER of f and k = 1 - f, with the sign bit set when it is k
// (gate_decode below).  The gated entry points hand the kernels that: bf16 then resolves the gate to 2^-9 of
// min(f, 1 - f) at both ends of [0, 1], whereas a bf16 f close to 1 would distort every decay product.
template <bool kUp, uint32_t kQSlabStride, uint32_t kFSlabStride, bool kEnc>
__device__ __forceinline__ void transform_half(uint8_t *qbuf, uint8_t *fbuf, float *tot, float *tot_g, int p)
{
    const int col = 2 * p;
    const int jch = (col & 63) >> 3;
    const uint32_t base = (col >> 6) * kQSlabStride + (col & 7) * 2;
    if (kFSlabStride != kQSlabStride && (col >> 6)) fbuf -= kQSlabStride - kFSlabStride;   // offsets below are the q tile's
    uint32_t xo[8];
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) xo[jj] = base + ((jch ^ jj) << 4);
    auto row_of = [](int i) { return kUp ? 32 + i : 31 - i; };     // i-th row visited
    uint32_t fw[8], qw[8], fn[8], qn[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int r = row_of(j);
        const uint32_t off = xo[r & 7] + r * 128;
        fn[j] = *reinterpret_cast<const uint32_t *>(fbuf + off);
        qn[j] = *reinterpret_cast<const uint32_t *>(qbuf + off);
    }
    float a0 = 1.f, a1 = 1.f;
#pragma unroll 1
    for (int b = 0; b < 4; ++b) {      // kept rolled: the body is long and every transform warp streams through it
#pragma unroll
        for (int j = 0; j < 8; ++j) { fw[j] = fn[j]; qw[j] = qn[j]; }
        if (b < 3) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int r = row_of(8 * (b + 1) + j);
                const uint32_t off = xo[r & 7] + r * 128;
                fn[j] = *reinterpret_cast<const uint32_t *>(fbuf + off);
                qn[j] = *reinterpret_cast<const uint32_t *>(qbuf + off);
            }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int r = row_of(8 * b + j);
            const uint32_t off = xo[r & 7] + r * 128;
            float f0, f1, k0 = 0.f, k1 = 0.f;
            if (kEnc) {
                gate_decode(fw[j], f0, k0);
                gate_decode(fw[j] >> 16, f1, k1);
            } else {
                f0 = bf16_lo(fw[j]);
                f1 = bf16_hi(fw[j]);
            }
            if (kUp) { a0 *= f0; a1 *= f1; }
            const float i0 = rcp_fast(a0), i1 = rcp_fast(a1);            // no floor: see the file header
            const float sq0 = kUp ? a0 : i0, sq1 = kUp ? a1 : i1;
            const float sk0 = kUp ? i0 : a0, sk1 = kUp ? i1 : a1;
            if (!kUp) { a0 *= f0; a1 *= f1; }
            // packed bf16 arithmetic: the scale factors are rounded to bf16 first, then one bf16x2 multiply
            // (resp. fused multiply-add for k = 1 - f) produces the operand pair
            const uint32_t sqp = pack_bf16(sq0, sq1), skp = pack_bf16(sk0, sk1);
            *reinterpret_cast<uint32_t *>(qbuf + off) = mul_bf16x2(qw[j], sqp);
            *reinterpret_cast<uint32_t *>(fbuf + off) = kEnc ? mul_bf16x2(pack_bf16(k0, k1), skp)
                                                             : fma_bf16x2(fw[j], skp ^ 0x80008000u, skp);
        }
    }
    // the products only shrink along the walk, so the last one tells whether the half stayed inside the range
    const float2 t2 = make_float2(fmaxf(a0, kProdFloor), fmaxf(a1, kProdFloor));
    if (tot) *reinterpret_cast<float2 *>(tot + col) = t2;
    if (tot_g) *reinterpret_cast<float2 *>(tot_g + col) = t2;
}

// kQSlabStride, kFSlabStride: distance in bytes between the two 64-column slabs of the q tile and of the f tile.
template <bool kEnc, uint32_t kQSlabStride = kSlab, uint32_t kFSlabStride = kSlab>
__device__ __forceinline__ void transform_stream(uint8_t *qbuf, uint8_t *fbuf, float *pm, float *ee, float *pm_g,
                                                 float *ee_g, int tid)
{
    if (tid >> 6) transform_half<true, kQSlabStride, kFSlabStride, kEnc>(qbuf, fbuf, ee, ee_g, tid & 63);
    else          transform_half<false, kQSlabStride, kFSlabStride, kEnc>(qbuf, fbuf, pm, pm_g, tid & 63);
}

// A partial chunk: the rows at or beyond n_valid (zeros, or in a packed batch the next sequence's tokens) become the
// neutral token f = 1, o = 0, each thread in what it is about to transform.  Done in the tiles and not in the transform's
// registers, which would cost two selects per row pair of every chunk or a second copy of its code.
template <bool kEnc, uint32_t kQSlabStride = kSlab, uint32_t kFSlabStride = kSlab>
__device__ __noinline__ void neutral_rows(uint8_t *qbuf, uint8_t *fbuf, int n_valid, int tid)
{
    const int col = 2 * (tid & 63), slab = col >> 6, lo = 32 * (tid >> 6);
    for (int r = max(n_valid, lo); r < lo + 32; ++r) {
        const uint32_t off = (((((col & 63) >> 3) ^ (r & 7)) << 4)) + (col & 7) * 2 + r * 128;
        *reinterpret_cast<uint32_t *>(fbuf + slab * kFSlabStride + off) = kEnc ? 0x80008000u : 0x3F803F80u;
        *reinterpret_cast<uint32_t *>(qbuf + slab * kQSlabStride + off) = 0u;
    }
}

// Causal mask + bf16 of 32 columns (32 * half ...) of one 64 x 64 fp32 accumulator in the M = 64
// layout (row r -> lane 32 * (r / 16) + r % 16) into a K-major slab.  `sub` = TMEM lane quarter.
__device__ __forceinline__ void tril_to_slab(uint32_t taddr, uint8_t *dstbuf, int sub, int half, int lane)
{
    uint32_t r[32];
    tmem_ld32(taddr, r);
    tmem_wait_ld();
    if (lane < 16) {
        const int t = 16 * sub + lane;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int s0 = 32 * half + 8 * j;
            uint32_t x[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) x[q] = (s0 + q <= t) ? r[8 * j + q] : 0u;
            *reinterpret_cast<uint4 *>(dstbuf + slab_chunk_off(t, 4 * half + j)) = pack8(x);
        }
    }
}

// Causal mask + bf16 of columns [32 * half, +32) of row t of a 64 x 64 fp32 accumulator whose rows sit one per
// TMEM lane (taddr = this thread's lane, first of the 32 columns) into a K-major slab.  The 32 threads of the
// warp hold 32 consecutive rows; a block that lies wholly above the diagonal is zero and is not read.
__device__ __forceinline__ void tril_row_block(uint32_t taddr, uint8_t *dstbuf, int t, int half)
{
    if (32 * half > (t | 31)) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            *reinterpret_cast<uint4 *>(dstbuf + slab_chunk_off(t, 4 * half + j)) = make_uint4(0u, 0u, 0u, 0u);
        return;
    }
    uint32_t r[32];
    tmem_ld32(taddr, r);
    tmem_wait_ld();
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int s0 = 32 * half + 8 * j;
        uint32_t x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) x[q] = (s0 + q <= t) ? r[8 * j + q] : 0u;
        *reinterpret_cast<uint4 *>(dstbuf + slab_chunk_off(t, 4 * half + j)) = pack8(x);
    }
}

// ---- work items ---------------------------------------------------------------------------------------
// A work item is a run of chunks that one CTA takes in one go: a whole sequence, or one segment of a sequence that was
// cut into G of them (why: chunk_tc_fwd.cu).  Item x of a launch (WorkArgs: common.cuh):
//   ordinary batch   x < main: unit x whole; beyond that item main + r * tail + t = segment r (Lc chunks, the last one
//                    shorter) of unit main + t;
//   packed batch     segment r of sequence b, head h at x = (b * G + r) * H + h; a sequence's segments have
//                    max(8, ceil(chunks / G)) chunks, those beyond its end are empty (G = 1: whole sequences).
// A cut unit has G chain slots, one per segment: first what the segment adds to the state (state-only pass), then, chained,
// the state at its start (backward: the gradient at its end).  Its S_N (dS_0) comes out of the chaining as well.
struct Item {
    int id;                        // -1: no more work
    int plane, row0, n;            // rows [row0, row0 + n) of plane `plane`
    int slot0;                     // first chunk-state slot
    int unit;                      // index of its state in S0, SN (dSN, dS0)
    int chain;                     // chain slot of the state (backward: the gradient) it starts from, -1: S0 (dSN)
    int last;                      // a whole unit: its final state is S_N (backward: its final gradient is dS_0)
};

// Sequence b of a packed batch has offsets that no tensor of N rows can have.
__device__ __forceinline__ bool packed_malformed(const WorkArgs &w, int b)
{
    return rows_malformed(w.cu[b], w.cu[b + 1], w.N);
}

// First CTA of a call's first kernel (all threads): the status block starts at zero, and malformed offsets are reported, of
// whatever sequence.  By this CTA because a CTA with nothing but a malformed sequence is through in a microsecond,
// and nothing orders its report behind the clearing (on a cold start it came first and was lost); what else is reported has
// the sweep of a chunk, or a wait that ran out, in front of it.
static __device__ __noinline__ void begin_call(StatusBlock *status, const int *cu, int B, int N)
{
    if (threadIdx.x == 0) clear_block(status);
    if (cu == nullptr) return;
    bool bad = false;
    for (int b = threadIdx.x; b < B; b += blockDim.x) bad |= rows_malformed(cu[b], cu[b + 1], N);
    if (__syncthreads_or(bad) && threadIdx.x == 0) report_error(status, HGRN2_ERR_INVALID_ARG, 4);
}

template <bool kPackedToo>
__device__ __forceinline__ Item work_item(const WorkArgs &w, int x)
{
    Item it;
    it.id = x;
    if (kPackedToo && w.cu != nullptr) {
        const int h = x % w.H, br = x / w.H, b = br / w.G, r = br - b * w.G;
        it.plane = h;
        it.unit = b * w.H + h;
        if (packed_malformed(w, b)) {                                // touch nothing
            it.row0 = it.n = it.slot0 = it.last = 0;
            it.chain = -1;
            return it;
        }
        const int start = w.cu[b], len = w.cu[b + 1] - start;
        int lo = 0, hi = len;
        if (w.G > 1) {
            const int Lc = max(8, ((len + kC - 1) / kC + w.G - 1) / w.G);
            lo = min(r * Lc * kC, len);
            hi = min(lo + Lc * kC, len);
        }
        it.row0 = start + lo;
        it.n = hi - lo;
        it.slot0 = h * w.spp + it.row0 / kC + br;
        it.last = w.G == 1;
        it.chain = w.G == 1 ? -1 : it.unit * w.G + r;
        return it;
    }
    if (x < w.main) {
        it.plane = it.unit = x;
        it.row0 = 0;
        it.n = w.N;
        it.slot0 = x * w.NC;
        it.chain = -1;
        it.last = 1;
        return it;
    }
    const int y = x - w.main, r = y / w.tail, t = y - r * w.tail;
    it.plane = it.unit = w.main + t;
    it.row0 = r * w.Lc * kC;
    it.n = min(w.Lc * kC, w.N - it.row0);
    it.slot0 = it.unit * w.NC + r * w.Lc;
    it.last = 0;
    it.chain = t * w.G + r;
    return it;
}

// The whole unit of which item x is a segment, starting from what its chain slot r holds.
__device__ __forceinline__ Item cut_unit(const WorkArgs &w, int x, int r)
{
    const int t = (x - w.main) % w.tail, unit = w.main + t;
    return Item{x, unit, 0, w.N, unit * w.NC, unit, t * w.G + r, 1};
}

// kPersist instantiations: a CTA works through several items, one after the other with all pipelines running on: the
// first is its own block index, the others are taken from CTAs of the grid that have not started (cluster launch
// control), so a launch of many short items pays a CTA's start-up and pipeline fill once per SM and keeps the hardware's
// dynamic balance.  The load warp takes them - as late as it can, when it asks for its current item's last tiles, so
// that an SM with a long item does not hoard another one - and publishes them in a ring that every role's warps
// read.  Item k + kRing is not published before every warp has given up item k, and any number of items in a row may be
// without tokens: so a role may hold back work that another one needs to finish an item (its last output, its last loads)
// only while it asks for the item right behind it.
// All of this is out of line: the roles run concurrently, and their combined code is about what the instruction
// cache holds (which is also why the other instantiations know nothing of it).
constexpr int kRing = 4;           // the load warp is at most this many items ahead of the slowest role
constexpr int kMaxCuts = 8;        // a CTA takes no further items once it has had this many segments
struct ItemRing {
    Item item[kRing], none;
    uint4 answer;                  // cluster launch control response (16-byte aligned)
    uint64_t full[kRing];          // load warp -> everyone
    uint64_t empty[kRing];         // one lane per warp -> load warp
    uint64_t answered;             // the hardware's response has landed
    int flagged[8];                // items (index + 1) whose decay left the operands' range, by position mod 8
    int cuts[kMaxCuts], n_cuts;    // the CTA's items that are segments (redo_claim)
    int asked;                     // responses asked for so far, for the abort epilogue
};
__device__ __forceinline__ void ring_init(ItemRing &q, int warps)
{
    for (int s = 0; s < kRing; ++s) {
        mbar_init(&q.full[s], 1);
        mbar_init(&q.empty[s], warps);
    }
    mbar_init(&q.answered, 1);
    for (int j = 0; j < 8; ++j) q.flagged[j] = 0;
    q.asked = 0;
    q.n_cuts = 0;
    q.none = Item{-1, 0, 0, 0, 0, 0, -1, 0};
}
// The same item in every lane, in a form that tells the compiler so: the loops over its chunks stay convergent code
// ("warp-wide issue", tc_common.cuh).
__device__ __forceinline__ Item warp_uniform(const Item &x)
{
    constexpr unsigned all = 0xffffffffu;
    return Item{__shfl_sync(all, x.id, 0),    __shfl_sync(all, x.plane, 0), __shfl_sync(all, x.row0, 0),  __shfl_sync(all, x.n, 0),
                __shfl_sync(all, x.slot0, 0), __shfl_sync(all, x.unit, 0),  __shfl_sync(all, x.chain, 0), __shfl_sync(all, x.last, 0)};
}
// Item k for a reading warp, in place: valid until the warp asks for item k + 1.  id < 0: no more work.  After an abort
// the warp is told so as one (the slot it would have read may be in flux).
static __device__ __noinline__ const Item *ring_next(ItemRing *q, int k, volatile int *abort_flag)
{
    const Item *it = &q->item[k % kRing];
    if (k > 0) {
        __syncwarp();
        if ((threadIdx.x & 31) == 0) mbar_arrive(&q->empty[(k - 1) % kRing]);
        mbar_wait(&q->full[k % kRing], (k / kRing) & 1, abort_flag);
        if (__any_sync(0xffffffffu, *abort_flag)) it = &q->none;
    }
    return it;
}
// Item k of a CTA whose first is `first`; false: no more.  Whole warp.
template <bool kPersist>
__device__ __forceinline__ bool next_item(ItemRing *q, int k, volatile int *abort_flag, const Item &first, Item &it)
{
    if constexpr (!kPersist) {
        it = first;
        return k == 0;
    } else {
        it = warp_uniform(*ring_next(q, k, abort_flag));
        return it.id >= 0;
    }
}
// Load warp: asks for item k (not before every warp has given up item k - kRing).  No more are taken once an item has been
// flagged for the exact path, which runs after the last one (the list of flagged items stays short), or after an abort.
static __device__ __noinline__ bool ring_ask(ItemRing *q, int k, volatile int *exact_flag, volatile int *abort_flag)
{
    if (k >= kRing) mbar_wait(&q->empty[k % kRing], (k / kRing - 1) & 1, abort_flag);
    if (__any_sync(0xffffffffu, *exact_flag || *abort_flag || q->n_cuts >= kMaxCuts)) return false;
    mbar_arrive_expect_tx(&q->answered, 16);
    if ((threadIdx.x & 31) == 0) {
        clc_try_cancel(&q->answer, &q->answered);
        ++q->asked;
    }
    __syncwarp();
    return true;
}
// Load warp: the answer to ring_ask (asked = its return value) becomes item k.
template <bool kPackedToo>
static __device__ __noinline__ const Item *ring_take(ItemRing *q, int k, bool asked, const WorkArgs &w, volatile int *abort_flag)
{
    int x = -1;
    if (asked) {
        mbar_wait(&q->answered, (q->asked - 1) & 1, abort_flag);
        if (!__any_sync(0xffffffffu, *abort_flag)) {
            x = clc_answer(&q->answer);
            fence_proxy_async_smem();                                // the answer has been read before the next one lands
        }
    }
    Item *it = &q->item[k % kRing];
    if ((threadIdx.x & 31) == 0) {
        if (x >= 0) *it = work_item<kPackedToo>(w, x);
        else *it = q->none;
        if (it->chain >= 0) q->cuts[q->n_cuts++] = x;
        mbar_arrive(&q->full[k % kRing]);
    }
    __syncwarp();
    return it;
}

// The exact path of a unit that runs as segments of whole chunks: the last of its G CTAs to finish redoes the whole unit,
// from its S_0 (dS_N), if any of them met a decay out of range, so S_N, dS_0 and every output are what they are for a unit
// that is not cut (redone segment by segment they would carry the state-only pass's bf16 operands).  redo = the
// unit's {flag, count}, zeroed by the chaining.  Called by one thread behind a barrier, its CTA's outputs complete.
__device__ __forceinline__ int redo_claim(int *redo, bool flagged, int G)
{
    if (flagged) atomicOr(redo, 1);
    __threadfence();
    if (atomicAdd(redo + 1, 1) != G - 1) return 0;
    __threadfence();
    return atomicOr(redo, 0);
}
__device__ __forceinline__ bool ring_flagged(const ItemRing &q, int id)
{
    bool hit = false;
    for (int j = 0; j < 8; ++j) hit |= q.flagged[j] == id + 1;
    return hit;
}

// ---- host side: tensor maps ---------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// [U][rows][128] bf16 tensor, tiles of [box_rows][64] with the 128-byte swizzle; rows beyond `rows`
// read as zero and are dropped on stores.
inline bool make_map(CUtensorMap *m, const void *base, uint64_t U, uint64_t rows, uint32_t box_rows)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {128, rows, U};
    cuuint64_t strides[2] = {256, rows * 256};
    cuuint32_t box[3] = {64, box_rows, 1};
    cuuint32_t es[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The same tensor as whole-width tiles of [box_rows][128] without swizzle (rows of 256 bytes, in order).
inline bool make_map_plain(CUtensorMap *m, const void *base, uint64_t U, uint64_t rows, uint32_t box_rows)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {128, rows, U};
    cuuint64_t strides[2] = {256, rows * 256};
    cuuint32_t box[3] = {128, box_rows, 1};
    cuuint32_t es[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace tc
}  // namespace hgrn2
