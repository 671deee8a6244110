// Chunkwise HGRN2 forward and backward on fp32 CUDA cores, parallel over the chunks of a sequence.
//
// This is the path for float32 I/O and for every head size the tensor-core kernels do not cover.  All products
// are fp32 FMAs on fp32 operands.  Chunk length 64; forward: local, scan, value kernels; backward: local, scan, value
// and key kernels.
//
//   local   one CTA per chunk: what the chunk adds to the state (forward) or state gradient (backward), into the
//           chunk's slot, and its total decay, into the chunk's rows of an output that a later kernel writes;
//   scan    chains the slots over a sequence's chunks, in place: afterwards a slot holds the state at the chunk's
//           start (the gradient at its end);
//   value, key   outputs of one chunk: chunks are independent once the boundary values are there.
//
// Packed batches have instances of their own: the search for a chunk's sequence in the others' code cost 2 % of
// 2 x 16 x 2048 float32.
//
// Formulas (q = o, k = 1 - f, v = i, b_t = sum_{r<=t} log f_r inside the chunk, m = after row 31,
// Pm = exp(b_m), E = exp(b_C - b_m); S_in, D_out = state at the chunk's start, state gradient at its end):
//
//   Qs_t = q_t exp(b_t - b_m),  Ks_s = k_s exp(b_m - b_s)
//   A = tril(Qs Ks^T)           Y  = A V + Qs (Pm S_in)
//   dA = tril(dY V^T)           dV = A^T dY + Ks (E D_out)
//   G  = dA Ks + Pm (dY S_in^T)         d_o = G exp(b_t - b_m)
//   J  = dA^T Qs,  Z = V D_out^T        dk  = (J + E Z) exp(b_m - b_s)
//   a = Qs G - Ks J,  e = Ks E Z,  R = Pm E sum_v D_out S_in
//   dg_t = sum_{j>=t} a_j + sum_{s<t} e_s + R,   d_f = dg / f - dk
//
// The decays are running products of f taken outwards from the middle of the chunk, so a factor is at most
// 32 steps long; while each half's total stays above 2^-100 everything is representable in fp32 and each term
// carries only the rounding of its own factors.  A chunk that leaves this range (f down to 0) forms its
// intra-chunk decays pairwise as exp(b_t - b_s) <= 1 instead, inside the same CTA (slower, exact everywhere);
// what crosses chunk boundaries only ever shrinks and needs no frame.
//
// What bounds these kernels is the rate at which shared-memory loads fill registers, one warp's 128 bytes per cycle,
// broadcast or not (measured: 4 cycles for any pattern of 16-byte loads).  A thread with a 4 x 4 block of a product loads 8
// values for 16 FMAs and is bound by them twice over; with 8 x 8, 16 values for 64 FMAs, loads and FMAs are level (alone
// on the SM: 46 and 64 TFLOP/s; the FMA pipes reach 72).  So the products of a chunk are dealt out to warps (A to some,
// the others' 64 x 64 blocks to pairs of warps) instead of every warp doing a small part of each, and operands are
// stored with the contracted index outermost, as rows of 16-byte pieces: a warp reads 4 pieces of one row and 8 of
// another, twice, per step.  Piece c of row r sits at c ^ (r / 4 % 8), which keeps the transposing stores free of bank
// conflicts.
#include "chunk_alu.cuh"

namespace hgrn2 {

namespace {

using alu::GateMode;
using alu::gate_values;
using alu::sigmoid_f;
using alu::value_of;

constexpr int kL = 64;              // tokens per chunk
constexpr int kW = 32;              // width of a slab of the contracted index
constexpr float kHalfFloor = kFMin; // 2^-100: the smallest half-chunk decay the mid-frame operands carry

struct Args {
    const void *o, *f, *i, *dy;
    const float *beta;              // gated: lower bounds [H][dk]
    const float *S0, *dSN;
    float *states, *dstates;        // boundary values, [slot][dk][dv]
    void *y, *d_o, *d_f, *d_i;
    float *SN, *dS0;
    float *dbeta;                   // gated backward: partial sums [slot][dk]
    const int *cu;                  // packed batch
    int B, H, N, NC, dk, dv;
    int spp;                        // packed: slots per head
    long long g0;                   // first unit (packed: head) of this launch
    StatusBlock *status;            // set: the launch's first CTA clears it
};

// A unit's rows, chunks, first boundary slot.  Plain layout: unit u owns rows [u N, u N + N), slots from
// (u - g0) NC.  Packed: head h, sequence b; slots from (h - g0) spp + cu[b] / 64 + b.
struct Where { long long row; int n, nc; long long slot, unit; };

__device__ __forceinline__ Where packed_where(const Args &a, int b, long long h)
{
    const int start = a.cu[b], end = a.cu[b + 1];
    const int n = rows_malformed(start, end, a.N) ? 0 : end - start;     // malformed offsets: touch nothing
    return Where{h * a.N + start, n, (n + kL - 1) / kL, (h - a.g0) * a.spp + start / kL + b, b * (long long)a.H + h};
}

template <typename T> __device__ __forceinline__ void store4(T *p, float a, float b, float c, float d);
template <> __device__ __forceinline__ void store4<float>(float *p, float a, float b, float c, float d)
{
    *reinterpret_cast<float4 *>(p) = make_float4(a, b, c, d);
}
template <> __device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16 *p, float a, float b, float c, float d)
{
    const __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
    *reinterpret_cast<uint2 *>(p) = make_uint2(reinterpret_cast<const uint32_t &>(lo), reinterpret_cast<const uint32_t &>(hi));
}

// Four consecutive elements of a sequence tensor as they sit in memory (one vector register set per load in flight).
template <typename T> struct Raw4;
template <> struct Raw4<float> { float4 v; };
template <> struct Raw4<__nv_bfloat16> { uint2 v; };
template <typename T> __device__ __forceinline__ Raw4<T> raw_load4(const T *p)
{
    Raw4<T> r;
    r.v = *reinterpret_cast<const decltype(r.v) *>(p);
    return r;
}
template <typename T> __device__ __forceinline__ Raw4<T> raw_zero4()
{
    Raw4<T> r;
    r.v = decltype(r.v){};
    return r;
}
__device__ __forceinline__ float4 widen(const Raw4<float> &r) { return r.v; }
__device__ __forceinline__ float4 widen(const Raw4<__nv_bfloat16> &r)
{
    return make_float4(__uint_as_float(r.v.x << 16), __uint_as_float(r.v.x & 0xFFFF0000u), __uint_as_float(r.v.y << 16),
                       __uint_as_float(r.v.y & 0xFFFF0000u));
}
template <int kMode> __device__ __forceinline__ float4 value4(float4 x)
{
    return make_float4(value_of<kMode>(x.x), value_of<kMode>(x.y), value_of<kMode>(x.z), value_of<kMode>(x.w));
}

// Offset (floats) of 16-byte piece c of row r in a tile of W floats per row.
template <int W> __device__ __forceinline__ int piece(int r, int c) { return r * W + ((c ^ ((r >> 2) & 7)) << 2); }
// Offset of element (r, x).
template <int W> __device__ __forceinline__ int elem(int r, int x) { return piece<W>(r, x >> 2) + (x & 3); }

// acc[m][n] += sum over rows x in [x0, x1) of A[x][m] B[x][n].  A thread's m: pieces mp and (MH = 2) mp + 4 of a row of A, its
// n: pieces np and (NH = 2) np + 8 of a row of B.  x0, x1 are multiples of 4.
template <int MH, int NH, int WA, int WB>
__device__ __forceinline__ void mul(float (&acc)[8][8], const float *A, int mp, const float *B, int np, int x0, int x1)
{
#pragma unroll 2
    for (int x = x0; x < x1; x += 4) {
        const int sw = (x >> 2) & 7;
        const float *a = A + x * WA, *b = B + x * WB;
        const int a0 = (mp ^ sw) << 2, a1 = ((mp + 4) ^ sw) << 2, b0 = (np ^ sw) << 2, b1 = ((np + 8) ^ sw) << 2;
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            float av[8];
            float2 bv[4];
            load4(a + y * WA + a0, reinterpret_cast<float(&)[4]>(av));
            if (MH == 2) load4(a + y * WA + a1, reinterpret_cast<float(&)[4]>(av[4]));
            load4(b + y * WB + b0, reinterpret_cast<float(&)[4]>(bv));
            if (NH == 2) load4(b + y * WB + b1, reinterpret_cast<float(&)[4]>(bv[2]));
#pragma unroll
            for (int i = 0; i < 4 * MH; ++i) {
                const float2 a2 = make_float2(av[i], av[i]);
#pragma unroll
                for (int j = 0; j < 2 * NH; ++j) {
                    const float2 d = fma_x2(a2, bv[j], make_float2(acc[i][2 * j], acc[i][2 * j + 1]));
                    acc[i][2 * j] = d.x;
                    acc[i][2 * j + 1] = d.y;
                }
            }
        }
    }
}
// acc[m][n] += sum_x A[m][x] B[n][x] over a slab of 32 x, both operands with the contracted index innermost: rows
// 4 (mp + 4 i) .. + 3 of A, rows 4 (np + 8 j) .. + 3 of B, [.][32].
template <int MH, int NH>
__device__ __forceinline__ void mul_rows(float (&acc)[8][8], const float *A, int mp, const float *B, int np)
{
    const float *a = A + 4 * mp * kW, *b = B + 4 * np * kW;
#pragma unroll 2
    for (int c = 0; c < kW / 4; ++c) {
        const int ca = (c ^ (mp & 7)) << 2, ca4 = (c ^ ((mp + 4) & 7)) << 2, cb = (c ^ (np & 7)) << 2;
        float av[4 * MH][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) load4(a + i * kW + ca, av[i]);
        if (MH == 2) {
#pragma unroll
            for (int i = 0; i < 4; ++i) load4(a + (16 + i) * kW + ca4, av[4 * (MH - 1) + i]);
        }
#pragma unroll
        for (int j = 0; j < 4 * NH; ++j) {
            float bv[4];
            load4(b + (j < 4 ? j : 28 + j) * kW + cb, bv);
#pragma unroll
            for (int i = 0; i < 4 * MH; ++i)
#pragma unroll
                for (int x = 0; x < 4; ++x) acc[i][j] = fmaf(av[i][x], bv[x], acc[i][j]);
        }
    }
}
// The products of mul (MH = NH = 2, or MH = 1) with m <= x (kLower) or m >= x only, every other one left out: a zero of a
// masked A does not hide an Inf or NaN in B, and no token may see one in a token that it does not depend on.
template <bool kLower, int MH, int WA, int WB>
__device__ __forceinline__ void mul_masked(float (&acc)[8][8], const float *A, int mp, const float *B, int np, int x0, int x1)
{
#pragma unroll 1
    for (int x = x0; x < x1; ++x) {
        float av[8], bv[8];
        load4(A + piece<WA>(x, mp), reinterpret_cast<float(&)[4]>(av));
        if (MH == 2) load4(A + piece<WA>(x, mp + 4), reinterpret_cast<float(&)[4]>(av[4]));
        load4(B + piece<WB>(x, np), reinterpret_cast<float(&)[4]>(bv));
        load4(B + piece<WB>(x, np + 8), reinterpret_cast<float(&)[4]>(bv[4]));
#pragma unroll
        for (int i = 0; i < 4 * MH; ++i) {
            const int m = 4 * mp + 4 * (i & 4) + (i & 3);
            if (kLower ? m <= x : m >= x)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
    }
}
// Whether rows [r0, r0 + rows) of B hold an Inf or NaN in this warp's columns (pieces 16 h .. 16 h + 15, np = 16 h + lane % 8).
template <int rows, int WB> __device__ __forceinline__ bool not_finite(const float *B, int r0, int np, int lane)
{
    float z = 0.f;
#pragma unroll
    for (int r = 0; r < rows; r += 4)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v[4];
            load4(B + piece<WB>(r0 + r + (lane >> 3), np + 8 * h), v);
#pragma unroll
            for (int j = 0; j < 4; ++j) z = fmaf(v[j], 0.f, z);
        }
    return __any_sync(0xFFFFFFFFu, z != 0.f);
}
__device__ __forceinline__ void zero(float (&acc)[8][8])
{
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
}
// First index of rows (columns) i .. i + 3 of a thread's block, i in {0, 4}.
__device__ __forceinline__ int at_m(int mp, int i) { return 4 * mp + 4 * i; }       // pieces mp, mp + 4
__device__ __forceinline__ int at_n(int np, int j) { return 4 * np + 8 * j; }       // pieces np, np + 8

// 1 / x to an ulp, for x well inside fp32's range (the running products below stay above 2^-100).
__device__ __forceinline__ float recip(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int n> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(n) : "memory"); }

// Whether a slot of a packed batch holds a chunk of sequence b.
__device__ __forceinline__ bool owns_slot(const int *cu, int b, int N, int slot)
{
    const int start = cu[b], end = cu[b + 1], c = slot - (start / kL + b);
    return !rows_malformed(start, end, N) && c >= 0 && c < (end - start + kL - 1) / kL;
}

// Which chunk blockIdx.x stands for: false = none (a slot of a packed batch that no chunk uses).  Whole warps.
template <bool kPacked> __device__ __forceinline__ bool chunk_of(const Args &a, Where &w, int &c)
{
    if constexpr (!kPacked) {
        const long long u = blockIdx.x / a.NC;
        c = blockIdx.x - (int)(u * a.NC);
        w = Where{(a.g0 + u) * a.N, a.N, a.NC, u * a.NC, a.g0 + u};
        return true;
    }
    const int h = blockIdx.x / a.spp, slot = blockIdx.x - h * a.spp;
    int lo = 0, hi = a.B - 1;                                         // the last sequence whose first slot is <= slot
    while (lo < hi) {
        const int mid = (lo + hi + 1) / 2;
        if (a.cu[mid] / kL + mid <= slot) lo = mid; else hi = mid - 1;
    }
    if (!owns_slot(a.cu, lo, a.N, slot)) {
        // Nobody's slot - or a malformed offset has misled the search, and the well-formed sequences must come out all the
        // same: every warp looks at all of them.
        unsigned hits = 0;
        for (lo = 0; lo < a.B; lo += 32) {
            const int b = lo + (threadIdx.x & 31);
            if ((hits = __ballot_sync(0xFFFFFFFFu, b < a.B && owns_slot(a.cu, b, a.N, slot))) != 0) break;
        }
        if (hits == 0) return false;
        lo += __ffs(hits) - 1;
    }
    w = packed_where(a, lo, a.g0 + h);
    c = slot - (a.cu[lo] / kL + lo);
    return true;
}

// Where a chunk's decay totals [dk] wait for the scan: in the chunk's rows of an output that is written later (y in the
// forward; d_o in the backward and in a forward that only re-creates states).  nullptr: the last chunk of a
// sequence has too few rows for them (fewer than 2 in float32 at dk <= dv, 16 at the very most); the scan then
// multiplies those rows' f itself.
template <typename T> __device__ __forceinline__ float *totals_at(const Args &a, bool bwd, const Where &w, int c)
{
    const bool in_y = !bwd && a.y != nullptr;
    const int width = in_y ? a.dv : a.dk, rows = min(kL, w.n - c * kL);
    if (rows * width * (int)sizeof(T) < a.dk * 4) return nullptr;
    return reinterpret_cast<float *>(static_cast<T *>(in_y ? a.y : a.d_o) + (w.row + (long long)c * kL) * width);
}

// Column of a 32-wide slab that a lane transforms: eight neighbouring lanes get columns four apart, so that their
// transposed 16-byte stores differ in r / 4 % 8.
__device__ __forceinline__ int lane_column(int lane) { return ((lane & 7) << 2) | (lane >> 3); }

// ---------------------------------------------------------------------------------------------------------------
// Local kernel.  forward: K^T V with K_s = k_s prod_{r>s} f_r; backward: Q^T dY with Q_t = q_t prod_{r<=t} f_r.
// CTA = chunk; TK x TV = the (padded) state; SPLIT groups of TK TV / 64 threads share the tokens (small states).
template <int TK, int TV, int SPLIT> struct LocalShape {
    static constexpr int NT = TK * TV / 64 * SPLIT, NW = NT / 32;
    static constexpr int CG = TK / 32, SEG = NW / CG, RP = kL / SEG;  // column groups, row segments, rows per segment
    static constexpr size_t kSmem = (size_t)(kL * (TK + TV) + SEG * TK) * sizeof(float);
};
template <typename T, int kMode, bool kPacked, bool kBwd, int TK, int TV, int SPLIT>
__global__ void __launch_bounds__(LocalShape<TK, TV, SPLIT>::NT)
fp32_local_kernel(const Args a)
{
    using P = LocalShape<TK, TV, SPLIT>;
    constexpr int RP = P::RP;
    extern __shared__ __align__(16) float sm[];
    float *sX = sm, *sV = sm + kL * TK, *sprod = sV + kL * TV;
    chain_wait();
    if (a.status != nullptr && blockIdx.x == 0 && threadIdx.x == 0) clear_block(a.status);
    Where w;
    int c;
    if (!chunk_of<kPacked>(a, w, c)) return;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int rows = min(kL, w.n - c * kL);
    const long long row0 = w.row + (long long)c * kL;
    const int kx = 32 * (wid % P::CG) + lane_column(lane), seg = wid / P::CG;
    const bool kin = kx < a.dk;
    {
        const T *qg = static_cast<const T *>(a.o) + row0 * a.dk + kx, *fg = static_cast<const T *>(a.f) + row0 * a.dk + kx;
        const T *vg = static_cast<const T *>(kBwd ? a.dy : a.i) + row0 * a.dv;
        const float beta = kMode == alu::kGatePre && kin ? a.beta[(size_t)(w.unit % a.H) * a.dk + kx] : 0.f;
        constexpr int VP = TV / 4, VL = kL * VP / P::NT;
        T fr[RP], qr[kBwd ? RP : 1];
        Raw4<T> vr[VL];
#pragma unroll
        for (int r = 0; r < RP; ++r) {
            const int t = seg * RP + r;
            if (kin && t < rows) {
                fr[r] = fg[t * a.dk];
                if (kBwd) qr[kBwd ? r : 0] = qg[t * a.dk];
            }
        }
#pragma unroll
        for (int x = 0; x < VL; ++x) {
            const int t = (tid + x * P::NT) / VP, p = (tid + x * P::NT) % VP;
            vr[x] = t < rows && 4 * p < a.dv ? raw_load4(vg + t * a.dv + 4 * p) : raw_zero4<T>();
        }
        float fv[RP], xv[RP], h = 1.f;
#pragma unroll
        for (int r = 0; r < RP; ++r) {
            float qv = 0.f, kv = 0.f;
            fv[r] = 1.f;
            if (kin && seg * RP + r < rows) {
                gate_values<kMode>(kBwd ? load_f(&qr[kBwd ? r : 0]) : 0.f, load_f(&fr[r]), beta, qv, fv[r], kv);
                fv[r] = fmaxf(fv[r], kFMin);
            }
            xv[r] = kBwd ? qv : kv;
            h *= fv[r];
        }
        sprod[seg * TK + kx] = h;
#pragma unroll
        for (int x = 0; x < VL; ++x) {
            const int t = (tid + x * P::NT) / VP, p = (tid + x * P::NT) % VP;
            float4 v = widen(vr[x]);
            if (!kBwd) v = value4<kMode>(v);
            *reinterpret_cast<float4 *>(sV + piece<TV>(t, p)) = v;
        }
        __syncthreads();
        float run = 1.f, all = 1.f;
#pragma unroll
        for (int s = 0; s < P::SEG; ++s) {
            const float x = sprod[s * TK + kx];
            all *= x;
            if (kBwd ? s < seg : s > seg) run *= x;
        }
        if (seg == 0 && kin) {
            float *tot = totals_at<T>(a, kBwd, w, c);
            if (tot) tot[kx] = all;
        }
#pragma unroll
        for (int x = 0; x < RP; ++x) {
            const int r = kBwd ? x : RP - 1 - x;
            if (kBwd) run *= fv[r];
            sX[elem<TK>(seg * RP + r, kx)] = xv[r] * run;
            if (!kBwd) run *= fv[r];
        }
        __syncthreads();
    }
    constexpr int PW = P::NW / SPLIT;                                 // warps of one token group
    const int part = wid / PW, wsub = wid % PW;
    const int mp = 8 * (wsub % (TK / 32)) + (lane >> 3), np = 16 * (wsub / (TK / 32)) + (lane & 7);
    float acc[8][8];
    zero(acc);
    mul<2, 2, TK, TV>(acc, sX, mp, sV, np, part * (kL / SPLIT), (part + 1) * (kL / SPLIT));
    if (SPLIT == 2) {
        constexpr int HT = P::NT / 2;
        __syncthreads();
        if (part == 1) {
#pragma unroll
            for (int x = 0; x < 64; ++x) sm[x * HT + tid - HT] = acc[x >> 3][x & 7];
        }
        __syncthreads();
        if (part == 1) return;
#pragma unroll
        for (int x = 0; x < 64; ++x) acc[x >> 3][x & 7] += sm[x * HT + tid];
    }
    float *out = (kBwd ? a.dstates : a.states) + (size_t)(w.slot + c) * a.dk * a.dv;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int k = at_m(mp, i & 4) + (i & 3);
        if (k < a.dk) {
            if (4 * np < a.dv) store4(out + (size_t)k * a.dv + 4 * np, acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
            if (4 * np + 32 < a.dv) store4(out + (size_t)k * a.dv + 4 * np + 32, acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
        }
    }
}

// ---------------------------------------------------------------------------------------------------------------
// Scan kernel: a thread chains four neighbouring state elements over the chunks of one sequence (backward: in
// reverse), four chunks' loads ahead.  Bound by the slots' traffic, once in and once out.
constexpr int kScanThreads = 128, kScanAhead = 4;
template <typename T, int kMode, bool kBwd>
__global__ void __launch_bounds__(kScanThreads)
fp32_scan_kernel(const Args a)
{
    chain_wait();
    const Where w = a.cu == nullptr
        ? Where{(a.g0 + blockIdx.x) * a.N, a.N, a.NC, (long long)blockIdx.x * a.NC, a.g0 + blockIdx.x}
        : packed_where(a, blockIdx.x % a.B, a.g0 + blockIdx.x / a.B);
    const int e = (blockIdx.y * kScanThreads + threadIdx.x) * 4;
    const size_t ss = (size_t)a.dk * a.dv;
    if (e >= a.dk * a.dv) return;
    const int k = e / a.dv;
    float *slots = (kBwd ? a.dstates : a.states) + (size_t)w.slot * ss + e;
    const float *init = kBwd ? a.dSN : a.S0;
    float *fin = kBwd ? a.dS0 : a.SN;
    float S[4] = {0.f, 0.f, 0.f, 0.f};
    if (init != nullptr) load4(init + (size_t)w.unit * ss + e, S);
    for (int n0 = 0; n0 < w.nc; n0 += kScanAhead) {
        float x[kScanAhead][4], lam[kScanAhead];
#pragma unroll
        for (int j = 0; j < kScanAhead; ++j) {
            const int c = kBwd ? w.nc - 1 - n0 - j : n0 + j;
            lam[j] = 1.f;
            if (n0 + j < w.nc) {
                load4(slots + (size_t)c * ss, x[j]);
                const float *tot = totals_at<T>(a, kBwd, w, c);
                if (tot) lam[j] = tot[k];
                else
                    for (int t = c * kL; t < w.n; ++t) {
                        float qv, fv, kv;
                        gate_values<kMode>(0.f, load_f(static_cast<const T *>(a.f) + (w.row + t) * a.dk + k),
                                           kMode == alu::kGatePre ? a.beta[(size_t)(w.unit % a.H) * a.dk + k] : 0.f, qv, fv, kv);
                        lam[j] *= fmaxf(fv, kFMin);
                    }
            }
        }
#pragma unroll
        for (int j = 0; j < kScanAhead; ++j)
            if (n0 + j < w.nc) {
                const int c = kBwd ? w.nc - 1 - n0 - j : n0 + j;
                store4(slots + (size_t)c * ss, S[0], S[1], S[2], S[3]);
#pragma unroll
                for (int i = 0; i < 4; ++i) S[i] = fmaf(lam[j], S[i], x[j][i]);
            }
    }
    if (fin != nullptr) store4(fin + (size_t)w.unit * ss + e, S[0], S[1], S[2], S[3]);
}

// ---------------------------------------------------------------------------------------------------------------
// Value kernel.  kDV = false: Y = A V + X S_in; kDV = true: dV = A^T dY + X D_out, with X the frame-free operand of the
// state term: q_t prod_{r<=t} f_r, or k_s prod_{r>s} f_r.  CTA = chunk, NV = padded value columns.  The key dimension is
// the contracted index of A and of the state term and comes in slabs of 32, double buffered.  Warps 0-3 form A and
// prepare the next slab's operands (gates through registers; a lane = one column, a warp = two segments of eight
// rows); warps 4-7 do nothing but multiply, so the transform hides behind them and they need no registers for it.
template <int NV> struct ValueShape {
    static constexpr int MHY = NV / 64;                               // Y: four warps of 16 x 64, or of 32 x 64
    static constexpr int kTile = kW * kL;
    static constexpr int kStage = 3 * kTile + kW * NV;                // Qs, Ks, X [32][64], state [32][NV]
    static constexpr size_t kSmem = (2 * kStage + kTile + 2 * 8 * kW) * sizeof(float);
};
constexpr int kValueThreads = 256;

// the first four warps only
__device__ __forceinline__ void sync_first_half() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

template <typename T, int kMode, bool kPacked, bool kDV, int NV>
__global__ void __launch_bounds__(kValueThreads, 2)
fp32_value_kernel(const Args a)
{
    chain_wait();
    using P = ValueShape<NV>;
    constexpr int kTile = P::kTile;
    extern __shared__ __align__(16) float sm[];
    // stage 0 | b | stage 1: with the last slab in one stage, V or dY goes into the other one, then tril(A) into what is
    // left of that and b
    float *sB = sm + P::kStage, *sprod = sm + 2 * P::kStage + kTile;  // sprod [2][8][32]
    auto stage = [&](int j) { return sm + (j & 1) * (P::kStage + kTile); };
    Where w;
    int c;
    if (!chunk_of<kPacked>(a, w, c)) return;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int rows = min(kL, w.n - c * kL);
    const long long row0 = w.row + (long long)c * kL;
    const float *st = (kDV ? a.dstates : a.states) + (size_t)(w.slot + c) * a.dk * a.dv;
    const int nslab = (a.dk + kW - 1) / kW;
    float *sA = nslab & 1 ? sB : sm + kL * NV, *sW = nslab & 1 ? sB + kL * kL : sm;
    float acc[8][8];
    zero(acc);

    auto fetch_state = [&](int j) {       // warps 4-7
        float *sS = stage(j) + 3 * kTile;
#pragma unroll
        for (int x = 0; x < kW * NV / 4 / 128; ++x) {
            const int k = (tid - 128 + x * 128) / (NV / 4), p = (tid - 128 + x * 128) % (NV / 4);
            float *dst = sS + piece<NV>(k, p);
            if (j * kW + k < a.dk && 4 * p < a.dv) cp_async16(dst, st + (j * kW + k) * a.dv + 4 * p);
            else *reinterpret_cast<float4 *>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        cp_async_commit();
    };

    if (wid >= 4) {
        // ================= Y or dV =================
        const int wy = wid - 4;
        const int mp = P::MHY == 2 ? 8 * (wy & 1) + (lane >> 3) : 4 * wy + (lane >> 3);
        const int np = (P::MHY == 2 ? 16 * (wy >> 1) : 0) + (lane & 7);
        fetch_state(0);
        cp_async_wait<0>();
        __syncthreads();
        for (int j = 0; j < nslab; ++j) {
            if (j + 1 < nslab) fetch_state(j + 1);
            const float *s = stage(j);
            mul<P::MHY, 2, kL, NV>(acc, s + 2 * kTile, mp, s + 3 * kTile, np, 0, kW);
            cp_async_wait<0>();
            __syncthreads();
        }
        // only the tokens on the causal side of this warp's rows contribute
        const int m_low = P::MHY == 2 ? 32 * (wy & 1) : 16 * wy;
        const int x0 = kDV ? m_low : 0, x1 = kDV ? kL : m_low + 16 * P::MHY;
        if (not_finite<16 * P::MHY, NV>(sW, m_low, np, lane)) mul_masked<kDV, P::MHY, kL, NV>(acc, sA, mp, sW, np, x0, x1);
        else mul<P::MHY, 2, kL, NV>(acc, sA, mp, sW, np, x0, x1);
        T *yg = static_cast<T *>(kDV ? a.d_i : a.y) + row0 * a.dv;
#pragma unroll
        for (int i = 0; i < 4 * P::MHY; ++i) {
            const int t = at_m(mp, i & 4) + (i & 3);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int v = at_n(np, 4 * h);
                if (t >= rows || v >= a.dv) continue;
                if (kDV && kMode == alu::kGatePre) {                  // d silu(z) / dz = s (1 + z (1 - s)), s = sigmoid(z)
                    float z[4];
                    load4(static_cast<const T *>(a.i) + (row0 + t) * a.dv + v, z);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float sg = sigmoid_f(z[j]);
                        acc[i][4 * h + j] *= sg * (1.0f + z[j] * (1.0f - sg));
                    }
                }
                store4(yg + t * a.dv + v, acc[i][4 * h], acc[i][4 * h + 1], acc[i][4 * h + 2], acc[i][4 * h + 3]);
            }
        }
        return;
    }

    // ================= A, and the operands of the next slab =================
    const int mp = 4 * wid + (lane >> 3), np = lane & 7;
    const bool low = wid < 2;                                         // rows 0..31 of A: columns 32..63 lie above the diagonal
    const int col = lane_column(lane);
    const T *og = static_cast<const T *>(a.o) + row0 * a.dk + col, *fg = static_cast<const T *>(a.f) + row0 * a.dk + col;
    const float *beta = kMode == alu::kGatePre ? a.beta + (size_t)(w.unit % a.H) * a.dk + col : nullptr;
    T qr[2][8], fr[2][8];                                             // segments wid and wid + 4
    auto fetch_gates = [&](int k0) {
        if (k0 + col >= a.dk) return;
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int t = (wid + 4 * x) * 8 + r;
                if (t < rows) {
                    qr[x][r] = og[t * a.dk + k0];
                    fr[x][r] = fg[t * a.dk + k0];
                }
            }
    };
    auto gate = [&](int k0, int x, int r, float &qv, float &fv, float &kv) {
        qv = 0.f; kv = 0.f; fv = 1.f;
        if (k0 + col < a.dk && (wid + 4 * x) * 8 + r < rows) {
            gate_values<kMode>(load_f(&qr[x][r]), load_f(&fr[x][r]), kMode == alu::kGatePre ? beta[k0] : 0.f, qv, fv, kv);
            fv = fmaxf(fv, kFMin);
        }
    };
    // Operands of slab j from the gates in registers; true: out of range - then Qs, Ks hold q, k and sB holds b.
    auto prepare = [&](int j) -> bool {
        const int k0 = j * kW;
        float *sQ = stage(j), *sK = sQ + kTile, *sX = sK + kTile, *sp = sprod + (j & 1) * 8 * kW;
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            float h = 1.f, qv, fv, kv;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                gate(k0, x, r, qv, fv, kv);
                h *= fv;
            }
            sp[(wid + 4 * x) * kW + col] = h;
        }
        sync_first_half();
        float pm = 1.f, ee = 1.f, run0 = 1.f, run1 = 1.f;             // decays: both halves', rows behind segment wid, before wid + 4
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const float lo = sp[s * kW + col], hi = sp[(s + 4) * kW + col];
            pm *= lo;
            ee *= hi;
            if (s > wid) run0 *= lo;
            if (s < wid) run1 *= hi;
        }
        // every warp's lanes see all 32 columns, so the decision is the same in all four warps
        const bool out_of_range = __any_sync(0xFFFFFFFFu, fminf(pm, ee) < kHalfFloor);
        if (!out_of_range) {
#pragma unroll
            for (int h = 1; h >= 0; --h) {                            // rows 8 wid .. + 7, from the last backwards
                float Q[4], K[4], fv;
#pragma unroll
                for (int r = 3; r >= 0; --r) {
                    gate(k0, 0, 4 * h + r, Q[r], fv, K[r]);
                    Q[r] *= recip(run0);
                    K[r] *= run0;
                    run0 *= fv;
                }
                const int at = piece<kL>(col, 2 * wid + h);
                *reinterpret_cast<float4 *>(sQ + at) = make_float4(Q[0], Q[1], Q[2], Q[3]);
                *reinterpret_cast<float4 *>(sK + at) = make_float4(K[0], K[1], K[2], K[3]);
                *reinterpret_cast<float4 *>(sX + at) = kDV ? make_float4(K[0] * ee, K[1] * ee, K[2] * ee, K[3] * ee)
                                                           : make_float4(Q[0] * pm, Q[1] * pm, Q[2] * pm, Q[3] * pm);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {                             // rows 8 (wid + 4) .. + 7, forwards
                float Q[4], K[4], fv;
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    gate(k0, 1, 4 * h + r, Q[r], fv, K[r]);
                    run1 *= fv;
                    Q[r] *= run1;
                    K[r] *= recip(run1);
                }
                const int at = piece<kL>(col, 2 * (wid + 4) + h);
                *reinterpret_cast<float4 *>(sQ + at) = make_float4(Q[0], Q[1], Q[2], Q[3]);
                *reinterpret_cast<float4 *>(sK + at) = make_float4(K[0], K[1], K[2], K[3]);
                *reinterpret_cast<float4 *>(sX + at) = kDV ? make_float4(K[0] * ee, K[1] * ee, K[2] * ee, K[3] * ee)
                                                           : make_float4(Q[0] * pm, Q[1] * pm, Q[2] * pm, Q[3] * pm);
            }
        } else {
            sync_first_half();                                        // sp has been read
            // (every loop over the gates is unrolled: an index that is not a constant would put them in local memory)
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                float run = 0.f, qv, fv, kv;
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    gate(k0, x, r, qv, fv, kv);
                    run += logf(fv);
                    sB[elem<kL>(col, (wid + 4 * x) * 8 + r)] = run;
                }
                sp[(wid + 4 * x) * kW + col] = run;
            }
            sync_first_half();
            float total = 0.f;
            for (int s = 0; s < 8; ++s) total += sp[s * kW + col];
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                float base = 0.f, qv, fv, kv;
                for (int s = 0; s < wid + 4 * x; ++s) base += sp[s * kW + col];
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    gate(k0, x, r, qv, fv, kv);
                    const int at = elem<kL>(col, (wid + 4 * x) * 8 + r);
                    const float b = sB[at] + base;
                    sQ[at] = qv;
                    sK[at] = kv;
                    sB[at] = b;
                    sX[at] = kDV ? kv * expf(total - b) : qv * expf(b);
                }
            }
        }
        return out_of_range;
    };

    fetch_gates(0);
    bool pairwise = prepare(0);
    if (nslab > 1) fetch_gates(kW);
    __syncthreads();
    constexpr bool kDirect = sizeof(T) == 4 && (kDV || kMode != alu::kGatePre);
    constexpr int WL = kL * NV / 4 / 128;
    const T *wg = static_cast<const T *>(kDV ? a.dy : a.i) + row0 * a.dv;
    for (int j = 0; j < nslab; ++j) {
        const float *sQ = stage(j), *sK = sQ + kTile;
        const bool last = j + 1 == nslab;
        if (last && kDirect) {
#pragma unroll
            for (int x = 0; x < WL; ++x) {
                const int t = (tid + x * 128) / (NV / 4), p = (tid + x * 128) % (NV / 4);
                if (t < rows && 4 * p < a.dv) cp_async16(sW + piece<NV>(t, p), wg + t * a.dv + 4 * p);
                else *reinterpret_cast<float4 *>(sW + piece<NV>(t, p)) = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            cp_async_commit();
        }
        if (!pairwise) {
            if (low) mul<1, 1, kL, kL>(acc, sQ, mp, sK, np, 0, kW);
            else mul<1, 2, kL, kL>(acc, sQ, mp, sK, np, 0, kW);
        } else {
#pragma unroll 1
            for (int x = 0; x < kW; ++x)
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int jj = 0; jj < 8; ++jj) {
                        const int t = at_m(mp, 0) + i, s = at_n(np, jj & 4) + (jj & 3);
                        if (s <= t) {
                            const int at = elem<kL>(x, t), as = elem<kL>(x, s);
                            acc[i][jj] = fmaf(sQ[at] * sK[as], expf(sB[at] - sB[as]), acc[i][jj]);
                        }
                    }
        }
        if (!last) {
            if (pairwise) sync_first_half();                          // every warp is done with sB
            pairwise = prepare(j + 1);
            if (j + 2 < nslab) fetch_gates((j + 2) * kW);
        } else {
            // tril(A) with the contracted index outermost
            sync_first_half();
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int jj = 0; jj < 8; ++jj)
                    if (at_n(np, jj & 4) + (jj & 3) > at_m(mp, 0) + i) acc[i][jj] = 0.f;
            if (kDV) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        *reinterpret_cast<float4 *>(sA + piece<kL>(at_m(mp, 0) + i, np + 8 * h)) =
                            make_float4(acc[i][4 * h], acc[i][4 * h + 1], acc[i][4 * h + 2], acc[i][4 * h + 3]);
            } else {
#pragma unroll
                for (int jj = 0; jj < 8; ++jj)
                    *reinterpret_cast<float4 *>(sA + piece<kL>(at_n(np, jj & 4) + (jj & 3), mp)) =
                        make_float4(acc[0][jj], acc[1][jj], acc[2][jj], acc[3][jj]);
            }
            if (!kDirect) {
#pragma unroll 8
                for (int x = 0; x < WL; ++x) {
                    const int t = (tid + x * 128) / (NV / 4), p = (tid + x * 128) % (NV / 4);
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (t < rows && 4 * p < a.dv) v = widen(raw_load4(wg + t * a.dv + 4 * p));
                    if (!kDV) v = value4<kMode>(v);
                    *reinterpret_cast<float4 *>(sW + piece<NV>(t, p)) = v;
                }
            }
            cp_async_wait<0>();
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------------------------------------------
// Key kernel: d_o and d_f of one chunk and 64 key dimensions.  The value dimension is the contracted index of
// dA = dY V^T (warps 0-3), X = dY S_in^T (4, 5) and Z = V D_out^T (6, 7) and comes in slabs of 32, double buffered; then
// G = Pm X + dA Ks (4, 5) and J = dA^T Qs (6, 7); then the elementwise part and the scans along time, a thread per column
// and 16 rows.  float32 slabs come by cp.async as they lie in memory (products of rows, scalar FMAs: transposing them on
// the way in costs more registers than there are); bf16 has to pass through registers anyway and is transposed there.
constexpr int kKeyThreads = 256;
constexpr int kKTile = kW * kL;                                       // [64][32], or transposed [32][64]
constexpr int kSq = kL * kL;                                          // [64][64]
constexpr size_t kKSmem = (6 * kSq + 8 * kL + 2 * kL + 8 * kL) * sizeof(float);

template <typename T, int kMode, bool kPacked>
__global__ void __launch_bounds__(kKeyThreads, 2)
fp32_key_kernel(const Args a)
{
    chain_wait();
    extern __shared__ __align__(16) float sm[];
    float *sprod = sm + 6 * kSq;                                      // [8][64]
    float *sR = sprod + 8 * kL;                                       // [2][64]
    float *ssum = sR + 2 * kL;                                        // [2][4][64] segment sums of a and e
    Where w;
    int c;
    if (!chunk_of<kPacked>(a, w, c)) return;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int k0 = blockIdx.y * kL;
    const int rows = min(kL, w.n - c * kL);
    const long long row0 = w.row + (long long)c * kL;
    const size_t ss = (size_t)a.dk * a.dv;
    const int role = wid < 4 ? 0 : wid < 6 ? 1 : 2;                   // dA | X, G | Z, J
    const int wm = role == 0 ? wid : wid & 1;
    const int mp = (role == 0 ? 4 : 8) * wm + (lane >> 3), np = lane & 7;
    constexpr bool kWide = sizeof(T) == 4;
    const T *gg = static_cast<const T *>(a.dy) + row0 * a.dv, *vg = static_cast<const T *>(a.i) + row0 * a.dv;
    const float *Sg = a.states + (size_t)(w.slot + c) * ss + k0 * a.dv, *Dg = a.dstates + (size_t)(w.slot + c) * ss + k0 * a.dv;

    // the chunk's o and f for later, as they are, into what no slab uses: float32 o in the place of the decays (element
    // by element the same place), f in that of Z; bf16 o and f both in that of Z
    float *sC = sm + 4 * kSq, *sZ = sm + 5 * kSq;
    const T *og = static_cast<const T *>(a.o) + row0 * a.dk + k0, *fg = static_cast<const T *>(a.f) + row0 * a.dk + k0;
    T *rawo = reinterpret_cast<T *>(kWide ? sC : sZ), *rawf = reinterpret_cast<T *>(sZ) + (kWide ? 0 : kSq);
    auto raw_at = [&](int t, int kx) { return kWide ? elem<kL>(t, kx) : t * kL + kx; };
    {
        constexpr int PP = kWide ? 16 : 8, E = kL / PP;               // 16-byte pieces per row, elements per piece
#pragma unroll
        for (int x = 0; x < kL * PP / kKeyThreads; ++x) {
            const int t = (tid + x * kKeyThreads) / PP, q = (tid + x * kKeyThreads) % PP;
            if (t < rows && k0 + E * q < a.dk) {
                cp_async16(rawo + raw_at(t, E * q), og + t * a.dk + E * q);
                cp_async16(rawf + raw_at(t, E * q), fg + t * a.dk + E * q);
            }
        }
        cp_async_commit();
    }

    // stage: dY | V | S | D.  float32: thread = row (and row + 32) and piece; V through registers where it is activated.
    // bf16: thread = block of four rows x four values, threads 0..127 of dY and S, 128..255 of V and D.
    constexpr bool kDirectV = kMode != alu::kGatePre;
    const int lr = tid >> 3, lp = tid & 7, g4 = 4 * ((tid >> 3) & 15);
    const bool second = tid >= 128;
    Raw4<T> xr[4];
    float4 sr[kWide ? 1 : 4];
    auto fetch = [&](int j) {
        const int v = j * kW + 4 * lp;
        const bool vin = v < a.dv;
        if constexpr (kWide) {
            float *st = sm + (j & 1) * 4 * kKTile;
            const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const int r = lr + 32 * x, at = piece<kW>(r, lp);
                if (vin && r < rows) cp_async16(st + at, gg + r * a.dv + v);
                else *reinterpret_cast<float4 *>(st + at) = none;
                if (!kDirectV) xr[x] = vin && r < rows ? raw_load4(vg + r * a.dv + v) : raw_zero4<T>();
                else if (vin && r < rows) cp_async16(st + kKTile + at, vg + r * a.dv + v);
                else *reinterpret_cast<float4 *>(st + kKTile + at) = none;
                if (vin && k0 + r < a.dk) {
                    cp_async16(st + 2 * kKTile + at, Sg + r * a.dv + v);
                    cp_async16(st + 3 * kKTile + at, Dg + r * a.dv + v);
                } else {
                    *reinterpret_cast<float4 *>(st + 2 * kKTile + at) = none;
                    *reinterpret_cast<float4 *>(st + 3 * kKTile + at) = none;
                }
            }
            cp_async_commit();
        } else {
            const T *xg = second ? vg : gg;
            const float *sg = second ? Dg : Sg;
            const bool kin = k0 + g4 < a.dk;                          // dk is a multiple of 16
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                xr[r] = vin && g4 + r < rows ? raw_load4(xg + (g4 + r) * a.dv + v) : raw_zero4<T>();
                sr[r] = vin && kin ? *reinterpret_cast<const float4 *>(sg + (g4 + r) * a.dv + v) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    };
    auto put = [&](float *tile, float4 x0, float4 x1, float4 x2, float4 x3) {   // transposed: row = value, pieces of four rows
        float *d = tile + piece<kL>(4 * lp, g4 >> 2);
        *reinterpret_cast<float4 *>(d) = make_float4(x0.x, x1.x, x2.x, x3.x);
        *reinterpret_cast<float4 *>(d + kL) = make_float4(x0.y, x1.y, x2.y, x3.y);
        *reinterpret_cast<float4 *>(d + 2 * kL) = make_float4(x0.z, x1.z, x2.z, x3.z);
        *reinterpret_cast<float4 *>(d + 3 * kL) = make_float4(x0.w, x1.w, x2.w, x3.w);
    };
    fetch(0);

    float acc[8][8];
    zero(acc);
    float racc = 0.f;
    const int nslab = (a.dv + kW - 1) / kW;
    for (int j = 0; j < nslab; ++j) {
        float *sG = sm + (j & 1) * 4 * kKTile, *sV = sG + kKTile, *sS = sV + kKTile, *sD = sS + kKTile;
        if constexpr (kWide) {
            if (!kDirectV)
#pragma unroll
                for (int x = 0; x < 2; ++x)
                    *reinterpret_cast<float4 *>(sV + piece<kW>(lr + 32 * x, lp)) = value4<kMode>(widen(xr[x]));
            cp_async_wait<0>();
        } else {
            float4 x[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) x[r] = kMode == alu::kGatePre && second ? value4<kMode>(widen(xr[r])) : widen(xr[r]);
            put(second ? sV : sG, x[0], x[1], x[2], x[3]);
            put(second ? sD : sS, sr[0], sr[1], sr[2], sr[3]);
        }
        __syncthreads();          // the slab is complete, and every warp is done with the other stage
        if (j + 1 < nslab) fetch(j + 1);
        if (role == 0) {
            if constexpr (kWide) {
                if (wm < 2) mul_rows<1, 1>(acc, sG, mp, sV, np);      // columns 32..63 lie above the diagonal
                else mul_rows<1, 2>(acc, sG, mp, sV, np);
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    float s4[4], d4[4];
                    load4(sS + piece<kW>(tid >> 1, 4 * (tid & 1) + x), s4);
                    load4(sD + piece<kW>(tid >> 1, 4 * (tid & 1) + x), d4);
#pragma unroll
                    for (int y = 0; y < 4; ++y) racc = fmaf(s4[y], d4[y], racc);
                }
            } else {
                if (wm < 2) mul<1, 1, kL, kL>(acc, sG, mp, sV, np, 0, kW);
                else mul<1, 2, kL, kL>(acc, sG, mp, sV, np, 0, kW);
                const int x0 = 16 * (tid >> 6);
#pragma unroll
                for (int x = 0; x < 16; ++x) racc = fmaf(sS[elem<kL>(x0 + x, tid & 63)], sD[elem<kL>(x0 + x, tid & 63)], racc);
            }
        } else {
            if constexpr (kWide) mul_rows<2, 2>(acc, role == 1 ? sG : sV, mp, role == 1 ? sS : sD, np);
            else mul<2, 2, kL, kL>(acc, role == 1 ? sG : sV, mp, role == 1 ? sS : sD, np, 0, kW);
        }
    }
    float *sA = sm, *sAT = sm + kSq, *sQ = sm + 2 * kSq, *sK = sm + 3 * kSq;
    const float *beta = kMode == alu::kGatePre ? a.beta + (size_t)(w.unit % a.H) * a.dk + k0 : nullptr;
    cp_async_wait<0>();
    __syncthreads();                                                  // o and f are there; the slabs are free from here on
    // products of f over eight rows (this warp's segment), both column groups
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const int kx = lane + 32 * x;
        float h = 1.f;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            float qv = 0.f, kv = 0.f, fv = 1.f;
            if (k0 + kx < a.dk && wid * 8 + r < rows)
                gate_values<kMode>(0.f, load_f(rawf + raw_at(wid * 8 + r, kx)), kMode == alu::kGatePre ? beta[kx] : 0.f, qv, fv, kv);
            h *= fmaxf(fv, kFMin);
        }
        sprod[wid * kL + kx] = h;
    }
    if (role == 0) {
        sR[kWide ? (tid & 1) * kL + (tid >> 1) : tid] = racc;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (at_n(np, j & 4) + (j & 3) > at_m(mp, 0) + i) acc[i][j] = 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                *reinterpret_cast<float4 *>(sA + piece<kL>(at_m(mp, 0) + i, np + 8 * h)) =
                    make_float4(acc[i][4 * h], acc[i][4 * h + 1], acc[i][4 * h + 2], acc[i][4 * h + 3]);
                *reinterpret_cast<float4 *>(sAT + piece<kL>(at_n(np, 4 * h) + i, mp)) =
                    make_float4(acc[0][4 * h + i], acc[1][4 * h + i], acc[2][4 * h + i], acc[3][4 * h + i]);
            }
    }
    __syncthreads();
    bool below = false;
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const float *q = sprod + lane + 32 * x;
        below |= fminf(q[0] * q[kL] * q[2 * kL] * q[3 * kL], q[4 * kL] * q[5 * kL] * q[6 * kL] * q[7 * kL]) < kHalfFloor;
    }
    const bool out_of_range = __any_sync(0xFFFFFFFFu, below);         // the same in every warp
    float odd = 0.f;                                                  // not 0: Inf or NaN among this thread's Qs, Ks
#pragma unroll 1
    for (int x = 0; x < 2; ++x) {
        const int kx = lane + 32 * x;
        float qv[8], kv[8], fv[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            qv[r] = 0.f; kv[r] = 0.f; fv[r] = 1.f;
            const int t = wid * 8 + r;
            if (k0 + kx < a.dk && t < rows) {
                gate_values<kMode>(load_f(rawo + raw_at(t, kx)), load_f(rawf + raw_at(t, kx)),
                                   kMode == alu::kGatePre ? beta[kx] : 0.f, qv[r], fv[r], kv[r]);
                fv[r] = fmaxf(fv[r], kFMin);
            }
        }
        const float *pr = sprod + kx;
        if (out_of_range) {                                           // raw q, k and b
            float run = 0.f;
            for (int s = 0; s < wid; ++s)
                for (int r = 0; r < 8; ++r) {
                    float q_, f_ = 1.f, k_;
                    if (k0 + kx < a.dk && 8 * s + r < rows)
                        gate_values<kMode>(0.f, load_f(fg + (8 * s + r) * a.dk + kx), kMode == alu::kGatePre ? beta[kx] : 0.f, q_, f_, k_);
                    run += logf(fmaxf(f_, kFMin));
                }
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                run += logf(fv[r]);
                const int at = elem<kL>(wid * 8 + r, kx);
                sQ[at] = qv[r];
                sK[at] = kv[r];
                sC[at] = run;
            }
        } else if (wid >= 4) {
            float run = 1.f;
            for (int s = 4; s < wid; ++s) run *= pr[s * kL];
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                run *= fv[r];
                const int at = elem<kL>(wid * 8 + r, kx);
                const float Q = qv[r] * run, K = kv[r] * recip(run);
                odd = fmaf(Q, 0.f, fmaf(K, 0.f, odd));
                sQ[at] = Q;
                sK[at] = K;
                sC[at] = run;
            }
        } else {
            float run = 1.f;
            for (int s = wid + 1; s < 4; ++s) run *= pr[s * kL];
#pragma unroll
            for (int r = 7; r >= 0; --r) {
                const int at = elem<kL>(wid * 8 + r, kx);
                const float inv = recip(run);
                const float Q = qv[r] * inv, K = kv[r] * run;
                odd = fmaf(Q, 0.f, fmaf(K, 0.f, odd));
                sQ[at] = Q;
                sK[at] = K;
                sC[at] = inv;
                run *= fv[r];
            }
        }
    }
    const bool masked = __syncthreads_or(odd != 0.f) != 0;
    if (role == 2) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float4 *>(sZ + piece<kL>(at_m(mp, i & 4) + (i & 3), np + 8 * h)) =
                    make_float4(acc[i][4 * h], acc[i][4 * h + 1], acc[i][4 * h + 2], acc[i][4 * h + 3]);
        zero(acc);
    }
    if (!out_of_range) {
        if (role == 1) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float *q = sprod + at_n(np, j & 4) + (j & 3);
                const float pm = q[0] * q[kL] * q[2 * kL] * q[3 * kL];
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[i][j] *= pm;
            }
            if (masked) mul_masked<false, 2, kL, kL>(acc, sAT, mp, sK, np, 0, 32 * (wm + 1));
            else mul<2, 2, kL, kL>(acc, sAT, mp, sK, np, 0, 32 * (wm + 1));
        } else if (role == 2) {
            if (masked) mul_masked<true, 2, kL, kL>(acc, sA, mp, sQ, np, 32 * wm, kL);
            else mul<2, 2, kL, kL>(acc, sA, mp, sQ, np, 32 * wm, kL);
        }
        __syncthreads();
    }
    // G (out of range: X) and J where dA was; out of range dA stays
    if (role == 1 || (role == 2 && !out_of_range)) {
        float *dst = role == 1 ? sAT : sA;
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float4 *>(dst + piece<kL>(at_m(mp, i & 4) + (i & 3), np + 8 * h)) =
                    make_float4(acc[i][4 * h], acc[i][4 * h + 1], acc[i][4 * h + 2], acc[i][4 * h + 3]);
    }
    // ---- elementwise part and scans along time: thread = one column, 16 rows
    const int col = tid & 63, q4 = tid >> 6;
    const bool cin = k0 + col < a.dk;
    T fr[16];
    if (cin) {
        const T *fc = fg + (16 * q4) * a.dk + col;
#pragma unroll
        for (int r = 0; r < 16; ++r)
            if (16 * q4 + r < rows) fr[r] = fc[r * a.dk];
    }
    __syncthreads();
    T *do_g = static_cast<T *>(a.d_o) + row0 * a.dk + k0 + col;
    float av[16], ev[16], dk[16], sa = 0.f, se = 0.f, lamC;
    if (!out_of_range) {
        const float *q = sprod + col;
        const float ee = q[4 * kL] * q[5 * kL] * q[6 * kL] * q[7 * kL];
        lamC = q[0] * q[kL] * q[2 * kL] * q[3 * kL] * ee;
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const int t = 16 * q4 + r, at = elem<kL>(t, col);
            const float G = sAT[at], J = sA[at], ez = ee * sZ[at], K = sK[at], C = sC[at];
            av[r] = sQ[at] * G - K * J;
            ev[r] = K * ez;
            dk[r] = (J + ez) * recip(C);
            if (cin && t < rows) {
                float dq = C * G;
                if (kMode == alu::kGatePre) {
                    const float s = sigmoid_f(load_f(og + t * a.dk + col));
                    dq *= s * (1.0f - s);
                }
                store_f(do_g + t * a.dk, dq);
            }
        }
    } else {                                                          // pairwise decays
        const float bC = sC[elem<kL>(kL - 1, col)];
        lamC = expf(bC);
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const int t = 16 * q4 + r, at = elem<kL>(t, col);
            const float b = sC[at];
            float dq = 0.f, J = 0.f;
#pragma unroll 1
            for (int x = 0; x < kL; ++x) {
                const int ax = elem<kL>(x, col);
                if (x <= t) dq = fmaf(sA[elem<kL>(t, x)] * sK[ax], expf(b - sC[ax]), dq);
                if (x >= t) J = fmaf(sA[elem<kL>(x, t)] * sQ[ax], expf(sC[ax] - b), J);
            }
            dq = fmaf(expf(b), sAT[at], dq);
            const float ik = expf(bC - b) * sZ[at];
            av[r] = sQ[at] * dq - sK[at] * J;
            ev[r] = sK[at] * ik;
            dk[r] = J + ik;
            if (cin && t < rows) {
                if (kMode == alu::kGatePre) {
                    const float s = sigmoid_f(load_f(og + t * a.dk + col));
                    dq *= s * (1.0f - s);
                }
                store_f(do_g + t * a.dk, dq);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        sa += av[r];
        se += ev[r];
    }
    ssum[q4 * kL + col] = sa;
    ssum[(4 + q4) * kL + col] = se;
    __syncthreads();
    float suf = lamC * (sR[col] + sR[kL + col]), pre = 0.f;           // R, then the later segments' a; the earlier segments' e
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        if (s > q4) suf += ssum[s * kL + col];
        if (s < q4) pre += ssum[(4 + s) * kL + col];
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) {                                    // exclusive prefix of e
        const float x = ev[r];
        ev[r] = pre;
        pre += x;
    }
    float dbeta = 0.f;
    if (cin) {
        T *df_g = static_cast<T *>(a.d_f) + row0 * a.dk + k0 + col;
        const float bt = kMode == alu::kGatePre ? beta[col] : 0.f;
#pragma unroll
        for (int r = 15; r >= 0; --r) {
            const int t = 16 * q4 + r;
            suf += av[r];
            if (t < rows) {
                const float fraw = load_f(&fr[r]);
                float q_, f_, k_;
                gate_values<kMode>(0.f, fraw, bt, q_, f_, k_);
                float d = (ev[r] + suf) * recip(fmaxf(f_, kFMin)) - dk[r];
                if (kMode == alu::kGatePre) {         // f = beta + (1 - beta) g:  df/dzf = (1 - beta) g (1 - g),  df/dbeta = 1 - g
                    const float g = sigmoid_f(fraw);
                    dbeta += d * (1.0f - g);
                    d *= (1.0f - bt) * g * (1.0f - g);
                }
                store_f(df_g + t * a.dk, d);
            }
        }
    }
    if (kMode == alu::kGatePre && a.dbeta != nullptr) {
        __syncthreads();                                              // ssum has been read
        ssum[q4 * kL + col] = dbeta;
        __syncthreads();
        if (tid < kL && k0 + tid < a.dk)
            a.dbeta[(size_t)(w.slot + c) * a.dk + k0 + tid] =
                (ssum[tid] + ssum[kL + tid]) + (ssum[2 * kL + tid] + ssum[3 * kL + tid]);
    }
}

// Every launch's x dimension is a number of slots or units.
bool grid_ok(const SeqArgs &s)
{
    const long long g = s.cu ? s.H : (long long)s.B * s.H, per = s.cu ? (long long)s.N / kL + s.B + 1 : (s.N + kL - 1ll) / kL;
    return per <= 0x7fffffff && g <= 0x7fffffff / per;
}
long long slots_per_group(const Args &a) { return a.cu ? a.spp : a.NC; }
long long units_per_group(const Args &a) { return a.cu ? a.B : 1; }

template <typename T, int kMode, bool kPacked, bool kBwd, int TK, int TV, int SPLIT>
cudaError_t launch_local_t(const Args &a, long long chunks, cudaStream_t stream)
{
    using P = LocalShape<TK, TV, SPLIT>;
    auto kernel = fp32_local_kernel<T, kMode, kPacked, kBwd, TK, TV, SPLIT>;
    cudaError_t err = ensure_dynamic_smem(reinterpret_cast<const void *>(kernel), P::kSmem);
    if (err != cudaSuccess) return err;
    return launch_chained(kernel, dim3((unsigned)chunks), P::NT, P::kSmem, stream, a);
}

// Boundary values of `groups` groups: every chunk's own contribution, then the chain over each sequence.
template <typename T, int kMode, bool kPacked, bool kBwd>
cudaError_t launch_state(const Args &a, long long groups, cudaStream_t stream)
{
    const long long chunks = groups * slots_per_group(a);
    cudaError_t err;
    if (a.dk > 64)
        err = a.dv > 64 ? launch_local_t<T, kMode, kPacked, kBwd, 128, 128, 1>(a, chunks, stream)
                        : launch_local_t<T, kMode, kPacked, kBwd, 128, 64, 2>(a, chunks, stream);
    else
        err = a.dv > 64 ? launch_local_t<T, kMode, kPacked, kBwd, 64, 128, 2>(a, chunks, stream)
                        : launch_local_t<T, kMode, kPacked, kBwd, 64, 64, 2>(a, chunks, stream);
    if (err != cudaSuccess) return err;
    const unsigned blocks = (a.dk * a.dv / 4 + kScanThreads - 1) / kScanThreads;
    return launch_chained(fp32_scan_kernel<T, kMode, kBwd>, dim3((unsigned)(groups * units_per_group(a)), blocks), kScanThreads, 0,
                          stream, a);
}

template <typename T, int kMode, bool kPacked, bool kDV, int NV>
cudaError_t launch_value_t(const Args &a, long long chunks, cudaStream_t stream)
{
    using P = ValueShape<NV>;
    auto kernel = fp32_value_kernel<T, kMode, kPacked, kDV, NV>;
    cudaError_t err = ensure_dynamic_smem(reinterpret_cast<const void *>(kernel), P::kSmem);
    if (err != cudaSuccess) return err;
    return launch_chained(kernel, dim3((unsigned)chunks), kValueThreads, P::kSmem, stream, a);
}
template <typename T, int kMode, bool kPacked, bool kDV>
cudaError_t launch_value(const Args &a, long long chunks, cudaStream_t stream)
{
    return a.dv > 64 ? launch_value_t<T, kMode, kPacked, kDV, 128>(a, chunks, stream) : launch_value_t<T, kMode, kPacked, kDV, 64>(a, chunks, stream);
}

template <typename T, int kMode, bool kPacked>
cudaError_t launch_key(const Args &a, long long chunks, cudaStream_t stream)
{
    cudaError_t err = ensure_dynamic_smem(reinterpret_cast<const void *>(fp32_key_kernel<T, kMode, kPacked>), kKSmem);
    if (err != cudaSuccess) return err;
    return launch_chained(fp32_key_kernel<T, kMode, kPacked>, dim3((unsigned)chunks, (a.dk + kL - 1) / kL), kKeyThreads, kKSmem, stream, a);
}

// groups = independent groups a launch can be restricted to: units, or heads of a packed batch
long long group_count(const SeqArgs &s) { return s.cu ? s.H : (long long)s.B * s.H; }

Args make_args(const SeqArgs &s, const float *beta)
{
    Args a{};
    a.o = s.o; a.f = s.f; a.i = s.i; a.dy = s.dy;
    a.beta = beta;
    a.S0 = s.S0; a.dSN = s.dSN;
    a.y = s.y; a.d_o = s.d_o; a.d_f = s.d_f; a.d_i = s.d_i;
    a.SN = s.SN; a.dS0 = s.dS0;
    a.cu = s.cu;
    a.B = s.B; a.H = s.H; a.N = s.N; a.dk = s.dk; a.dv = s.dv;
    a.NC = (s.N + kL - 1) / kL;
    a.spp = s.cu ? s.N / kL + s.B + 1 : 0;
    return a;
}
// Slots the caller's buffers have room for: they are sized for the call's own chunk length C <= 64.
long long slots_at_hand(const SeqArgs &s)
{
    return group_count(s) * (s.cu ? s.N / s.C + s.B + 1ll : (s.N + s.C - 1) / s.C);
}
// Backward without saved states: groups whose two sets of boundary values fit the workspace's room together.
long long groups_per_round(const SeqArgs &s)
{
    const long long spg = s.cu ? s.N / kL + s.B + 1ll : (s.N + kL - 1) / kL, fit = slots_at_hand(s) / (2 * spg);
    return fit < group_count(s) ? fit : group_count(s);
}

template <typename T, int kMode, bool kPacked>
cudaError_t fwd_t(const SeqArgs &s, const float *beta)
{
    if (!grid_ok(s)) return cudaErrorInvalidConfiguration;
    Args a = make_args(s, beta);
    const long long g = group_count(s);
    a.states = s.states ? s.states : s.room;
    a.status = s.clear_status ? s.status : nullptr;
    cudaError_t err = launch_state<T, kMode, kPacked, false>(a, g, s.stream);
    a.status = nullptr;
    if (err != cudaSuccess || s.y == nullptr) return err;
    return launch_value<T, kMode, kPacked, false>(a, g * slots_per_group(a), s.stream);
}

template <typename T, int kMode, bool kPacked>
cudaError_t bwd_t(const SeqArgs &s, const float *beta, float *dbeta)
{
    if (!grid_ok(s)) return cudaErrorInvalidConfiguration;
    Args a = make_args(s, beta);
    const long long g = group_count(s), spg = slots_per_group(a);
    const size_t ss = (size_t)s.dk * s.dv;
    a.status = s.clear_status ? s.status : nullptr;
    a.dbeta = dbeta;
    // The workspace has room for one set of boundary values.  With the forward's at hand (s.states) it takes the
    // gradients'; otherwise the groups run in rounds that keep both of their sets there.
    const long long per = s.states ? g : groups_per_round(s);
    for (long long g0 = 0; g0 < g; g0 += per) {
        const long long n = g - g0 < per ? g - g0 : per;
        a.g0 = g0;
        a.states = s.states;
        a.dstates = s.room;
        cudaError_t err;
        if (!s.states) {
            a.states = s.room;
            a.dstates = s.room + (size_t)n * spg * ss;
            Args r = a;
            r.SN = nullptr;
            if ((err = launch_state<T, kMode, kPacked, false>(r, n, s.stream)) != cudaSuccess) return err;
            a.status = nullptr;
        }
        if ((err = launch_state<T, kMode, kPacked, true>(a, n, s.stream)) != cudaSuccess) return err;
        a.status = nullptr;
        if ((err = launch_value<T, kMode, kPacked, true>(a, n * spg, s.stream)) != cudaSuccess) return err;
        if ((err = launch_key<T, kMode, kPacked>(a, n * spg, s.stream)) != cudaSuccess) return err;
        if (dbeta) a.dbeta += (size_t)n * spg * s.dk;
    }
    return cudaSuccess;
}

}  // namespace

// False for one unit (one head of a packed batch) without saved states whose workspace has no room for both sets of
// boundary values: that call runs on the serial kernels, which keep the state gradient on chip.
bool fp32_bwd_supported(const SeqArgs &s) { return s.states || groups_per_round(s) >= 1; }
int fp32_dbeta_rows(int N) { return (N + kL - 1) / kL; }

cudaError_t launch_fp32_fwd(const SeqArgs &s)
{
    if (s.io == HGRN2_BF16)
        return s.cu ? fwd_t<__nv_bfloat16, alu::kGateIsF, true>(s, nullptr) : fwd_t<__nv_bfloat16, alu::kGateIsF, false>(s, nullptr);
    return s.cu ? fwd_t<float, alu::kGateIsF, true>(s, nullptr) : fwd_t<float, alu::kGateIsF, false>(s, nullptr);
}
cudaError_t launch_fp32_bwd(const SeqArgs &s)
{
    if (s.io == HGRN2_BF16)
        return s.cu ? bwd_t<__nv_bfloat16, alu::kGateIsF, true>(s, nullptr, nullptr)
                    : bwd_t<__nv_bfloat16, alu::kGateIsF, false>(s, nullptr, nullptr);
    return s.cu ? bwd_t<float, alu::kGateIsF, true>(s, nullptr, nullptr) : bwd_t<float, alu::kGateIsF, false>(s, nullptr, nullptr);
}
cudaError_t launch_fp32_fwd_gated(const SeqArgs &s, const float *beta)
{
    return s.io == HGRN2_BF16 ? fwd_t<__nv_bfloat16, alu::kGatePre, false>(s, beta) : fwd_t<float, alu::kGatePre, false>(s, beta);
}
cudaError_t launch_fp32_bwd_gated(const SeqArgs &s, const float *beta, float *dbeta)
{
    return s.io == HGRN2_BF16 ? bwd_t<__nv_bfloat16, alu::kGatePre, false>(s, beta, dbeta)
                              : bwd_t<float, alu::kGatePre, false>(s, beta, dbeta);
}

}  // namespace hgrn2
