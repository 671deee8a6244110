// Chunkwise HGRN2 forward and backward on fp32 CUDA cores, parallel over the chunks of a sequence.
//
// This is the path for float32 I/O and for every head size the tensor-core kernels do not cover.  All products
// are fp32 FMAs on fp32 operands.  Chunk length 64; per direction two kernels:
//
//   state pass   the only serial one: a CTA owns a 32 x BV block of one unit's state (forward) or state gradient
//                (backward) in registers, walks the chunks and leaves the value at every chunk boundary in memory;
//   output pass  one CTA per chunk and 64 columns of an output; chunks are independent once the boundary values
//                are there.
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
// Bound by FMA issue (72 TFLOP/s measured on this chip).  One CTA walking a unit's chunks with everything in shared
// memory, scalar shared loads and an exp per decay pair took 34.0 ms for forward + backward of 2 x 16 units of 2048 tokens
// at d = 128 in float32 and 12.9 ms for 4 x 16 units at d = 64 in bf16; these kernels take 0.80 and 0.56 ms, and 59 instead
// of 1564 us for 2 units of 256 tokens at d = 64.
//
// Inner products of two operands stored with the contracted index innermost, and outer products of two stored
// with it outermost, both read 16-byte pieces of rows; every tile keeps piece c of row r at c ^ (r / 4 % 8), so
// either access hits all banks once.  A thread owns a 4 x 4 block of a 64 x 64 result (8 x 4 lanes, so the four
// rows of a warp's lanes and its eight column groups each come in one wavefront): 8 shared loads per 64 FMAs.
#include "chunk_alu.cuh"

namespace hgrn2 {

namespace {

using alu::GateMode;
using alu::gate_values;
using alu::sigmoid_f;
using alu::value_of;

constexpr int kL = 64;              // tokens per chunk
constexpr int kW = 32;              // width of a slab of the contracted index
constexpr int kOutThreads = 256;
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
// (u - g0) NC.  Packed (see PackedArgs): head h, sequence b; slots from (h - g0) spp + cu[b] / 64 + b.
struct Where { long long row; int n, nc; long long slot, unit; };

__device__ __forceinline__ Where packed_where(const Args &a, int b, long long h)
{
    const int start = a.cu[b];
    int n = a.cu[b + 1] - start;
    if (start < 0 || n < 0 || start + n > a.N) n = 0;          // malformed offsets: touch nothing
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

struct Frag { float4 r[4]; };
// Pieces c of the four rows r0 .. r0 + 3 (r0 a multiple of 4).
template <int W> __device__ __forceinline__ Frag rows4(const float *t, int r0, int c)
{
    Frag f;
    const float *p = t + piece<W>(r0, c);
#pragma unroll
    for (int i = 0; i < 4; ++i) f.r[i] = *reinterpret_cast<const float4 *>(p + i * W);
    return f;
}
__device__ __forceinline__ void dot4(float (&acc)[4][4], const Frag &a, const Frag &b)
{
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            acc[i][j] = fmaf(a.r[i].x, b.r[j].x, acc[i][j]);
            acc[i][j] = fmaf(a.r[i].y, b.r[j].y, acc[i][j]);
            acc[i][j] = fmaf(a.r[i].z, b.r[j].z, acc[i][j]);
            acc[i][j] = fmaf(a.r[i].w, b.r[j].w, acc[i][j]);
        }
}
__device__ __forceinline__ void rank1(float (&acc)[4][4], float a0, float a1, float a2, float a3, float4 b)
{
    const float a[4] = {a0, a1, a2, a3};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        acc[i][0] = fmaf(a[i], b.x, acc[i][0]);
        acc[i][1] = fmaf(a[i], b.y, acc[i][1]);
        acc[i][2] = fmaf(a[i], b.z, acc[i][2]);
        acc[i][3] = fmaf(a[i], b.w, acc[i][3]);
    }
}
// acc[m][n] += sum_x A[m][x] B[n][x] over kPieces pieces (4 x each)
template <int WA, int WB, int kPieces>
__device__ __forceinline__ void mul_inner_inner(float (&acc)[4][4], const float *A, int m0, const float *B, int n0)
{
#pragma unroll 4
    for (int c = 0; c < kPieces; ++c) dot4(acc, rows4<WA>(A, m0, c), rows4<WB>(B, n0, c));
}
// acc[m][n] += sum_x A[m][x] B[x][n], x in pieces [c0, c1)
template <int WA, int WB>
__device__ __forceinline__ void mul_inner_outer(float (&acc)[4][4], const float *A, int m0, const float *B, int n0, int c0, int c1)
{
#pragma unroll 4
    for (int c = c0; c < c1; ++c) {
        const Frag a = rows4<WA>(A, m0, c);
        const float *b = B + piece<WB>(4 * c, n0 >> 2);
        const float4 b0 = *reinterpret_cast<const float4 *>(b), b1 = *reinterpret_cast<const float4 *>(b + WB);
        const float4 b2 = *reinterpret_cast<const float4 *>(b + 2 * WB), b3 = *reinterpret_cast<const float4 *>(b + 3 * WB);
        rank1(acc, a.r[0].x, a.r[1].x, a.r[2].x, a.r[3].x, b0);
        rank1(acc, a.r[0].y, a.r[1].y, a.r[2].y, a.r[3].y, b1);
        rank1(acc, a.r[0].z, a.r[1].z, a.r[2].z, a.r[3].z, b2);
        rank1(acc, a.r[0].w, a.r[1].w, a.r[2].w, a.r[3].w, b3);
    }
}
// acc[m][n] += sum_x A[x][m] B[x][n], x in groups of four [c0, c1)
template <int WA, int WB>
__device__ __forceinline__ void mul_outer_outer(float (&acc)[4][4], const float *A, int m0, const float *B, int n0, int c0, int c1)
{
#pragma unroll 4
    for (int c = c0; c < c1; ++c) {
        const float *a = A + piece<WA>(4 * c, m0 >> 2), *b = B + piece<WB>(4 * c, n0 >> 2);
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const float4 av = *reinterpret_cast<const float4 *>(a + x * WA);
            rank1(acc, av.x, av.y, av.z, av.w, *reinterpret_cast<const float4 *>(b + x * WB));
        }
    }
}
__device__ __forceinline__ void zero(float (&acc)[4][4])
{
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
}

__device__ __forceinline__ void cp_async16(float *dst, const float *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int n> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(n) : "memory"); }

// ---------------------------------------------------------------------------------------------------------------
// State pass.  forward: S <- Diag(Lam_c) S + K^T V, K_s = k_s prod_{r>s} f_r; backward (chunks in reverse):
// D <- Diag(Lam_c) D + Q^T dY, Q_t = q_t prod_{r<=t} f_r.  The value before the update goes to the chunk's slot.
// Grid (units, dk blocks of 32, dv blocks of BV), BV in {32, 64}, 2 BV threads; a thread's loads of the next chunk are
// in flight while the current one is multiplied.
template <typename T, int kMode, bool kBwd, int BV>
__global__ void __launch_bounds__(2 * BV)
fp32_state_kernel(const Args a)
{
    constexpr int NT = 2 * BV, SEG = NT / 32, RP = kL / SEG;         // row segments, rows per segment
    constexpr int VP = BV / 4;                                        // pieces per row of the V tile
    constexpr int VL = kL * VP / NT;                                  // pieces a thread loads
    __shared__ __align__(16) float sX[kL * kW];
    __shared__ __align__(16) float sV[kL * BV];
    __shared__ float sprod[2][SEG][kW];

    if (a.status != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) {
        a.status->code = 0;
        a.status->where = 0;
        a.status->exact_units = 0;
    }
    Where w;
    if (a.cu == nullptr) {
        w = Where{(a.g0 + blockIdx.x) * a.N, a.N, a.NC, (long long)blockIdx.x * a.NC, a.g0 + blockIdx.x};
    } else {
        const int b = blockIdx.x % a.B;
        w = packed_where(a, b, a.g0 + blockIdx.x / a.B);
    }
    const int tid = threadIdx.x, lane = tid & 31, seg = tid >> 5;
    const int k0 = blockIdx.y * kW, v0 = blockIdx.z * BV;
    const int kx = k0 + lane;
    const bool kin = kx < a.dk;
    const int m0 = 16 * (seg & 1) + 4 * (lane >> 3), n0 = 32 * (seg >> 1) + 4 * (lane & 7);
    const bool own = k0 + m0 < a.dk && v0 + n0 < a.dv;                // dk, dv are multiples of 16: blocks are in or out
    const T *xg = static_cast<const T *>(a.o) + w.row * a.dk + kx;
    const T *fg = static_cast<const T *>(a.f) + w.row * a.dk + kx;
    const T *vg = static_cast<const T *>(kBwd ? a.dy : a.i) + w.row * a.dv + v0;
    const float beta = kMode == alu::kGatePre && kin ? a.beta[(size_t)(w.unit % a.H) * a.dk + kx] : 0.f;
    const size_t ss = (size_t)a.dk * a.dv, blk = (size_t)(k0 + m0) * a.dv + v0 + n0;

    float acc[4][4];
    zero(acc);
    const float *init = kBwd ? a.dSN : a.S0;
    if (own && init != nullptr) {
#pragma unroll
        for (int i = 0; i < 4; ++i) load4(init + (size_t)w.unit * ss + blk + (size_t)i * a.dv, acc[i]);
    }
    float *out = kBwd ? a.dstates : a.states;

    T fr[RP], qr[kBwd ? RP : 1];
    Raw4<T> vr[VL];
    auto fetch = [&](int c) {
        const int t0 = c * kL, rows = min(kL, w.n - t0);
#pragma unroll
        for (int r = 0; r < RP; ++r) {
            const int t = seg * RP + r;
            if (kin && t < rows) {
                fr[r] = fg[(size_t)(t0 + t) * a.dk];
                if (kBwd) qr[kBwd ? r : 0] = xg[(size_t)(t0 + t) * a.dk];
            }
        }
#pragma unroll
        for (int x = 0; x < VL; ++x) {
            const int t = (tid + x * NT) / VP, p = (tid + x * NT) % VP;
            vr[x] = t < rows && v0 + 4 * p < a.dv ? raw_load4(vg + (size_t)(t0 + t) * a.dv + 4 * p) : raw_zero4<T>();
        }
    };
    if (w.nc > 0) fetch(kBwd ? w.nc - 1 : 0);
    for (int it = 0; it < w.nc; ++it) {
        const int c = kBwd ? w.nc - 1 - it : it;
        const int rows = min(kL, w.n - c * kL);
        if (own) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                store4(out + (size_t)(w.slot + c) * ss + blk + (size_t)i * a.dv, acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
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
        float (*sp)[kW] = sprod[it & 1];
        sp[seg][lane] = h;
        __syncthreads();                                              // also: the previous chunk's product has read sX, sV
        float P = 1.f;
#pragma unroll
        for (int s = 0; s < SEG; ++s)
            if (kBwd ? s < seg : s > seg) P *= sp[s][lane];
#pragma unroll
        for (int x = 0; x < RP; ++x) {
            const int r = kBwd ? x : RP - 1 - x, t = seg * RP + r;
            if (kBwd) P *= fv[r];
            sX[elem<kW>(t, lane)] = xv[r] * P;
            if (!kBwd) P *= fv[r];
        }
#pragma unroll
        for (int x = 0; x < VL; ++x) {
            const int t = (tid + x * NT) / VP, p = (tid + x * NT) % VP;
            float4 v = widen(vr[x]);
            if (!kBwd) v = value4<kMode>(v);
            *reinterpret_cast<float4 *>(sV + piece<BV>(t, p)) = v;
        }
        float lam[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            lam[i] = sp[0][m0 + i];
#pragma unroll
            for (int s = 1; s < SEG; ++s) lam[i] *= sp[s][m0 + i];
        }
        __syncthreads();
        if (it + 1 < w.nc) fetch(kBwd ? c - 1 : c + 1);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] *= lam[i];
        mul_outer_outer<kW, BV>(acc, sX, m0, sV, n0, 0, kL / 4);
    }
    float *fin = kBwd ? a.dS0 : a.SN;
    if (own && fin != nullptr) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            store4(fin + (size_t)w.unit * ss + blk + (size_t)i * a.dv, acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    }
}

// Which chunk blockIdx.x stands for: false = none (a slot of a packed batch that no chunk uses).
__device__ __forceinline__ bool chunk_of(const Args &a, Where &w, int &c)
{
    if (a.cu == nullptr) {
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
    w = packed_where(a, lo, a.g0 + h);
    c = slot - (a.cu[lo] / kL + lo);
    return c >= 0 && c < w.nc;
}

// ---------------------------------------------------------------------------------------------------------------
// Output pass over value columns.  kDV = false: Y = A V + Qs (Pm S_in); kDV = true: dV = A^T dY + Ks (E D_out).
// CTA = (chunk, 64 value columns); the key dimension is the contracted index of both A and the state term and
// comes in slabs of 32, double buffered, the next slab's elements in registers while the current one is multiplied.
constexpr int kVStage = 2 * kL * kW + kW * kL;                        // Qs, Ks [64][32], state rows [32][64]
constexpr size_t kVSmem = (2 * kVStage + kL * kL + 2 * 8 * kW) * sizeof(float);

template <typename T, int kMode, bool kDV>
__global__ void __launch_bounds__(kOutThreads, 2)
fp32_value_kernel(const Args a)
{
    extern __shared__ __align__(16) float sm[];
    float *sW = sm + 2 * kVStage;                                     // V or dY, [64][64]
    float *sprod = sW + kL * kL;                                      // [2][8][32]
    Where w;
    int c;
    if (!chunk_of(a, w, c)) return;
    const int tid = threadIdx.x, lane = tid & 31, seg = tid >> 5;
    const int wm = seg >> 1, wn = seg & 1;
    const int m0 = 16 * wm + 4 * (lane >> 3), n0 = 32 * wn + 4 * (lane & 7);
    const int v0 = blockIdx.y * kL;
    const int rows = min(kL, w.n - c * kL);
    const long long row0 = w.row + (long long)c * kL;
    const size_t ss = (size_t)a.dk * a.dv;
    const float *st = (kDV ? a.dstates : a.states) + (size_t)(w.slot + c) * ss;
    const T *og = static_cast<const T *>(a.o) + row0 * a.dk, *fg = static_cast<const T *>(a.f) + row0 * a.dk;
    const T *wg = static_cast<const T *>(kDV ? a.dy : a.i) + row0 * a.dv;
    const float *beta = kMode == alu::kGatePre ? a.beta + (size_t)(w.unit % a.H) * a.dk : nullptr;
    const bool above = wm < 2 && wn == 1;                             // this warp's part of A lies above the diagonal

    T qr[8], fr[8];
    float4 sr[2];
    auto fetch = [&](int k0) {
        const int kx = k0 + lane;
#pragma unroll
        for (int r = 0; r < 8; ++r)
            if (kx < a.dk && seg * 8 + r < rows) {
                qr[r] = og[(size_t)(seg * 8 + r) * a.dk + kx];
                fr[r] = fg[(size_t)(seg * 8 + r) * a.dk + kx];
            }
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int k = k0 + (tid >> 4) + 16 * x, p = tid & 15;
            sr[x] = k < a.dk && v0 + 4 * p < a.dv ? *reinterpret_cast<const float4 *>(st + (size_t)k * a.dv + v0 + 4 * p)
                                                  : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    fetch(0);
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const int t = (tid >> 4) + 16 * x, p = tid & 15;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (t < rows && v0 + 4 * p < a.dv) v = widen(raw_load4(wg + (size_t)t * a.dv + v0 + 4 * p));
        if (!kDV) v = value4<kMode>(v);
        *reinterpret_cast<float4 *>(sW + piece<kL>(t, p)) = v;
    }

    float accA[4][4], accY[4][4];
    zero(accA);
    zero(accY);
    const int nslab = (a.dk + kW - 1) / kW;
    for (int j = 0; j < nslab; ++j) {
        float *sQ = sm + (j & 1) * kVStage, *sK = sQ + kL * kW, *sS = sK + kL * kW;
        float *sp = sprod + (j & 1) * 8 * kW;
        const int k0 = j * kW;
        float qv[8], kv[8], fv[8], h = 1.f;
        const float bt = kMode == alu::kGatePre && k0 + lane < a.dk ? beta[k0 + lane] : 0.f;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            qv[r] = 0.f; kv[r] = 0.f; fv[r] = 1.f;
            if (k0 + lane < a.dk && seg * 8 + r < rows) {
                gate_values<kMode>(load_f(&qr[r]), load_f(&fr[r]), bt, qv[r], fv[r], kv[r]);
                fv[r] = fmaxf(fv[r], kFMin);
            }
            h *= fv[r];
        }
        sp[seg * kW + lane] = h;
        const float4 s0 = sr[0], s1 = sr[1];
        __syncthreads();
        float pr[8];
#pragma unroll
        for (int s = 0; s < 8; ++s) pr[s] = sp[s * kW + lane];
        const float pm = pr[0] * pr[1] * pr[2] * pr[3], ee = pr[4] * pr[5] * pr[6] * pr[7];
        // scale of the two state rows this thread brings
        float rs[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const float *q = sp + (kDV ? 4 * kW : 0) + (tid >> 4) + 16 * x;
            rs[x] = q[0] * q[kW] * q[2 * kW] * q[3 * kW];
        }
        // every warp's lanes see all 32 columns, so the decision is the same in every warp
        const bool out_of_range = __any_sync(0xFFFFFFFFu, fminf(pm, ee) < kHalfFloor);
        if (!out_of_range) {
            float P = 1.f;
            if (seg >= 4) {
#pragma unroll
                for (int s = 4; s < 8; ++s)
                    if (s < seg) P *= pr[s];
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    P *= fv[r];
                    const int at = elem<kW>(seg * 8 + r, lane);
                    sQ[at] = qv[r] * P;
                    sK[at] = kv[r] * (1.0f / P);
                }
            } else {
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    if (s > seg) P *= pr[s];
#pragma unroll
                for (int r = 7; r >= 0; --r) {
                    const int at = elem<kW>(seg * 8 + r, lane);
                    sQ[at] = qv[r] * (1.0f / P);
                    sK[at] = kv[r] * P;
                    P *= fv[r];
                }
            }
            *reinterpret_cast<float4 *>(sS + piece<kL>(tid >> 4, tid & 15)) = make_float4(s0.x * rs[0], s0.y * rs[0], s0.z * rs[0], s0.w * rs[0]);
            *reinterpret_cast<float4 *>(sS + piece<kL>((tid >> 4) + 16, tid & 15)) = make_float4(s1.x * rs[1], s1.y * rs[1], s1.z * rs[1], s1.w * rs[1]);
            __syncthreads();
            if (j + 1 < nslab) fetch(k0 + kW);
            if (!above) mul_inner_inner<kW, kW, kW / 4>(accA, sQ, m0, sK, n0);
            mul_inner_outer<kW, kL>(accY, kDV ? sK : sQ, m0, sS, n0, 0, kW / 4);
        } else {
            // pairwise decays: q, k and b (in the place of the state rows) of the slab, then the state term
            float *sb = sS;
            float b[8], run = 0.f;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                run += logf(fv[r]);
                b[r] = run;
            }
            __syncthreads();                                          // sp has been read
            sp[seg * kW + lane] = run;
            __syncthreads();
            float base = 0.f, total = 0.f;
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                if (s < seg) base += sp[s * kW + lane];
                total += sp[s * kW + lane];
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                b[r] += base;
                const int at = elem<kW>(seg * 8 + r, lane);
                sQ[at] = qv[r];
                sK[at] = kv[r];
                sb[at] = b[r];
            }
            __syncthreads();
            if (j + 1 < nslab) fetch(k0 + kW);
#pragma unroll 1
            for (int x = 0; x < kW; ++x)
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj)
                        if (n0 + jj <= m0 + i) {
                            const int at = elem<kW>(m0 + i, x), as = elem<kW>(n0 + jj, x);
                            accA[i][jj] = fmaf(sQ[at] * sK[as], expf(sb[at] - sb[as]), accA[i][jj]);
                        }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int at = elem<kW>(seg * 8 + r, lane);
                if (kDV) sK[at] = kv[r] * expf(total - b[r]);
                else sQ[at] = qv[r] * expf(b[r]);
            }
            *reinterpret_cast<float4 *>(sS + piece<kL>(tid >> 4, tid & 15)) = s0;
            *reinterpret_cast<float4 *>(sS + piece<kL>((tid >> 4) + 16, tid & 15)) = s1;
            __syncthreads();
            mul_inner_outer<kW, kL>(accY, kDV ? sK : sQ, m0, sS, n0, 0, kW / 4);
        }
    }
    __syncthreads();
    // tril(A), as [t][s] for Y and as [s][t] for dV, over the slabs
    float *sA = sm;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (n0 + j > m0 + i) accA[i][j] = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (kDV)
            *reinterpret_cast<float4 *>(sA + piece<kL>(n0 + i, m0 >> 2)) = make_float4(accA[0][i], accA[1][i], accA[2][i], accA[3][i]);
        else
            *reinterpret_cast<float4 *>(sA + piece<kL>(m0 + i, n0 >> 2)) = make_float4(accA[i][0], accA[i][1], accA[i][2], accA[i][3]);
    }
    __syncthreads();
    // only the tokens on the causal side of this warp's rows contribute
    mul_inner_outer<kL, kL>(accY, sA, m0, sW, n0, kDV ? 4 * wm : 0, kDV ? kL / 4 : 4 * (wm + 1));
    if (v0 + n0 < a.dv) {
        T *yg = static_cast<T *>(kDV ? a.d_i : a.y) + row0 * a.dv + v0 + n0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (m0 + i < rows) {
                if (kDV && kMode == alu::kGatePre) {                  // d silu(z) / dz = s (1 + z (1 - s)), s = sigmoid(z)
                    float z[4];
                    load4(static_cast<const T *>(a.i) + (row0 + m0 + i) * a.dv + v0 + n0, z);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float sg = sigmoid_f(z[j]);
                        accY[i][j] *= sg * (1.0f + z[j] * (1.0f - sg));
                    }
                }
                store4(yg + (size_t)(m0 + i) * a.dv, accY[i][0], accY[i][1], accY[i][2], accY[i][3]);
            }
    }
}

// ---------------------------------------------------------------------------------------------------------------
// Output pass over key columns: d_o and d_f of one chunk and 64 key dimensions.  The value dimension is the
// contracted index of dA, dY S_in^T and V D_out^T and comes in slabs of 32 (two stages: states by cp.async, dY and V
// through registers); then the intra-chunk products with Qs, Ks; then the scans along time.
constexpr int kKTile = kL * kW;                                       // [64][32]
constexpr size_t kKSmem = (8 * kKTile + 8 * kL + 5 * kL + 8 * kL) * sizeof(float);

template <typename T, int kMode>
__global__ void __launch_bounds__(kOutThreads, 2)
fp32_key_kernel(const Args a)
{
    extern __shared__ __align__(16) float sm[];
    float *sprod = sm + 8 * kKTile;                                   // [8][64]
    float *sR = sprod + 8 * kL;                                       // [64]
    float *ssum = sR + kL;                                            // [2][4][64] segment sums of a and e
    Where w;
    int c;
    if (!chunk_of(a, w, c)) return;
    const int tid = threadIdx.x, lane = tid & 31, seg = tid >> 5;
    const int wm = seg >> 1, wn = seg & 1;
    const int m0 = 16 * wm + 4 * (lane >> 3), n0 = 32 * wn + 4 * (lane & 7);
    const int k0 = blockIdx.y * kL;
    const int rows = min(kL, w.n - c * kL);
    const long long row0 = w.row + (long long)c * kL;
    const size_t ss = (size_t)a.dk * a.dv;
    const float *Sg = a.states + (size_t)(w.slot + c) * ss, *Dg = a.dstates + (size_t)(w.slot + c) * ss;
    const T *gg = static_cast<const T *>(a.dy) + row0 * a.dv, *vg = static_cast<const T *>(a.i) + row0 * a.dv;
    const bool above = wm < 2 && wn == 1;

    // stage layout: dY | V | S | D, each [64][32]
    Raw4<T> gr[2], vr[2];
    const int lr = tid >> 3, lp = tid & 7;                            // row (and row + 32), piece
    auto fetch_seq = [&](int v0) {
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int t = lr + 32 * x;
            const bool in = t < rows && v0 + 4 * lp < a.dv;
            gr[x] = in ? raw_load4(gg + (size_t)t * a.dv + v0 + 4 * lp) : raw_zero4<T>();
            vr[x] = in ? raw_load4(vg + (size_t)t * a.dv + v0 + 4 * lp) : raw_zero4<T>();
        }
    };
    auto fetch_state = [&](float *stage, int v0) {
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int k = lr + 32 * x, at = piece<kW>(k, lp);
            if (k0 + k < a.dk && v0 + 4 * lp < a.dv) {
                cp_async16(stage + 2 * kKTile + at, Sg + (size_t)(k0 + k) * a.dv + v0 + 4 * lp);
                cp_async16(stage + 3 * kKTile + at, Dg + (size_t)(k0 + k) * a.dv + v0 + 4 * lp);
            } else {
                *reinterpret_cast<float4 *>(stage + 2 * kKTile + at) = make_float4(0.f, 0.f, 0.f, 0.f);
                *reinterpret_cast<float4 *>(stage + 3 * kKTile + at) = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        cp_async_commit();
    };
    fetch_state(sm, 0);
    fetch_seq(0);

    float accA[4][4], accX[4][4], accZ[4][4];
    zero(accA);
    zero(accX);
    zero(accZ);
    float racc = 0.f;
    const int nslab = (a.dv + kW - 1) / kW;
    for (int j = 0; j < nslab; ++j) {
        float *st = sm + (j & 1) * 4 * kKTile;
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int at = piece<kW>(lr + 32 * x, lp);
            *reinterpret_cast<float4 *>(st + at) = widen(gr[x]);
            *reinterpret_cast<float4 *>(st + kKTile + at) = value4<kMode>(widen(vr[x]));
        }
        cp_async_wait<0>();
        __syncthreads();          // the slab is complete, and every warp is done with the other stage
        if (j + 1 < nslab) {
            fetch_state(sm + ((j + 1) & 1) * 4 * kKTile, (j + 1) * kW);
            fetch_seq((j + 1) * kW);
        }
        const float *sG = st, *sV = st + kKTile, *sS = st + 2 * kKTile, *sD = st + 3 * kKTile;
        if (!above) mul_inner_inner<kW, kW, kW / 4>(accA, sG, m0, sV, n0);
        mul_inner_inner<kW, kW, kW / 4>(accX, sG, m0, sS, n0);
        mul_inner_inner<kW, kW, kW / 4>(accZ, sV, m0, sD, n0);
        {
            const int k = tid >> 2;
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const int at = piece<kW>(k, 2 * (tid & 3) + x);
                const float4 s4 = *reinterpret_cast<const float4 *>(sS + at), d4 = *reinterpret_cast<const float4 *>(sD + at);
                racc = fmaf(s4.x, d4.x, racc);
                racc = fmaf(s4.y, d4.y, racc);
                racc = fmaf(s4.z, d4.z, racc);
                racc = fmaf(s4.w, d4.w, racc);
            }
        }
    }
    racc += __shfl_xor_sync(0xFFFFFFFFu, racc, 1);
    racc += __shfl_xor_sync(0xFFFFFFFFu, racc, 2);
    if ((tid & 3) == 0) sR[tid >> 2] = racc;

    // ---- gates of the 64 key dimensions; thread = two columns, eight rows
    const T *og = static_cast<const T *>(a.o) + row0 * a.dk + k0, *fg = static_cast<const T *>(a.f) + row0 * a.dk + k0;
    const float *beta = kMode == alu::kGatePre ? a.beta + (size_t)(w.unit % a.H) * a.dk + k0 : nullptr;
    float qv[2][8], kv[2][8], fv[2][8];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const int kx = lane + 32 * x;
        float h = 1.f;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            qv[x][r] = 0.f; kv[x][r] = 0.f; fv[x][r] = 1.f;
            const int t = seg * 8 + r;
            if (k0 + kx < a.dk && t < rows) {
                gate_values<kMode>(load_f(og + (size_t)t * a.dk + kx), load_f(fg + (size_t)t * a.dk + kx),
                                   kMode == alu::kGatePre ? beta[kx] : 0.f, qv[x][r], fv[x][r], kv[x][r]);
                fv[x][r] = fmaxf(fv[x][r], kFMin);
            }
            h *= fv[x][r];
        }
        sprod[seg * kL + kx] = h;
    }
    __syncthreads();                                                  // the slabs are free from here on
    float *sA = sm, *sQ = sm + 2 * kKTile, *sK = sm + 4 * kKTile, *sC = sm + 6 * kKTile;   // [64][64] each
    bool low = false;
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const float *q = sprod + lane + 32 * x;
        low |= fminf(q[0] * q[kL] * q[2 * kL] * q[3 * kL], q[4 * kL] * q[5 * kL] * q[6 * kL] * q[7 * kL]) < kHalfFloor;
    }
    const bool out_of_range = __any_sync(0xFFFFFFFFu, low);           // the same in every warp
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (n0 + j > m0 + i) accA[i][j] = 0.f;
        *reinterpret_cast<float4 *>(sA + piece<kL>(m0 + i, n0 >> 2)) = make_float4(accA[i][0], accA[i][1], accA[i][2], accA[i][3]);
    }
    float G[4][4], J[4][4];
    zero(G);
    zero(J);
    T *do_g = static_cast<T *>(a.d_o) + row0 * a.dk + k0 + n0;
    const bool kown = k0 + n0 < a.dk;
    float a_[4][4], e_[4][4], dk_[4][4];
    if (!out_of_range) {
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int kx = lane + 32 * x;
            const float *pr = sprod + kx;
            float P = 1.f;
            if (seg >= 4) {
                for (int s = 4; s < seg; ++s) P *= pr[s * kL];
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    P *= fv[x][r];
                    const int at = elem<kL>(seg * 8 + r, kx);
                    sQ[at] = qv[x][r] * P;
                    sK[at] = kv[x][r] * (1.0f / P);
                    sC[at] = P;
                }
            } else {
                for (int s = seg + 1; s < 4; ++s) P *= pr[s * kL];
#pragma unroll
                for (int r = 7; r >= 0; --r) {
                    const int at = elem<kL>(seg * 8 + r, kx);
                    const float inv = 1.0f / P;
                    sQ[at] = qv[x][r] * inv;
                    sK[at] = kv[x][r] * P;
                    sC[at] = inv;
                    P *= fv[x][r];
                }
            }
        }
        __syncthreads();
        mul_inner_outer<kL, kL>(G, sA, m0, sK, n0, 0, 4 * (wm + 1));
        mul_outer_outer<kL, kL>(J, sA, m0, sQ, n0, 4 * wm, kL / 4);
        __syncthreads();
        float pm[4], ee[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float *q = sprod + n0 + j;
            pm[j] = q[0] * q[kL] * q[2 * kL] * q[3 * kL];
            ee[j] = q[4 * kL] * q[5 * kL] * q[6 * kL] * q[7 * kL];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int at = piece<kL>(m0 + i, n0 >> 2);
            float Q[4], K[4], C[4], dq[4];
            load4(sQ + at, Q);
            load4(sK + at, K);
            load4(sC + at, C);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float g = fmaf(pm[j], accX[i][j], G[i][j]), ez = ee[j] * accZ[i][j];
                dq[j] = C[j] * g;
                a_[i][j] = Q[j] * g - K[j] * J[i][j];
                e_[i][j] = K[j] * ez;
                dk_[i][j] = (J[i][j] + ez) / C[j];
                G[i][j] = dq[j];
            }
        }
    } else {
        // pairwise decays
        float *sb = sC;
        float b[2][8];
        __syncthreads();                                              // sprod has been read
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            float run = 0.f;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                run += logf(fv[x][r]);
                b[x][r] = run;
            }
            sprod[seg * kL + lane + 32 * x] = run;
        }
        __syncthreads();
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int kx = lane + 32 * x;
            float base = 0.f;
            for (int s = 0; s < seg; ++s) base += sprod[s * kL + kx];
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int at = elem<kL>(seg * 8 + r, kx);
                sQ[at] = qv[x][r];
                sK[at] = kv[x][r];
                sb[at] = b[x][r] + base;
            }
        }
        __syncthreads();
        float bC[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) bC[j] = sb[elem<kL>(kL - 1, n0 + j)];
#pragma unroll 1
        for (int x = 0; x < kL; ++x)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int t = m0 + i, at = elem<kL>(t, n0 + j), ax = elem<kL>(x, n0 + j);
                    if (x <= t) G[i][j] = fmaf(sA[elem<kL>(t, x)] * sK[ax], expf(sb[at] - sb[ax]), G[i][j]);
                    if (x >= t) J[i][j] = fmaf(sA[elem<kL>(x, t)] * sQ[ax], expf(sb[ax] - sb[at]), J[i][j]);
                }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int at = elem<kL>(m0 + i, n0 + j);
                const float bt = sb[at], dq = fmaf(expf(bt), accX[i][j], G[i][j]), ik = expf(bC[j] - bt) * accZ[i][j];
                a_[i][j] = sQ[at] * dq - sK[at] * J[i][j];
                e_[i][j] = sK[at] * ik;
                dk_[i][j] = J[i][j] + ik;
                G[i][j] = dq;
            }
        __syncthreads();
    }
    if (kown)
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (m0 + i < rows) {
                if (kMode == alu::kGatePre) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float s = sigmoid_f(load_f(og + (size_t)(m0 + i) * a.dk + n0 + j));
                        G[i][j] *= s * (1.0f - s);
                    }
                }
                store4(do_g + (size_t)(m0 + i) * a.dk, G[i][0], G[i][1], G[i][2], G[i][3]);
            }
    // a, e and dk in the places of Qs, Ks and the decays
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int at = piece<kL>(m0 + i, n0 >> 2);
        *reinterpret_cast<float4 *>(sQ + at) = make_float4(a_[i][0], a_[i][1], a_[i][2], a_[i][3]);
        *reinterpret_cast<float4 *>(sK + at) = make_float4(e_[i][0], e_[i][1], e_[i][2], e_[i][3]);
        *reinterpret_cast<float4 *>(sC + at) = make_float4(dk_[i][0], dk_[i][1], dk_[i][2], dk_[i][3]);
    }
    __syncthreads();
    // ---- scans along time: thread = one column, 16 rows
    const int col = tid & 63, q4 = tid >> 6;
    float av[16], ev[16], sa = 0.f, se = 0.f;
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int at = elem<kL>(16 * q4 + r, col);
        av[r] = sQ[at];
        ev[r] = sK[at];
        sa += av[r];
        se += ev[r];
    }
    ssum[q4 * kL + col] = sa;
    ssum[(4 + q4) * kL + col] = se;
    __syncthreads();
    float lamC, suf = 0.f, pre = 0.f;
    {
        const float *q = sprod + col;
        float x = q[0];
#pragma unroll
        for (int s = 1; s < 8; ++s) x = out_of_range ? x + q[s * kL] : x * q[s * kL];
        lamC = out_of_range ? expf(x) : x;
    }
    const float base = lamC * sR[col];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        if (s > q4) suf += ssum[s * kL + col];
        if (s < q4) pre += ssum[(4 + s) * kL + col];
    }
    // exclusive prefix of e in place, then the suffix of a downwards
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const float x = ev[r];
        ev[r] = pre;
        pre += x;
    }
    float dbeta = 0.f;
    if (k0 + col < a.dk) {
        T *df_g = static_cast<T *>(a.d_f) + row0 * a.dk + k0 + col;
        const float bt = kMode == alu::kGatePre ? beta[col] : 0.f;
#pragma unroll
        for (int r = 15; r >= 0; --r) {
            const int t = 16 * q4 + r;
            suf += av[r];
            if (t < rows) {
                const float fraw = load_f(fg + (size_t)t * a.dk + col);
                float q_, f_, k_;
                gate_values<kMode>(0.f, fraw, bt, q_, f_, k_);
                float d = (base + ev[r] + suf) / fmaxf(f_, kFMin) - sC[elem<kL>(t, col)];
                if (kMode == alu::kGatePre) {         // f = beta + (1 - beta) g:  df/dzf = (1 - beta) g (1 - g),  df/dbeta = 1 - g
                    const float g = sigmoid_f(fraw);
                    dbeta += d * (1.0f - g);
                    d *= (1.0f - bt) * g * (1.0f - g);
                }
                store_f(df_g + (size_t)t * a.dk, d);
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

template <typename T, int kMode, bool kBwd>
cudaError_t launch_state(const Args &a, long long units, cudaStream_t stream)
{
    const unsigned kb = (a.dk + kW - 1) / kW;
    if (a.dv > 32)
        fp32_state_kernel<T, kMode, kBwd, 64><<<dim3((unsigned)units, kb, (a.dv + 63) / 64), 128, 0, stream>>>(a);
    else
        fp32_state_kernel<T, kMode, kBwd, 32><<<dim3((unsigned)units, kb, 1), 64, 0, stream>>>(a);
    return cudaGetLastError();
}

template <typename T, int kMode, bool kDV>
cudaError_t launch_value(const Args &a, long long chunks, cudaStream_t stream)
{
    cudaError_t err = ensure_dynamic_smem(reinterpret_cast<const void *>(fp32_value_kernel<T, kMode, kDV>), kVSmem);
    if (err != cudaSuccess) return err;
    fp32_value_kernel<T, kMode, kDV><<<dim3((unsigned)chunks, (a.dv + kL - 1) / kL), kOutThreads, kVSmem, stream>>>(a);
    return cudaGetLastError();
}

template <typename T, int kMode>
cudaError_t launch_key(const Args &a, long long chunks, cudaStream_t stream)
{
    cudaError_t err = ensure_dynamic_smem(reinterpret_cast<const void *>(fp32_key_kernel<T, kMode>), kKSmem);
    if (err != cudaSuccess) return err;
    fp32_key_kernel<T, kMode><<<dim3((unsigned)chunks, (a.dk + kL - 1) / kL), kOutThreads, kKSmem, stream>>>(a);
    return cudaGetLastError();
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
long long slots_per_group(const Args &a) { return a.cu ? a.spp : a.NC; }
// Slots the caller's buffers have room for: they are sized for the call's own chunk length C <= 64.
long long slots_at_hand(const SeqArgs &s)
{
    return group_count(s) * (s.cu ? s.N / s.C + s.B + 1 : (s.N + s.C - 1) / s.C);
}
// Backward without saved states: groups whose two sets of boundary values fit the workspace's room together.
long long groups_per_round(const SeqArgs &s)
{
    const long long spg = s.cu ? s.N / kL + s.B + 1 : (s.N + kL - 1) / kL, fit = slots_at_hand(s) / (2 * spg);
    return fit < group_count(s) ? fit : group_count(s);
}
long long units_per_group(const Args &a) { return a.cu ? a.B : 1; }

template <typename T, int kMode>
cudaError_t fwd_t(const SeqArgs &s, const float *beta)
{
    Args a = make_args(s, beta);
    const long long g = group_count(s);
    a.states = s.states ? s.states : s.room;
    a.status = s.clear_status ? s.status : nullptr;
    cudaError_t err = launch_state<T, kMode, false>(a, g * units_per_group(a), s.stream);
    a.status = nullptr;
    if (err != cudaSuccess || s.y == nullptr) return err;
    return launch_value<T, kMode, false>(a, g * slots_per_group(a), s.stream);
}

template <typename T, int kMode>
cudaError_t bwd_t(const SeqArgs &s, const float *beta, float *dbeta)
{
    Args a = make_args(s, beta);
    const long long g = group_count(s), spg = slots_per_group(a), upg = units_per_group(a);
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
            if ((err = launch_state<T, kMode, false>(r, n * upg, s.stream)) != cudaSuccess) return err;
            a.status = nullptr;
        }
        if ((err = launch_state<T, kMode, true>(a, n * upg, s.stream)) != cudaSuccess) return err;
        a.status = nullptr;
        if ((err = launch_value<T, kMode, true>(a, n * spg, s.stream)) != cudaSuccess) return err;
        if ((err = launch_key<T, kMode>(a, n * spg, s.stream)) != cudaSuccess) return err;
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
    return s.io == HGRN2_BF16 ? fwd_t<__nv_bfloat16, alu::kGateIsF>(s, nullptr) : fwd_t<float, alu::kGateIsF>(s, nullptr);
}
cudaError_t launch_fp32_bwd(const SeqArgs &s)
{
    return s.io == HGRN2_BF16 ? bwd_t<__nv_bfloat16, alu::kGateIsF>(s, nullptr, nullptr) : bwd_t<float, alu::kGateIsF>(s, nullptr, nullptr);
}
cudaError_t launch_fp32_fwd_gated(const SeqArgs &s, const float *beta)
{
    return s.io == HGRN2_BF16 ? fwd_t<__nv_bfloat16, alu::kGatePre>(s, beta) : fwd_t<float, alu::kGatePre>(s, beta);
}
cudaError_t launch_fp32_bwd_gated(const SeqArgs &s, const float *beta, float *dbeta)
{
    return s.io == HGRN2_BF16 ? bwd_t<__nv_bfloat16, alu::kGatePre>(s, beta, dbeta) : bwd_t<float, alu::kGatePre>(s, beta, dbeta);
}

}  // namespace hgrn2
