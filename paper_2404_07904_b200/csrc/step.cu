// Decode steps (Eq. 3 applied once, or a few times, per call), bandwidth-bound:  S[k][v] <- f[k] S[k][v] +
// (1 - f[k]) i[v],  and y[v] = sum_k o[k] S_new[k][v] on the way.
//
// Sixteen threads share a column: thread row group rg adds up the rows rg, rg + 16, ...  A thread owns kVec float4
// column groups (two where the head is wide enough: a row's gates then serve eight columns); the state is read once,
// all of a batch's 16-byte loads issued before the first dependent instruction, and written once.  A unit's columns
// may be spread over kSplit CTAs: columns do not interact, and which rows a thread adds up in which order stays the
// same, so every split and both kernels give the same bits.  No atomics: the cross-row reduction goes through shared
// memory in a fixed order.
#include "common.cuh"

namespace hgrn2 {

namespace {

constexpr int kRG = 16;                // row groups of a unit
// Up to here a one-token step spreads a unit over four CTAs: fewer than two units per SM are all latency, which more
// and smaller CTAs with all their loads in flight shorten (64 units: 4.1 instead of 5.1 us per call, 288 units: 7.1
// instead of 8.2), and beyond two per SM the split costs bandwidth (576 units: 16.4 instead of 15.2 us).
constexpr long long kFewUnits = 2 * 148;

template <int DV> struct Cols {
    static constexpr int kVec = DV >= 64 ? 2 : 1;             // float4 column groups per thread
    static constexpr int kThreads = kRG * DV / (4 * kVec);    // of a whole unit
};

// One token.  kSplit CTAs per unit, kBatch rows loaded ahead per thread.
template <typename T, int DV, int kSplit, int kBatch>
__global__ void __launch_bounds__(Cols<DV>::kThreads / kSplit)
step_kernel(const T *__restrict__ o, const T *__restrict__ f, const T *__restrict__ i,
            float *__restrict__ S, T *__restrict__ y, int dk, long long units)
{
    constexpr int VEC = Cols<DV>::kVec, NT = Cols<DV>::kThreads / kSplit;
    constexpr int CW = DV / kSplit;            // columns of this CTA
    constexpr int CG = CW / (4 * VEC);         // threads side by side
    constexpr int C4 = DV / 4;                 // float4s per row
    __shared__ float s_o[128], s_f[128];
    __shared__ __align__(16) float s_i[CW];
    __shared__ __align__(16) float s_red[kRG][CW];

    const int tid = threadIdx.x;
    const int c4 = tid % CG;                   // float4 columns c4 and (VEC = 2) c4 + CG
    const int rg = tid / CG;

    for (long long x = blockIdx.x; x < units * kSplit; x += gridDim.x) {
        const long long u = x / kSplit;
        const int col0 = (int)(x - u * kSplit) * CW;
        float4 *Su = reinterpret_cast<float4 *>(S + u * (long long)dk * DV + col0) + c4;
        // the first batch of the state is under way before anything waits for the gates
        float4 s[kBatch][VEC];
#pragma unroll
        for (int j = 0; j < kBatch; ++j)
#pragma unroll
            for (int e = 0; e < VEC; ++e)
                if (rg + j * kRG < dk) s[j][e] = __ldcs(Su + (long long)(rg + j * kRG) * C4 + e * CG);
        for (int k = tid; k < dk; k += NT) {
            s_o[k] = load_f(o + u * dk + k);
            s_f[k] = load_f(f + u * dk + k);
        }
        for (int v = tid; v < CW; v += NT) s_i[v] = load_f(i + u * DV + col0 + v);
        __syncthreads();

        float4 iv[VEC], acc[VEC];
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
            iv[e] = *reinterpret_cast<const float4 *>(s_i + 4 * (c4 + e * CG));
            acc[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int k0 = rg; k0 < dk; k0 += kRG * kBatch) {
            if (k0 != rg) {
#pragma unroll
                for (int j = 0; j < kBatch; ++j)
#pragma unroll
                    for (int e = 0; e < VEC; ++e)
                        if (k0 + j * kRG < dk) s[j][e] = __ldcs(Su + (long long)(k0 + j * kRG) * C4 + e * CG);
            }
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                const int k = k0 + j * kRG;
                if (k < dk) {
                    const float fk = s_f[k], kk = 1.0f - fk, ok = s_o[k];
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        float4 &t = s[j][e];
                        t.x = fmaf(fk, t.x, kk * iv[e].x);
                        t.y = fmaf(fk, t.y, kk * iv[e].y);
                        t.z = fmaf(fk, t.z, kk * iv[e].z);
                        t.w = fmaf(fk, t.w, kk * iv[e].w);
                        __stcs(Su + (long long)k * C4 + e * CG, t);
                        acc[e].x = fmaf(ok, t.x, acc[e].x);
                        acc[e].y = fmaf(ok, t.y, acc[e].y);
                        acc[e].z = fmaf(ok, t.z, acc[e].z);
                        acc[e].w = fmaf(ok, t.w, acc[e].w);
                    }
                }
            }
        }
#pragma unroll
        for (int e = 0; e < VEC; ++e) *reinterpret_cast<float4 *>(&s_red[rg][4 * (c4 + e * CG)]) = acc[e];
        __syncthreads();
        for (int v = tid; v < CW; v += NT) {
            float t = 0.f;
#pragma unroll
            for (int r = 0; r < kRG; ++r) t += s_red[r][v];
            store_f(y + u * DV + col0 + v, t);
        }
        __syncthreads();
    }
}

// Several successive tokens in one launch (multi-token / speculative decode): a unit's state is read once, kept in
// registers while Eq. 3 is applied Tn times, and written once, so the state traffic per token falls Tn-fold.
// d_k = d_v = D.  Row order, arithmetic and summation order are those of step_kernel, so the results are
// bit-identical to Tn single steps.  Sequence tensors are [unit][token][D].
//
// The state traffic (83 us for 4096 units of 128 x 128) and three operations per element and token (45 us for eight
// tokens) have to overlap, which only CTAs in different phases provide: hence half a unit per CTA, four or five CTAs per
// SM, and no barrier per token - the partial sums of eight tokens are added up together.  What the loop over rows
// must not do is read much shared memory: a warp's load takes a cycle per 128 bytes of REGISTERS filled, broadcast
// or not, so gates staged as ready-made pairs (24 bytes per row for four columns) cost as much as the arithmetic
// twice over.  One 8-byte (f, o) per row serves eight columns here.  4096 units, bf16: 8 tokens 139 -> 112 us (83 is
// the state traffic alone), 16 tokens 250 -> 169 us; quarter units per CTA 141 us, one token per loop body 115 us.
template <typename T, int D, int kSplit, int TB>
__global__ void __launch_bounds__(Cols<D>::kThreads / kSplit)
step_multi_kernel(const T *__restrict__ o, const T *__restrict__ f, const T *__restrict__ i,
                  float *__restrict__ S, T *__restrict__ y, int Tn, long long units)
{
    constexpr int VEC = Cols<D>::kVec, NT = Cols<D>::kThreads / kSplit;
    constexpr int CW = D / kSplit, CG = CW / (4 * VEC), C4 = D / 4;
    constexpr int R = D / kRG;                 // rows per thread
    __shared__ __align__(16) float2 s_fo[TB][D];              // filled 16 bytes at a time
    __shared__ __align__(16) float s_i[TB][CW];
    __shared__ __align__(16) float s_red[TB][kRG][CW];

    const int tid = threadIdx.x;
    const int c4 = tid % CG;
    const int rg = tid / CG;

    for (long long x = blockIdx.x; x < units * kSplit; x += gridDim.x) {
        const long long u = x / kSplit;
        const int col0 = (int)(x - u * kSplit) * CW;
        float4 *Su = reinterpret_cast<float4 *>(S + u * (long long)D * D + col0) + c4;
        float4 s[R][VEC];
#pragma unroll
        for (int j = 0; j < R; ++j)
#pragma unroll
            for (int e = 0; e < VEC; ++e) s[j][e] = __ldcs(Su + (long long)(rg + j * kRG) * C4 + e * CG);

        for (int t0 = 0; t0 < Tn; t0 += TB) {
            const int nb = min(TB, Tn - t0);
            const long long row0 = (u * Tn + t0) * D;
            for (int idx = tid; idx < nb * D / 4; idx += NT) {
                float fv[4], ov[4];
                load4(f + row0 + 4 * idx, fv);
                load4(o + row0 + 4 * idx, ov);
                float4 *dst = reinterpret_cast<float4 *>(&s_fo[0][0] + 4 * idx);
                dst[0] = make_float4(fv[0], ov[0], fv[1], ov[1]);
                dst[1] = make_float4(fv[2], ov[2], fv[3], ov[3]);
            }
            for (int idx = tid; idx < nb * CW; idx += NT)
                s_i[idx / CW][idx % CW] = load_f(i + row0 + (idx / CW) * D + col0 + idx % CW);
            __syncthreads();
#pragma unroll 2
            for (int tt = 0; tt < nb; ++tt) {
                float4 iv[VEC];
                float2 a[VEC][2];
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    iv[e] = *reinterpret_cast<const float4 *>(&s_i[tt][4 * (c4 + e * CG)]);
                    a[e][0] = a[e][1] = make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    const float2 fo = s_fo[tt][rg + j * kRG];
                    const float kk = 1.0f - fo.x;
                    const float2 f2 = make_float2(fo.x, fo.x), k2 = make_float2(kk, kk), o2 = make_float2(fo.y, fo.y);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        float2 lo = make_float2(s[j][e].x, s[j][e].y), hi = make_float2(s[j][e].z, s[j][e].w);
                        lo = fma_x2(f2, lo, mul_x2(k2, make_float2(iv[e].x, iv[e].y)));
                        hi = fma_x2(f2, hi, mul_x2(k2, make_float2(iv[e].z, iv[e].w)));
                        a[e][0] = fma_x2(o2, lo, a[e][0]);
                        a[e][1] = fma_x2(o2, hi, a[e][1]);
                        s[j][e] = make_float4(lo.x, lo.y, hi.x, hi.y);
                    }
                }
#pragma unroll
                for (int e = 0; e < VEC; ++e)
                    *reinterpret_cast<float4 *>(&s_red[tt][rg][4 * (c4 + e * CG)]) = make_float4(a[e][0].x, a[e][0].y, a[e][1].x, a[e][1].y);
            }
            __syncthreads();
            for (int idx = tid; idx < nb * CW; idx += NT) {
                const int tt = idx / CW, v = idx % CW;
                float sum = 0.f;
#pragma unroll
                for (int r = 0; r < kRG; ++r) sum += s_red[tt][r][v];
                store_f(y + row0 + tt * D + col0 + v, sum);
            }
            // the next block's gates overwrite what every thread read before the last barrier, its partial sums are
            // written behind the barrier after that
        }
#pragma unroll
        for (int j = 0; j < R; ++j)
#pragma unroll
            for (int e = 0; e < VEC; ++e) __stcs(Su + (long long)(rg + j * kRG) * C4 + e * CG, s[j][e]);
        __syncthreads();
    }
}

unsigned step_grid(long long ctas) { return (unsigned)(ctas < (1ll << 30) ? ctas : (1ll << 30)); }

// TB = tokens staged, and reduced, together
template <typename T, int D, int kSplit, int TB = 8>
cudaError_t launch_step_multi_t(const StepArgs &a)
{
    const long long units = (long long)a.B * a.H;
    if (units == 0 || a.T == 0) return cudaSuccess;
    step_multi_kernel<T, D, kSplit, TB><<<step_grid(units * kSplit), Cols<D>::kThreads / kSplit, 0, a.stream>>>(
        static_cast<const T *>(a.o), static_cast<const T *>(a.f), static_cast<const T *>(a.i), a.S,
        static_cast<T *>(a.y), a.T, units);
    return cudaGetLastError();
}

template <typename T, int DV, int kSplit, int kBatch>
cudaError_t launch_step_t(const StepArgs &a)
{
    const long long units = (long long)a.B * a.H;
    if (units == 0) return cudaSuccess;
    step_kernel<T, DV, kSplit, kBatch><<<step_grid(units * kSplit), Cols<DV>::kThreads / kSplit, 0, a.stream>>>(
        static_cast<const T *>(a.o), static_cast<const T *>(a.f), static_cast<const T *>(a.i), a.S,
        static_cast<T *>(a.y), a.dk, units);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_step_dv(const StepArgs &a)
{
    const bool few = !a.whole && (long long)a.B * a.H <= kFewUnits;
    switch (a.dv) {
        case 16:  return launch_step_t<T, 16, 1, 8>(a);
        case 32:  return launch_step_t<T, 32, 1, 8>(a);
        case 64:  return few ? launch_step_t<T, 64, 4, 4>(a) : launch_step_t<T, 64, 1, 4>(a);
        case 128: return few ? launch_step_t<T, 128, 4, 8>(a) : launch_step_t<T, 128, 1, 4>(a);
        default:  return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_step(const StepArgs &a)
{
    return a.io == HGRN2_BF16 ? launch_step_dv<__nv_bfloat16>(a) : launch_step_dv<float>(a);
}

bool step_multi_supported(int dk, int dv) { return dk == dv && (dk == 64 || dk == 128); }

cudaError_t launch_step_multi(const StepArgs &a)
{
    if (!step_multi_supported(a.dk, a.dv)) return cudaErrorInvalidValue;
    if (a.io == HGRN2_BF16)
        return a.dk == 64 ? launch_step_multi_t<__nv_bfloat16, 64, 1>(a)
               : a.whole  ? launch_step_multi_t<__nv_bfloat16, 128, 1, 4>(a) : launch_step_multi_t<__nv_bfloat16, 128, 2>(a);
    return a.dk == 64 ? launch_step_multi_t<float, 64, 1>(a)
           : a.whole  ? launch_step_multi_t<float, 128, 1, 4>(a) : launch_step_multi_t<float, 128, 2>(a);
}

}  // namespace hgrn2
