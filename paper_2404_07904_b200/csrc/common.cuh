// Shared device/host helpers of the HGRN2 library (sm_100a only).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <vector>

#include "hgrn2.h"

namespace hgrn2 {

// Smallest forget-gate value the chunked kernels distinguish from zero: below it the
// in-chunk cumulative decay is formed as if f were this value.
constexpr float kFMin = 7.888609052210118e-31f;   // 2^-100
// d_f divides the decay gradient (a sum that cancels down to ~f times its terms) by f.  With the gated entry
// points' encoded gate, f is whatever the sigmoid gave, down to exactly 0; the divisor is kept above 2^-20 there:
// below it the quotient would be the sum's rounding noise times up to 2^100.
constexpr float kFDivMinK = 9.5367431640625e-7f;  // 2^-20

// Layout of the 256-byte status block at the start of every workspace.
struct StatusBlock {
    int32_t code;      // hgrn2_status, 0 = ok; first error wins
    int32_t where;     // kernel-specific location tag of the first error
    int32_t exact_units;   // tensor-core path: units the call redid on the exact fp32 path (decay out of range)
    int32_t pad[61];
};
static_assert(sizeof(StatusBlock) == 256, "status block is 256 bytes");

// A kernel launched with launch_chained may start while its predecessor in the stream still runs its last CTAs
// (programmatic dependent launch): the launch itself, and what the kernel does before chain_wait(), then cost nothing.
// Every thread of it calls chain_wait() before it touches global memory or leaves: behind it everything the stream
// did before is complete and visible, and the next kernel may be brought in.  What a predecessor may have written is
// read with plain loads (not __ldg, nor through const __restrict__): it has changed during this kernel's lifetime.
// A call of few tokens is a handful of kernels of a few microseconds each, so the starts count: prefill of 5000 tokens
// (three kernels) 48.2 -> 45.2 us, 2 units of 256 tokens on the fp32 path forward and backward (seven) 61.5 -> 55.4 us;
// nothing measurable at full size.
__device__ __forceinline__ void chain_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t stream, A &&...args)
{
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
    if (err != cudaSuccess) cudaGetLastError();       // it is this call's error: the next one's launches ask for theirs
    return err;
}

template <typename T> __device__ __forceinline__ float load_f(const T *p);
template <> __device__ __forceinline__ float load_f<float>(const float *p) { return *p; }
template <> __device__ __forceinline__ float load_f<__nv_bfloat16>(const __nv_bfloat16 *p)
{
    return __bfloat162float(*p);
}

// Packed fp32 arithmetic (sm_100): one instruction per two results, each rounded exactly like the scalar op.
__device__ __forceinline__ float2 mul_x2(float2 a, float2 b)
{
    float2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(reinterpret_cast<unsigned long long &>(d))
        : "l"(reinterpret_cast<unsigned long long &>(a)), "l"(reinterpret_cast<unsigned long long &>(b)));
    return d;
}
__device__ __forceinline__ float2 fma_x2(float2 a, float2 b, float2 c)
{
    float2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(reinterpret_cast<unsigned long long &>(d))
        : "l"(reinterpret_cast<unsigned long long &>(a)), "l"(reinterpret_cast<unsigned long long &>(b)),
          "l"(reinterpret_cast<unsigned long long &>(c)));
    return d;
}

// four consecutive elements, aligned to their own size
template <typename T> __device__ __forceinline__ void load4(const T *p, float (&x)[4]);
template <> __device__ __forceinline__ void load4<float>(const float *p, float (&x)[4])
{
    const float4 v = *reinterpret_cast<const float4 *>(p);
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
}
template <> __device__ __forceinline__ void load4<__nv_bfloat16>(const __nv_bfloat16 *p, float (&x)[4])
{
    const uint2 v = *reinterpret_cast<const uint2 *>(p);
    x[0] = __uint_as_float(v.x << 16); x[1] = __uint_as_float(v.x & 0xFFFF0000u);
    x[2] = __uint_as_float(v.y << 16); x[3] = __uint_as_float(v.y & 0xFFFF0000u);
}

template <typename T> __device__ __forceinline__ void store_f(T *p, float x);
template <> __device__ __forceinline__ void store_f<float>(float *p, float x) { *p = x; }
template <> __device__ __forceinline__ void store_f<__nv_bfloat16>(__nv_bfloat16 *p, float x)
{
    *p = __float2bfloat16_rn(x);
}

__device__ __forceinline__ void clear_block(StatusBlock *sb)
{
    sb->code = 0;
    sb->where = 0;
    sb->exact_units = 0;
}
__device__ __forceinline__ void report_error(StatusBlock *sb, int code, int where)
{
    if (sb != nullptr && atomicCAS(&sb->code, 0, code) == 0) sb->where = where;
}

// A kernel's dynamic shared-memory limit has to be raised once per device before its first launch with more than
// 48 KB; later calls find the (kernel, device) pair here and skip the runtime call.
inline cudaError_t ensure_dynamic_smem(const void *kernel, size_t bytes)
{
    struct Entry { const void *kernel; int device; size_t bytes; };
    static std::mutex mu;
    static std::vector<Entry> done;
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    std::lock_guard<std::mutex> lock(mu);
    for (Entry &e : done)
        if (e.kernel == kernel && e.device == dev) {
            if (e.bytes >= bytes) return cudaSuccess;
            err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
            if (err == cudaSuccess) e.bytes = bytes;
            return err;
        }
    err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (err == cudaSuccess) done.push_back(Entry{kernel, dev, bytes});
    return err;
}

// Rows [start, end) of a packed sequence cannot be rows of a tensor of N.  (end - start may leave int's range.)
__device__ __forceinline__ bool rows_malformed(int start, int end, int N) { return start < 0 || end < start || end > N; }

// ---- internal launchers (defined in the .cu files, called from api.cu) ----------------------

struct SeqArgs {
    int B, H, N, dk, dv, C, NC;
    int io;                       // hgrn2_dtype
    const void *o, *f, *i;        // inputs
    const float *S0;              // nullable
    void *y;                      // fwd out (nullable: states only)
    float *SN;                    // nullable
    float *states;                // [B*H][NC][dk][dv] chunk-start states: fwd writes (nullable), bwd reads
    const void *dy;               // bwd
    const float *dSN;             // nullable
    void *d_o, *d_f, *d_i;        // bwd out
    float *dS0;                   // nullable
    StatusBlock *status;
    float *room = nullptr;        // fp32 path: the workspace's room for one set of boundary states
    void *seg_scratch;            // tensor-core path: scratch for sequences split into segments (nullable)
    float *exact_scratch = nullptr;   // tensor-core backward: [work item][dk][dv] floats for the exact path
    float *totals = nullptr;      // tensor-core path: per-chunk decay totals inside the saved data (set by its launchers)
    bool clear_status = false;    // the first kernel of the call zeroes the status word itself
    int start_aborted = 0;        // tensor-core path, debugging: every CTA starts as if its first wait had run out
    bool gate_enc = false;         // the f tensor holds the signed gate encoding (gated entry points)
    const int *cu = nullptr;      // packed batch: device array of B + 1 row offsets (B = sequences, N = total rows per head)
    cudaStream_t stream;
};

struct StepArgs {
    int B, H, dk, dv, io;
    int T = 1;             // tokens per launch (launch_step_multi)
    bool whole = false;    // y overlaps o or f: one CTA per unit, which reads all of a unit's gates before it writes its y
    const void *o, *f, *i;
    float *S;
    void *y;
    cudaStream_t stream;
};

// Tensor-core path: what a CTA needs, besides its launch's other arguments, to redo an item on the exact fp32 path
// (chunk_alu.cuh) after its sweep has found a decay that the rescaled operands cannot represent.  Plain pointers (the
// kernels proper work through tensor maps); o == nullptr switches the exact path off.
struct ExactArgs {
    const __nv_bfloat16 *o = nullptr, *f = nullptr, *i = nullptr, *dy = nullptr;
    __nv_bfloat16 *y = nullptr, *d_o = nullptr, *d_f = nullptr, *d_i = nullptr;
    __nv_bfloat16 *states = nullptr;    // saved chunk states: [slot][128][128] bf16
    float *scratch = nullptr;           // backward: [item][128][128] floats
};

// Tensor-core path: the work items of a launch (tc_chunk.cuh).  Packed (variable-length) batches: the sequence tensors
// are [H][T][d] and sequence b occupies the token rows [cu[b], cu[b + 1]) of every head; state u = b * H + h.
// Chunk-start states of a packed batch live in slots: segment b * G + r of a head starts at slot
// (its first row) / 64 + b * G + r of the head's spp = T / 64 + B * G + 1 (never overlapping the next segment's).
struct WorkArgs {
    int N = 0, NC = 0;             // rows per plane; chunks of a whole sequence (ordinary batch)
    int main = 0, tail = 0;        // units taken whole, units cut into segments (ordinary batch)
    int G = 1, Lc = 0;             // segments per cut unit, chunks per segment
    const int *cu = nullptr;       // packed batch: row offsets on the device
    int B = 0, H = 1, spp = 0;     // packed batch: sequences, heads, state slots per head
};

// How an ordinary batch is cut: units [0, main) run whole, the `tail` units behind them as G segments of Lc chunks (the
// last one shorter).  tail == 0: nothing is cut.
struct SegPlan {
    int main, tail, G, Lc;
    bool gain;             // the cut is expected to pay
};
SegPlan     tc_plan(uint64_t U, int NC);
int         tc_packed_segments(uint64_t U, int T);
int         sm_count();        // SMs of the current device (0: no device)
constexpr uint32_t kFlagNoSegments = 0x40000000u;      // desc->flags, internal: no sequence is cut (needs no scratch for it)
struct TcWork {
    WorkArgs wk;
    uint64_t items = 0;    // CTAs of the launch
    uint64_t cut = 0;      // units run as G segments each
    uint64_t planes = 0;   // planes of the sequence tensors
    uint64_t slots = 0;    // chunk-state slots
    uint64_t chunks = 0;   // of an item, on average
    float *chain = nullptr, *lam = nullptr;    // chain slots [cut][G][128][128] and the segments' decays [cut][G][128]
    int *redo = nullptr;   // whole-chunk sequences: [cut][2], see redo_claim (tc_chunk.cuh)
};
TcWork      tc_work(SeqArgs &a);
cudaError_t launch_seg_chain(bool bwd, const TcWork &t, const float *init, float *fin, cudaStream_t stream);
// State-only passes (chunk_tc_state.cu): the segments of t that its chain needs - all of them for the states behind the
// last (in front of the first) one - or one span per plane.
cudaError_t launch_tc_state(bool bwd, const void *o, const void *f, const void *w, const TcWork &t, bool all, bool gate_enc,
                            StatusBlock *status, bool clear, int start_aborted, cudaStream_t stream);
cudaError_t launch_tc_span(bool bwd, const void *o, const void *f, const void *w, uint64_t planes, int N, float *out,
                           float *lam, StatusBlock *status, bool clear, int start_aborted, cudaStream_t stream);
cudaError_t launch_step(const StepArgs &a);
bool        step_multi_supported(int dk, int dv);
cudaError_t launch_step_multi(const StepArgs &a);
int         alu_default_chunk(int dk, int dv);
bool        alu_chunk_supported(int dk, int dv, int C);
cudaError_t launch_alu_fwd(const SeqArgs &a);
cudaError_t launch_alu_bwd(const SeqArgs &a);
// fp32 kernels, parallel over chunks (chunk_fp32.cu)
bool        fp32_bwd_supported(const SeqArgs &a);
int         fp32_dbeta_rows(int N);          // rows of partial sums per unit (gated backward)
cudaError_t launch_fp32_fwd(const SeqArgs &a);
cudaError_t launch_fp32_bwd(const SeqArgs &a);
cudaError_t launch_fp32_fwd_gated(const SeqArgs &a, const float *beta);
cudaError_t launch_fp32_bwd_gated(const SeqArgs &a, const float *beta, float *partial);

}  // namespace hgrn2
