// Shared declarations of libsste's translation units: the context, argument
// checks and the small device helpers every kernel uses.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "sste.h"

// The context owns nothing but views into the caller's workspace.
struct sste_ctx {
    int device;
    int sm_count;
    unsigned int *status_dev;   // device status word (first word of the workspace)
    unsigned int *counter_dev;  // ticket counter of the beta reduction
    double *partials_dev;       // 2 doubles per reduction block
    void *cu_tensor_map_encode; // cuTensorMapEncodeTiled, resolved through the runtime
    float *splitk_partials;         // fp32 partial tiles of split-K products; null if the workspace is minimal
    unsigned int *splitk_tickets;   // arrival counters of the split tiles, zero between launches
    size_t splitk_partial_bytes;
    unsigned int *zero_after;       // a word that every product empties when it starts; null but in a layer call's own copy
};

constexpr int SSTE_MAX_REDUCE_BLOCKS = 1024;
constexpr size_t SSTE_WS_STATUS_OFF = 0;
constexpr size_t SSTE_WS_COUNTER_OFF = 64;
constexpr size_t SSTE_WS_PARTIALS_OFF = 256;
constexpr size_t SSTE_WS_BYTES = SSTE_WS_PARTIALS_OFF + 2 * sizeof(double) * SSTE_MAX_REDUCE_BLOCKS;
// optional tail of the workspace, used by split-K products: arrival counters, then partial tiles
constexpr int SSTE_SPLITK_TICKETS = 8192;
constexpr size_t SSTE_WS_SPLITK_TICKETS_OFF = (SSTE_WS_BYTES + 1023) / 1024 * 1024;
constexpr size_t SSTE_WS_SPLITK_PARTIALS_OFF = SSTE_WS_SPLITK_TICKETS_OFF + SSTE_SPLITK_TICKETS * sizeof(unsigned int);
// room that a dense copy of the weight in the workspace leaves to the partials: the most a plan asks for on 148 SMs
// (73 split tiles x 4 ranges x 256 KB)
constexpr size_t SSTE_DENSE_COPY_RESERVE = size_t(80) << 20;
constexpr size_t SSTE_WS_RECOMMENDED_BYTES = SSTE_WS_SPLITK_PARTIALS_OFF + (size_t(192) << 20);

static inline bool sste_mult128(int v) { return v > 0 && (v % 128) == 0; }
static inline bool sste_aligned(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

#define SSTE_CUDA_TRY(expr)                         \
    do {                                            \
        cudaError_t e__ = (expr);                   \
        if (e__ != cudaSuccess) return SSTE_ERR_CUDA; \
    } while (0)

// Make `ctx->device` current for the duration of a call.
struct sste_device_guard {
    int prev = -1;
    bool ok = true;
    explicit sste_device_guard(int dev)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) { ok = false; return; }
        if (prev != dev && cudaSetDevice(dev) != cudaSuccess) ok = false;
        if (prev == dev) prev = -1;
    }
    ~sste_device_guard()
    {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

// Runs `fn` once per device ordinal (and again after a failure); thread-safe.
struct DeviceOnce {
    static constexpr int MAX_DEVICES = 64;
    std::mutex mu;
    bool done[MAX_DEVICES] = {};
    template <typename F>
    bool run(int device, F fn)
    {
        if (device < 0 || device >= MAX_DEVICES) return fn();
        std::lock_guard<std::mutex> lock(mu);
        if (!done[device]) done[device] = fn();
        return done[device];
    }
};

// ---------------------------------------------------------------- device helpers

__device__ __forceinline__ float sste_bf16_bits_to_f32(uint32_t bits16) { return __uint_as_float(bits16 << 16); }

// fp32 -> bf16 bits, round to nearest even (finite inputs)
__device__ __forceinline__ uint32_t sste_f32_to_bf16_bits(float f)
{
    return static_cast<uint32_t>(__bfloat16_as_ushort(__float2bfloat16_rn(f)));
}

__device__ __forceinline__ uint32_t sste_f32_to_e4m3(float f)
{
    return static_cast<uint32_t>(__nv_cvt_float_to_fp8(f, __NV_SATFINITE, __NV_E4M3));
}

__device__ __forceinline__ uint32_t sste_f32_to_e5m2(float f)
{
    return static_cast<uint32_t>(__nv_cvt_float_to_fp8(f, __NV_SATFINITE, __NV_E5M2));
}

// FP8 per-tensor scaling (Sec. 5.2): scale = fp8_max / amax, 1 for an all-zero tensor.  Every kernel that
// quantises or rescales forms the scale from the tensor's amax with exactly these single-rounded operations.
__device__ __forceinline__ float sste_scale_from_amax(float amax, float fp8_max)
{
    return (amax == 0.0f) ? 1.0f : __fdiv_rn(fp8_max, amax);
}
// factor that undoes the scales of two quantised operands in a product's epilogue: fl(fl(1/sa) * fl(1/sb))
__device__ __forceinline__ float sste_out_scale(const float *a_amax, float a_fp8_max, const float *b_amax, float b_fp8_max)
{
    if (!a_amax || !b_amax) return 1.0f;
    const float ia = __fdiv_rn(1.0f, sste_scale_from_amax(*a_amax, a_fp8_max));
    const float ib = __fdiv_rn(1.0f, sste_scale_from_amax(*b_amax, b_fp8_max));
    return __fmul_rn(ia, ib);
}
static inline float sste_fp8_max(sste_dtype dt) { return dt == SSTE_E4M3 ? 448.0f : dt == SSTE_E5M2 ? 57344.0f : 0.0f; }

// Byte offset of (row m, K-offset k) inside a 2 KB metadata atom of 128 rows x 128 logical K.
__device__ __host__ __forceinline__ uint32_t sste_meta_atom_byte16(uint32_t m, uint32_t k)
{
    return 16u * (m & 7u) + 2u * ((m >> 3) & 1u) + 256u * (m >> 4) + 128u * ((k >> 4) & 1u) + 4u * (k >> 5) +
           ((k >> 3) & 1u);
}
__device__ __host__ __forceinline__ uint32_t sste_meta_atom_byte8(uint32_t m, uint32_t k) { return 16u * m + (k >> 3); }

// ---------------------------------------------------------------- programmatic dependent launch
// Every kernel of the path is launched with programmatic stream serialisation: its CTAs may be scheduled,
// and run their prologue (barrier and tensor-memory set-up, descriptor prefetch, index arithmetic), while the
// previous kernel of the stream is still draining.  sste_pdl_wait() returns once that previous kernel has
// finished and its writes are visible; before it a kernel reads tables only.  sste_pdl_trigger(), issued
// first thing, is what lets the NEXT kernel of the stream be scheduled early (it takes effect when every CTA
// of this grid has issued it or exited, so the successor never competes with CTAs not yet started).
__device__ __forceinline__ void sste_pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// The read-only path (__ldg, and what the compiler makes of `const T *__restrict__`) is for data that does not change while the kernel
// runs, waiting included: such loads may be moved in front of the wait (they were, in kernels that had a branch before it).  So
// the pointers that the kernel reads through are given to the wait and come out of it as new values, and reading is plain, or past
// the L1 cache for vectors that a block reads once (prune, FP8, 768 x 768 4.96 -> 4.73 us, 3072 x 768 6.2 -> 6.0).
template <typename T>
__device__ __forceinline__ void sste_fresh(T &pointer) { asm volatile("" : "+l"(pointer) : : "memory"); }
template <typename T>
__device__ __forceinline__ T sste_ld(const T *p) { return *p; }
__device__ __forceinline__ uint4 sste_ld_once(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
template <typename... T>
__device__ __forceinline__ void sste_pdl_wait(T &...read_after)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    (sste_fresh(read_after), ...);
}

template <typename... KArgs, typename... Args>
inline cudaError_t sste_launch(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                               Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// Process-wide count of kernels this library has launched (read by sste_debug_launch_count).
void sste_count_launches(int n);

// An amax pass and the kernel that quantises with its result, without a memset in front: the pass leaves the maximum in
// *scratch (zero before), the second kernel stores it in *amax_dev, and the next product of a context whose zero_after is
// scratch empties it.
sste_status sste_amax_scratch(sste_ctx *ctx, const void *x, size_t n, float *amax_dev, void *scratch, void *stream);
sste_status sste_quantize_scratch(sste_ctx *ctx, const void *x, size_t n, float *amax_dev, void *scratch, void *q, void *stream);
sste_status sste_mvue_scratch(sste_ctx *ctx, const void *dY, int T, int O, uint64_t seed, uint32_t tensor_id, uint32_t step,
                              uint64_t token_offset, int counter_cols, float *g_amax_dev, void *scratch, void *gvals,
                              void *gmeta, void *dense_q_out, void *stream);
// sste_project_amax without a memset: 8 bytes of scratch, zero before and after.
sste_status sste_project_amax_scratch(sste_ctx *ctx, const void *W, int O, int I, const float *beta_dev, float *amax_dev,
                                      void *scratch, void *stream);

// words of a maximum that a kernel's blocks share: the tail of a layer's scratch, zero between launches
constexpr int SSTE_MAX_SLOTS = (SSTE_LAYER_SCRATCH_BYTES - 8) / 4;
// sste_amax and sste_quantize_fp8 (E4M3) in one launch, where the tensor is small enough.
bool sste_amax_quantize_fits(const sste_ctx *ctx, size_t n);
sste_status sste_amax_quantize(sste_ctx *ctx, const void *x, size_t n, float *amax_dev, unsigned int *slots, void *q, void *stream);
// The same for sste_project_amax and sste_project_compress (E4M3).
bool sste_project_fp8_fits(const sste_ctx *ctx, int O, int I);
sste_status sste_project_fp8(sste_ctx *ctx, const void *W, int O, int I, const float *beta_dev, float *amax_dev, unsigned int *slots,
                             void *vals, void *meta, void *dense_out, void *stream);

// grad_W and grad_X of a layer (the two products behind sste_linear_bwd_weight and sste_linear_bwd_input, same arguments), in
// one launch where that is possible.
sste_status sste_bwd_products(sste_ctx *ctx, const void *gvals, const void *gmeta, const void *X, const void *dY, int O, int I,
                              int T, sste_dtype gdt, sste_dtype wdt, const void *w_dense, const void *vals, const void *meta,
                              const float *g_amax, const float *x_amax, const float *w_amax, void *dW, void *dX,
                              sste_dtype odt, void *stream);
// Whether that is one launch for these sizes (multiples of 128; elt: bytes of an operand's element); beside: whether it also beats the
// two side by side on two streams.
bool sste_bwd_in_one_launch(const sste_ctx *ctx, int elt, int O, int I, int T, bool dense_copy, sste_dtype odt, bool beside);

// two sste_crop_2d in one launch (arguments as checked by that call)
sste_status sste_crop_two(sste_ctx *ctx, const void *src0, int rows_p0, int cols_p0, void *dst0, int rows0, int cols0,
                          const void *src1, int rows_p1, int cols_p1, void *dst1, int rows1, int cols1, void *stream);

// sste_pad_2d of dY [rows, cols] into dYp [T, O] and sste_mvue_sparsify (bf16) of the result, in one pass.
sste_status sste_mvue_padded(sste_ctx *ctx, const void *dY, int rows, int cols, void *dYp, int T, int O, uint64_t seed,
                             uint32_t tensor_id, uint32_t step, uint64_t token_offset, int counter_cols, void *gvals,
                             void *gmeta, void *stream);
