// Shared device/host helpers of libslim (CUDA side only).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include "slim.h"

namespace slim {

// Bit a device-detected error sets in the caller's status word.
__device__ __forceinline__ void flag_error(uint32_t* status_dev, int code) {
    if (status_dev) atomicOr(status_dev, 1u << code);
}

__host__ __device__ __forceinline__ int ceil_div(int a, int b) { return (a + b - 1) / b; }

// x / b correctly rounded, for many x and one b: Markstein's theorem (IBM J. Res. Dev. 34, 1990): with y = 1 / b
// correctly rounded and q within an ulp of x / b, q + (x - q b) y, two fused operations, is x / b correctly
// rounded, unless b's significand is all ones.  That case, and magnitudes near the ends of the range, take the
// ordinary division.  (An |x| below 2^-100 may come out inexact: then x / b is below 2^-39 and the callers round it to zero.)
struct Divisor {
    float b, y;
    bool plain;
    __device__ __forceinline__ explicit Divisor(float d) : b(d) {
        y = __frcp_rn(d);
        plain = (__float_as_uint(d) & 0x7FFFFFu) == 0x7FFFFFu || !(d >= 0x1p-60f && d <= 0x1p60f);
    }
    __device__ __forceinline__ float of(float x) const {
        if (plain) return __fdiv_rn(x, b);
        float q = __fmul_rn(x, y);
        q = __fmaf_rn(__fmaf_rn(-q, b, x), y, q);
        return __fmaf_rn(__fmaf_rn(-q, b, x), y, q);
    }
};

// Programmatic dependent launch for the short kernels that follow each other (compressing a 4096 x 11008 layer, 8
// launches: 238 -> 228 us):
// a grid is set up while the one before it in the stream ends, and starts to read and write when that one is complete.
// What that grid may have written is read with ordinary loads behind the wait: __ldg and const __restrict__ promise data that stays
// the same for the whole life of the grid, which begins before the wait, and such a load may be moved ahead of it.
__device__ __forceinline__ void after_previous_grid() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... P, typename... A>
cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Per-device facts the launchers need (filled once per device, read-only after).
struct DeviceInfo {
    int cc_major;
    int sm_count;
};
const DeviceInfo* device_info(slim_status_t* err);

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link against libcuda);
// nullptr when the driver does not have it.  Thread-safe.
void* tensor_map_encoder();

// The words that CTAs hand to one another have a region of this fixed size right after the sync words, whatever the problem: the
// small-batch kernel's T = X R^T, the pair kernel's {part written, tile ready}.  Each carries the number of the call that wrote it
// (handover.h), so kernels and shapes may take turns there as long as every one of them that does counts each of its calls,
// also those that hand nothing over (the pair kernel without adapters), and nothing is written there without a number.
constexpr size_t kSmallTBytes = 512 << 10;
constexpr int kSmallMaxRank = 3072;

// T = X R^T is handed from one product to the next in bf16 (one rounding) or, where keeps_T32() holds, as two bf16 numbers
// whose sum is the 32-bit value to 17 bits: these are the shapes that the CUDA-core kernel, which keeps T in 32 bits, served
// before the tensor-core kernels took them.  The T L^T product then runs twice over the same L (on the GPU, 1728 -> 5120, int4
// adapters, 600 tokens: 25.0 -> 26.6 us; 5504 -> 4096, 4 tokens: 8.4 -> 8.6, 16 tokens: 11.0 -> 12.0).  Relative error of Y against 64 bits,
// X, L, R normal: 0.00170 with one rounding of T, 0.00165 so and on the CUDA cores, of which 0.00165 are the rounding of Y.
inline bool keeps_T32(int b, int d_out, int d_in, int r) {
    if (b > 16) return d_in % 128 != 0 || d_out % 128 != 0;
    return d_in % 256 != 0 || d_in > 32768 || (b > 8 && r > 2560);
}
// The first number: the bf16 nearest to v (where that would overflow, the next towards zero).
__device__ __forceinline__ float bf16_head(float v) {
    const float h = __bfloat162float(__float2bfloat16_rn(v));
    return fabsf(h) <= 3.4e38f ? h : __uint_as_float(__float_as_uint(v) & 0xFFFF0000u);
}
// The rest, for the second (infinities and NaN are in the first).
__device__ __forceinline__ float bf16_tail(float v) {
    const float rest = v - bf16_head(v);
    return fabsf(rest) <= 3.4e38f ? rest : 0.f;
}

// Launch bookkeeping for slim_last_launch_count().
void count_launch(int n);
void reset_launch_count();
void note_token_tile(int n);      // token-tile width of the prefill main launch, for slim_last_token_tile()

// ---- launchers (defined in the kernel files) --------------------------------
slim_status_t launch_pack(const int8_t* codes, const uint8_t* mask, int d_out, int d_in,
                          uint8_t* vals, uint8_t* meta, uint32_t* status_dev, cudaStream_t st);
slim_status_t launch_unpack(const uint8_t* vals, const uint8_t* meta, int d_out, int d_in,
                            int8_t* codes, uint8_t* mask, cudaStream_t st);

size_t simple_workspace_bytes(int b, int d_out, int d_in, int r);
slim_status_t launch_simple(const __nv_bfloat16* X, int b, const uint8_t* vals, const uint8_t* meta,
                            float s, const __nv_bfloat16* L, const __nv_bfloat16* R, int r,
                            int d_out, int d_in, __nv_bfloat16* Y, void* ws, cudaStream_t st);

// Up to 64 tokens.  `tiled` (decode-tiled copy, up to 16 tokens) or vals / meta; Ls == nullptr: L and R are bf16
// matrices, else the code bytes of quantized adapters.
bool small_supports(int b, int d_out, int d_in, int r);
slim_status_t launch_small(const __nv_bfloat16* X, int b, const uint8_t* vals, const uint8_t* meta, const uint8_t* tiled, float s,
                           const void* L, const void* R, const __nv_bfloat16* Ls, const __nv_bfloat16* Rs, int r, int d_out, int d_in,
                           __nv_bfloat16* Y, void* ws, uint32_t* status_dev, cudaStream_t st);

slim_status_t launch_repack_tiled(const uint8_t* vals, const uint8_t* meta, int d_out, int d_in, uint8_t* out, cudaStream_t st);

slim_status_t launch_pack_adapter(const __nv_bfloat16* A, int rows, int cols, uint8_t* codes, __nv_bfloat16* scales, cudaStream_t st);
slim_status_t launch_unpack_adapter(const uint8_t* codes, const __nv_bfloat16* scales, int rows, int cols, __nv_bfloat16* out,
                                    cudaStream_t st);

slim_status_t launch_unpack_adapters(const uint8_t* Lq, const __nv_bfloat16* Ls, const uint8_t* Rq, const __nv_bfloat16* Rs, int d_out, int r,
                                     int d_in, __nv_bfloat16* L, __nv_bfloat16* R, cudaStream_t st);

slim_status_t launch_mask_top2(const int8_t* codes, const float* xbar, int d_out, int d_in, uint8_t* mask, uint32_t* status_dev,
                               cudaStream_t st);
size_t quant_workspace_bytes(int d_out, int d_in);
slim_status_t launch_quant(const float* W, int d_out, int d_in, int8_t* codes, float* scale_alpha, void* ws,
                           uint32_t* status_dev, cudaStream_t st);

bool prefill_supports(int b, int d_out, int d_in, int r);
size_t prefill_workspace_bytes(int b, int d_out, int d_in, int r);
slim_status_t launch_prefill(const __nv_bfloat16* X, int b, const uint8_t* vals, const uint8_t* meta,
                             float s, const __nv_bfloat16* L, const __nv_bfloat16* R, int r,
                             int d_out, int d_in, __nv_bfloat16* Y, void* ws, uint32_t* status_dev,
                             cudaStream_t st, bool force_pair = false, bool automatic = false);

}  // namespace slim
