// Quantized adapters (Sec. 3.3 "Low-rank Adapter Quantization": 4-bit AbsMax, groups of 128 elements
// share one parameter).  Storage and arithmetic as include/slim.h states them: a group is 128
// consecutive elements of a row (rows run along the contraction axis), its bf16 scale is absmax / 7
// (binary32 division, nearest-even to bf16), a code is clamp(rint(a / scale), -8, 7) with the division
// in binary32, two codes per byte (even column in the low nibble).
#include "common.cuh"

namespace slim {

// One warp per (row, group): a lane holds four consecutive elements (one 8-byte load where rows are multiples of
// four elements).  Warps walk the groups with the next group's load in flight.
__device__ __forceinline__ uint2 load_group(const __nv_bfloat16* __restrict__ A, uint32_t item, int cols, int groups, int lane)
{
    const int c0 = (int)(item % (uint32_t)groups) * 128 + lane * 4;
    const __nv_bfloat16* src = A + (size_t)(item / (uint32_t)groups) * cols + c0;
    if (cols % 4 == 0) return c0 < cols ? __ldg(reinterpret_cast<const uint2*>(src)) : make_uint2(0u, 0u);
    uint32_t w[2] = {0, 0};                                   // cols is even: elements come in pairs
#pragma unroll
    for (int i = 0; i < 2; ++i) if (c0 + 2 * i < cols) w[i] = __ldg(reinterpret_cast<const uint32_t*>(src) + i);
    return make_uint2(w[0], w[1]);
}

__global__ void __launch_bounds__(256)
pack_adapter_kernel(const __nv_bfloat16* __restrict__ A, uint32_t items, int cols, int groups,
                    uint8_t* __restrict__ codes, __nv_bfloat16* __restrict__ scales)
{
    const int lane = threadIdx.x & 31;
    const uint32_t stride = gridDim.x * 8;
    uint32_t item = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (item >= items) return;
    uint2 next = load_group(A, item, cols, groups, lane);
    for (; item < items; item += stride) {
        const uint2 u = next;
        if (item + stride < items) next = load_group(A, item + stride, cols, groups, lane);
        const uint32_t row = item / (uint32_t)groups, grp = item % (uint32_t)groups;
        const int c0 = (int)grp * 128 + lane * 4;
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x)), b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
        const float v[4] = {a.x, a.y, b.x, b.y};
        // magnitudes order like their bit patterns
        const float m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(fmaxf(fabsf(v[0]), fabsf(v[1])), fmaxf(fabsf(v[2]), fabsf(v[3]))))));
        const __nv_bfloat16 sb = m > 0.f ? __float2bfloat16_rn(__fdiv_rn(m, 7.0f)) : __float2bfloat16_rn(0.f);
        const float sc = __bfloat162float(sb);
        if (lane == 0) scales[(size_t)row * groups + grp] = sb;
        const Divisor by(sc > 0.f ? sc : 1.f);
        uint32_t q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            q[i] = sc > 0.f ? (uint32_t)max(-8, min(7, __float2int_rn(by.of(v[i])))) & 0xFu : 0u;      // nearest, ties to even
        // cols is even, so elements come in pairs: either both of a byte exist or neither
        uint8_t* dst = codes + (size_t)row * (cols / 2) + c0 / 2;
        if (c0 + 3 < cols) {
            const uint16_t w = (uint16_t)(q[0] | (q[1] << 4) | (q[2] << 8) | (q[3] << 12));
            if (cols % 4 == 0) *reinterpret_cast<uint16_t*>(dst) = w;
            else { dst[0] = (uint8_t)w; dst[1] = (uint8_t)(w >> 8); }
        } else if (c0 + 1 < cols) {
            dst[0] = (uint8_t)(q[0] | (q[1] << 4));
        }
    }
}

// One thread per byte of codes: two bf16 values out.
__global__ void unpack_adapter_kernel(const uint8_t* __restrict__ codes, const __nv_bfloat16* __restrict__ scales, int rows,
                                      int cols, int groups, __nv_bfloat16* __restrict__ out)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t half = (size_t)cols / 2;
    if (i >= (size_t)rows * half) return;
    const int row = (int)(i / half), c = 2 * (int)(i % half);
    const float sc = __bfloat162float(scales[(size_t)row * groups + c / 128]);
    const uint32_t B = codes[i];
    const int lo = (int)(B & 0xFu), hi = (int)(B >> 4);
    const float a = (float)(lo >= 8 ? lo - 16 : lo) * sc, b = (float)(hi >= 8 ? hi - 16 : hi) * sc;
    *reinterpret_cast<__nv_bfloat162*>(out + (size_t)row * cols + c) = __floats2bfloat162_rn(a, b);
}

slim_status_t launch_pack_adapter(const __nv_bfloat16* A, int rows, int cols, uint8_t* codes, __nv_bfloat16* scales, cudaStream_t st)
{
    const int groups = (cols + 127) / 128;
    const long long items = (long long)rows * groups;
    if (items > 0x7FFFFFFFll) return SLIM_ERR_INVALID_ARG;
    const long long blocks = (items + 7) / 8;
    pack_adapter_kernel<<<(unsigned)(blocks < 1184 ? blocks : 1184), 256, 0, st>>>(A, (uint32_t)items, cols, groups, codes, scales);      // 1184: eight blocks for each of 148 SMs
    count_launch(1);
    return cudaGetLastError() == cudaSuccess ? SLIM_OK : SLIM_ERR_CUDA;
}

slim_status_t launch_unpack_adapter(const uint8_t* codes, const __nv_bfloat16* scales, int rows, int cols, __nv_bfloat16* out,
                                    cudaStream_t st)
{
    const size_t n = (size_t)rows * (cols / 2);
    unpack_adapter_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(codes, scales, rows, cols, (cols + 127) / 128, out);
    count_launch(1);
    return cudaGetLastError() == cudaSuccess ? SLIM_OK : SLIM_ERR_CUDA;
}

}  // namespace slim
