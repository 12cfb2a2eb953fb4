// Quantized adapters (Sec. 3.3 "Low-rank Adapter Quantization": 4-bit AbsMax, groups of 128 elements
// share one parameter).  Storage and arithmetic as include/slim.h states them: a group is 128
// consecutive elements of a row (rows run along the contraction axis), its bf16 scale is absmax / 7
// (binary32 division, nearest-even to bf16), a code is clamp(rint(a / scale), -8, 7) with the division
// in binary32, two codes per byte (even column in the low nibble).
#include "common.cuh"

namespace slim {

// A group's scale, from its largest magnitude, and the codes of VALS of its elements.
template <int VALS>
__device__ __forceinline__ uint32_t adapter_codes(const float (&v)[VALS], float m, __nv_bfloat16* scale)
{
    *scale = m > 0.f ? __float2bfloat16_rn(__fdiv_rn(m, 7.0f)) : __float2bfloat16_rn(0.f);
    const float sc = __bfloat162float(*scale);
    const Divisor by(sc > 0.f ? sc : 1.f);
    uint32_t w = 0;
#pragma unroll
    for (int i = 0; i < VALS; ++i)
        w |= (sc > 0.f ? (uint32_t)max(-8, min(7, __float2int_rn(by.of(v[i])))) & 0xFu : 0u) << (4 * i);      // nearest, ties to even
    return w;
}

// Rows of a multiple of eight elements: 16 lanes per (row, group), eight elements a lane (one 16-byte load, one 4-byte
// store), two groups' loads in flight.  Bound by instructions: four elements a lane took the adapters of a 4096 -> 11008 layer,
// rank 416, 13.3 + 5.8 us, this 10.3 + 5.4.
__global__ void __launch_bounds__(256)
pack_adapter_kernel(const __nv_bfloat16* A, uint32_t items, int cols, int groups, uint8_t* codes, __nv_bfloat16* scales)
{
    after_previous_grid();
    constexpr int K = 2;
    const int lane = threadIdx.x & 15;
    const uint32_t first = (blockIdx.x * 16 + (threadIdx.x >> 4)) * K;
    uint4 u[K];
    uint32_t row[K];
    int c[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t item = first + k;
        row[k] = item / (uint32_t)groups;
        c[k] = (int)(item - row[k] * (uint32_t)groups) * 128 + lane * 8;
        u[k] = item < items && c[k] < cols ? *reinterpret_cast<const uint4*>(A + (size_t)row[k] * cols + c[k]) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        float v[8];
        const uint32_t w[4] = {u[k].x, u[k].y, u[k].z, u[k].w};
        float m = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[i]));
            v[2 * i] = f.x; v[2 * i + 1] = f.y;
            m = fmaxf(m, fmaxf(fabsf(f.x), fabsf(f.y)));
        }
#pragma unroll
        for (int o = 8; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        __nv_bfloat16 sc;
        const uint32_t q = adapter_codes<8>(v, m, &sc);
        if (first + k < items) {
            if (lane == 0) scales[first + k] = sc;
            if (c[k] < cols) *reinterpret_cast<uint32_t*>(codes + ((size_t)row[k] * cols + c[k]) / 2) = q;
        }
    }
}

// Any even number of columns: a warp per (row, group), four elements (two pairs) a lane.
__global__ void __launch_bounds__(256)
pack_adapter_pairs_kernel(const __nv_bfloat16* A, uint32_t items, int cols, int groups, uint8_t* codes, __nv_bfloat16* scales)
{
    after_previous_grid();
    const int lane = threadIdx.x & 31;
    const uint32_t item = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (item >= items) return;
    const uint32_t row = item / (uint32_t)groups;
    const int c = (int)(item - row * (uint32_t)groups) * 128 + lane * 4;
    float v[4];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const uint32_t w = c + 2 * i < cols ? *reinterpret_cast<const uint32_t*>(A + (size_t)row * cols + c + 2 * i) : 0u;
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w));
        v[2 * i] = f.x; v[2 * i + 1] = f.y;
    }
    float m = fmaxf(fmaxf(fabsf(v[0]), fabsf(v[1])), fmaxf(fabsf(v[2]), fabsf(v[3])));
#pragma unroll
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    __nv_bfloat16 sc;
    const uint32_t q = adapter_codes<4>(v, m, &sc);
    if (lane == 0) scales[item] = sc;
    uint8_t* dst = codes + ((size_t)row * cols + c) / 2;
    if (c < cols) dst[0] = (uint8_t)q;
    if (c + 2 < cols) dst[1] = (uint8_t)(q >> 8);
}

// Expansion to bf16 of one matrix or of a layer's two: a thread takes four bytes of codes (eight values, one 16-byte
// store) where rows are multiples of eight elements, else four times two bytes or one.  (One byte a thread and a launch per matrix took
// 11 us for the adapters of a 1728 -> 5120 layer, rank 176; a dependent launch of one byte a thread 11.2 us for 5000 x 1004, 4.3 so.)
struct Unpack { const uint8_t* codes; const __nv_bfloat16* scales; __nv_bfloat16* out; int cols, groups; size_t items; };

// I: the type of an item's number; TWO: two matrices.
template <int BYTES, typename I, bool TWO>
__global__ void __launch_bounds__(256)
unpack_adapter_kernel(const Unpack a, const Unpack b)
{
    after_previous_grid();
    constexpr int kItems = BYTES == 4 ? 1 : 4;
#pragma unroll
    for (int n = 0; n < kItems; ++n) {
        I i = ((I)blockIdx.x * kItems + n) * 256 + threadIdx.x;
        const bool second = TWO && i >= (I)a.items;
        if (second) i -= (I)a.items;
        const Unpack& m = second ? b : a;
        if (i >= (I)m.items) return;
        const uint32_t per_row = (uint32_t)m.cols / (2 * BYTES), row = (uint32_t)(i / per_row), c = (uint32_t)(i - (I)row * per_row) * (2 * BYTES);
        const float sc = __bfloat162float(m.scales[(size_t)row * m.groups + c / 128]);
        const size_t at = (size_t)row * m.cols + c;
        const uint8_t* from = m.codes + at / 2;
        const uint32_t w = BYTES == 4 ? *reinterpret_cast<const uint32_t*>(from) : BYTES == 2 ? *reinterpret_cast<const uint16_t*>(from) : *from;
        uint32_t o[4];
#pragma unroll
        for (int k = 0; k < BYTES; ++k) {
            const int lo = (int)(w << (28 - 8 * k)) >> 28, hi = (int)(w << (24 - 8 * k)) >> 28;
            __nv_bfloat162 v = __floats2bfloat162_rn((float)lo * sc, (float)hi * sc);
            o[k] = *reinterpret_cast<uint32_t*>(&v);
        }
        if (BYTES == 4) *reinterpret_cast<uint4*>(m.out + at) = make_uint4(o[0], o[1], o[2], o[3]);
        else if (BYTES == 2) *reinterpret_cast<uint2*>(m.out + at) = make_uint2(o[0], o[1]);
        else *reinterpret_cast<uint32_t*>(m.out + at) = o[0];
    }
}

slim_status_t launch_pack_adapter(const __nv_bfloat16* A, int rows, int cols, uint8_t* codes, __nv_bfloat16* scales, cudaStream_t st)
{
    const int groups = (cols + 127) / 128;
    const long long items = (long long)rows * groups;
    if (items > 0x7FFFFFFFll) return SLIM_ERR_INVALID_ARG;
    if (cols % 8 == 0) launch_dependent(pack_adapter_kernel, dim3((unsigned)((items + 31) / 32)), dim3(256), 0, st, A, (uint32_t)items, cols, groups, codes, scales);
    else launch_dependent(pack_adapter_pairs_kernel, dim3((unsigned)((items + 7) / 8)), dim3(256), 0, st, A, (uint32_t)items, cols, groups, codes, scales);
    count_launch(1);
    return cudaGetLastError() == cudaSuccess ? SLIM_OK : SLIM_ERR_CUDA;
}

static Unpack unpack_of(const uint8_t* codes, const __nv_bfloat16* scales, int rows, int cols, __nv_bfloat16* out, int bytes) {
    return Unpack{codes, scales, out, cols, (cols + 127) / 128, (size_t)rows * (cols / 2) / bytes};
}
template <int BYTES, bool TWO>
static slim_status_t launch_unpack(const Unpack& a, const Unpack& b, cudaStream_t st) {
    const size_t items = a.items + b.items, per_block = BYTES == 4 ? 256 : 1024;      // 2^32 and more: 64-bit numbers
    launch_dependent(items <= 0xFFFFF000u ? unpack_adapter_kernel<BYTES, uint32_t, TWO> : unpack_adapter_kernel<BYTES, uint64_t, TWO>,
                     dim3((unsigned)((items + per_block - 1) / per_block)), dim3(256), 0, st, a, b);
    count_launch(1);
    return cudaGetLastError() == cudaSuccess ? SLIM_OK : SLIM_ERR_CUDA;
}

slim_status_t launch_unpack_adapter(const uint8_t* codes, const __nv_bfloat16* scales, int rows, int cols, __nv_bfloat16* out,
                                    cudaStream_t st)
{
    const Unpack none = {};
    return cols % 8 == 0   ? launch_unpack<4, false>(unpack_of(codes, scales, rows, cols, out, 4), none, st)
           : cols % 4 == 0 ? launch_unpack<2, false>(unpack_of(codes, scales, rows, cols, out, 2), none, st)
                           : launch_unpack<1, false>(unpack_of(codes, scales, rows, cols, out, 1), none, st);
}

slim_status_t launch_unpack_adapters(const uint8_t* Lq, const __nv_bfloat16* Ls, const uint8_t* Rq, const __nv_bfloat16* Rs, int d_out, int r,
                                     int d_in, __nv_bfloat16* L, __nv_bfloat16* R, cudaStream_t st)
{
    return launch_unpack<4, true>(unpack_of(Lq, Ls, d_out, r, L, 4), unpack_of(Rq, Rs, r, d_in, R, 4), st);       // r % 16 == 0, d_in % 64 == 0
}

}  // namespace slim
