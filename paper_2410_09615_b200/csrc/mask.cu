// slim_mask_top2: the 2:4 mask of the pipeline's second step (Sec. 3, Fig. 1; metric: Sec. 3.2, the product
// of weight and input magnitudes).  One thread per group of four along d_in: metric |code| * xbar[k] (one
// binary32 multiplication; xbar == nullptr: |code|), the two largest kept, equal metrics to the lower
// index.  1 B read + 1 B written per weight, and the integer pipe: a group costs it 13
// operations, the six comparisons being subtractions on the other pipe whose sign bits are voted on.  4096 x 11008: 57 us with
// one thread per group, 30 with four groups a thread and comparisons on the integer pipe (about 30 operations), now 20.
#include "common.cuh"

namespace slim {

// Bit 31: a < b, for a and b other than -0.  (A difference of two distinct numbers is never zero when nothing is flushed, that of
// two equal ones +0; inf - inf is positive here.)
__device__ __forceinline__ uint32_t less(float a, float b) {
    float d;
    asm("sub.rn.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return __float_as_uint(d);
}
__device__ __forceinline__ uint32_t majority(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (a & c) | (b & c); }

__device__ __forceinline__ uint32_t top2(uint32_t c, const float4* x)
{
    // codes as floats: code + 128 in the significand of 2^23, less 2^23 + 128; then magnitudes
    const uint32_t biased = c ^ 0x80808080u;
    float m[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) m[k] = fabsf(__uint_as_float(__byte_perm(biased, 0x4B000000u, 0x7440 + k)) - 8388736.f);
    // the product plus zero, in one rounding: the product itself, but +0 for -0 (an input magnitude may be -0)
    if (x) { m[0] = __fmaf_rn(m[0], x->x, 0.f); m[1] = __fmaf_rn(m[1], x->y, 0.f); m[2] = __fmaf_rn(m[2], x->z, 0.f); m[3] = __fmaf_rn(m[3], x->w, 0.f); }
    // l_ij, i < j, in bit 31: entry i loses to entry j (equal metrics: the lower index wins).  An entry is kept when it beats
    // at least two of the other three: a majority of three, one logic operation.
    const uint32_t l01 = less(m[0], m[1]), l02 = less(m[0], m[2]), l03 = less(m[0], m[3]), l12 = less(m[1], m[2]), l13 = less(m[1], m[3]), l23 = less(m[2], m[3]);
    const uint32_t k0 = majority(~l01, ~l02, ~l03), k1 = majority(l01, ~l12, ~l13), k2 = majority(l02, l12, ~l23), k3 = majority(l03, l13, l23);
    // prmt with its sign mode: a byte of ones for a set bit 31
    uint32_t p, q;
    asm("prmt.b32 %0, %1, %2, 0xFBFB;" : "=r"(p) : "r"(k0), "r"(k1));
    asm("prmt.b32 %0, %1, %2, 0xFBFB;" : "=r"(q) : "r"(k2), "r"(k3));
    return __byte_perm(p, q, 0x7610) & 0x01010101u;
}

// A thread owns V (four, or one where a row is no multiple of four groups) groups of columns and walks rows: its input
// magnitudes stay in registers, and it has the loads of ROWS rows in flight.  A block is up to 256 V groups of columns by as many
// rows as make up 256 threads and leave two blocks an SM (100000 x 64: 27.8 us with one row a block, 4.8 so); where blocks of
// several rows a thread would not give every SM one, a thread takes one (64 x 4096: 3.2 us with four, 2.0 so).
template <int V> struct Words;
template <> struct Words<4> { using T = uint4; };
template <> struct Words<1> { using T = uint32_t; };

// Codes are read once: past the L1.  (Volatile: not moved ahead of the wait.)
__device__ __forceinline__ uint4 load_once(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t load_once(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.global.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

template <bool XBAR, int V, int ROWS, bool LANES>
__global__ void __launch_bounds__(256)
mask_top2_kernel(const typename Words<V>::T* codes, const float* xbar, int per_row, int d_out, typename Words<V>::T* mask, uint32_t* status)
{
    using T = typename Words<V>::T;
    after_previous_grid();
    const int g = blockIdx.x * blockDim.x + threadIdx.x, lanes = LANES ? blockDim.y : 1;
    if (g >= per_row) return;
    float4 x[V];
#pragma unroll
    for (int v = 0; v < V && XBAR; ++v) {
        x[v] = reinterpret_cast<const float4*>(xbar)[(size_t)g * V + v];
        if (blockIdx.y == 0 && !(x[v].x >= 0.f && x[v].x <= 3.0e38f && x[v].y >= 0.f && x[v].y <= 3.0e38f && x[v].z >= 0.f && x[v].z <= 3.0e38f && x[v].w >= 0.f && x[v].w <= 3.0e38f))
            flag_error(status, SLIM_ERR_INVALID_ARG);
    }
    const size_t step = (size_t)lanes * per_row;
    for (uint32_t row0 = blockIdx.y * ROWS * lanes + (LANES ? threadIdx.y : 0u); row0 < (uint32_t)d_out; row0 += gridDim.y * ROWS * lanes) {
        const size_t at = (size_t)row0 * per_row + g;
        T c[ROWS] = {};
        const T* from = codes + at;
#pragma unroll
        for (int i = 0; i < ROWS; ++i, from += step) if (row0 + i * lanes < (uint32_t)d_out) c[i] = load_once(from);
        T* to = mask + at;
#pragma unroll
        for (int i = 0; i < ROWS; ++i, to += step) {
            T o;
#pragma unroll
            for (int v = 0; v < V; ++v)
                reinterpret_cast<uint32_t*>(&o)[v] = top2(reinterpret_cast<const uint32_t*>(&c[i])[v], XBAR ? &x[v] : nullptr);
            if (row0 + i * lanes < (uint32_t)d_out) *to = o;
        }
    }
}

template <int V, int ROWS>
static void launch_mask(const int8_t* codes, const float* xbar, int d_out, int d_in, uint8_t* mask, uint32_t* status_dev, cudaStream_t st)
{
    using T = typename Words<V>::T;
    const int per_row = d_in / (4 * V), cols = per_row < 256 ? per_row : 256, blocks = ceil_div(per_row, cols);
    const int most = 256 / cols, spread = d_out / (ROWS * 2 * 148), lanes = spread < 1 ? 1 : spread < most ? spread : most;
    const int strips = ceil_div(d_out, ROWS * lanes);
    if (ROWS > 1 && (long long)strips * blocks < 148) { launch_mask<V, 1>(codes, xbar, d_out, d_in, mask, status_dev, st); return; }
    const T* c = reinterpret_cast<const T*>(codes);
    T* m = reinterpret_cast<T*>(mask);
    auto* kernel = lanes > 1 ? (xbar ? mask_top2_kernel<true, V, ROWS, true> : mask_top2_kernel<false, V, ROWS, true>)
                             : (xbar ? mask_top2_kernel<true, V, ROWS, false> : mask_top2_kernel<false, V, ROWS, false>);
    launch_dependent(kernel, dim3((unsigned)blocks, (unsigned)(strips < 65535 ? strips : 65535)),
                     dim3((unsigned)cols, (unsigned)lanes), 0, st, c, xbar, per_row, d_out, m, status_dev);
}

slim_status_t launch_mask_top2(const int8_t* codes, const float* xbar, int d_out, int d_in, uint8_t* mask, uint32_t* status_dev,
                               cudaStream_t st)
{
    if (d_in % 16 == 0) launch_mask<4, 4>(codes, xbar, d_out, d_in, mask, status_dev, st);
    else launch_mask<1, 16>(codes, xbar, d_out, d_in, mask, status_dev, st);
    count_launch(1);
    return cudaGetLastError() == cudaSuccess ? SLIM_OK : SLIM_ERR_CUDA;
}

}  // namespace slim
