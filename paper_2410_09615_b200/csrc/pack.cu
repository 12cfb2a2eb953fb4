// Packer / metadata encoder and its inverse.  Integer-only, HBM-bound:
// 2 B read + 0.375 B written per dense weight.
#include "common.cuh"

namespace slim {

// One thread handles 16 consecutive columns (four groups) of one row: two
// 16-byte loads, one 4-byte and one 2-byte store.  Consecutive threads walk
// consecutive columns, so a warp reads 512 contiguous bytes of codes and mask.
// The four mask bytes of a group become a 4-bit number; a 16-entry table in shared memory gives its index nibble and
// the byte selector that picks the two codes.  Bound by the integer pipe and the L2: 4096 x 11008 53 us with a loop over
// positions, 26 with the table in a 64-bit number and emulated byte comparisons (about 30 operations a group), 21 with byte tests for any
// mask byte and each group for itself (22 operations), now 19.
//
// A table entry: bits 0-15 the selector of the two kept codes, bits 16-19 the index nibble (lower | upper << 2), bit 31 more than
// two positions are kept.  A set of fewer than two is completed with the lowest positions not kept.
__device__ __forceinline__ uint32_t index_entry(uint32_t m) {
    const int kept = __popc(m);
    int p0 = 0, p1 = 1;
    if (kept == 1 || kept == 2) {
        p0 = __ffs(m) - 1;
        p1 = kept == 2 ? 31 - __clz(m) : p0;
        if (kept == 1) { if (p0 == 0) p1 = 1; else p0 = 0; }
    }
    return (uint32_t)(p0 | p1 << 4) | 0x4400u | (uint32_t)(p0 | p1 << 2) << 16 | (kept > 2 ? 1u << 31 : 0u);
}

// Four bytes of value nibbles from eight codes, a byte each.
__device__ __forceinline__ uint32_t nibbles(uint32_t t0, uint32_t t1) {
    return __byte_perm((t0 & 0x000F000Fu) | ((t0 >> 4) & 0x00F000F0u), (t1 & 0x000F000Fu) | ((t1 >> 4) & 0x00F000F0u), 0x6420);
}

__global__ void __launch_bounds__(256)
pack_kernel(const int8_t* codes, const uint8_t* mask, long long n_chunks, uint8_t* vals, uint8_t* meta, uint32_t* status_dev)
{
    __shared__ uint32_t table[16];
    if (threadIdx.x < 16) table[threadIdx.x] = index_entry(threadIdx.x);
    after_previous_grid();
    __syncthreads();
    uint32_t err = 0;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n_chunks;
         c += (long long)gridDim.x * blockDim.x) {
        const uint4 cv = reinterpret_cast<const uint4*>(codes)[c], mv = reinterpret_cast<const uint4*>(mask)[c];
        const uint32_t cw[4] = {cv.x, cv.y, cv.z, cv.w}, mw[4] = {mv.x, mv.y, mv.z, mv.w};
        uint32_t vout, mout;
        // Masks of zeros and ones, as they come: a multiplication each (on the other pipe) for the table's index and for the kept bytes, and
        // the nibbles of two groups are put together at a time.  `two[g]`: the two codes of a group, `e[g]` its table entry.
        uint32_t e[4], two[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            e[g] = table[(mw[g] * 0x10204080u) >> 28];                        // bits 0, 8, 16, 24 -> 28 .. 31
            two[g] = __byte_perm(cw[g] & (mw[g] * 0xFFu), 0u, e[g]);          // bytes: lower, upper
        }
        const uint32_t t0 = __byte_perm(two[0], two[1], 0x5410), t1 = __byte_perm(two[2], two[3], 0x5410);
        const uint32_t range = ((t0 ^ (t0 >> 1)) | (t1 ^ (t1 >> 1))) & 0x78787878u;          // bits 3 .. 7 of a code are its sign
        const uint32_t other = (mw[0] | mw[1] | mw[2] | mw[3]) & 0xFEFEFEFEu, many = (e[0] | e[1] | e[2] | e[3]) & 0x80000000u;
        if ((range | other | many) == 0) {
            vout = nibbles(t0, t1);
            const uint32_t n = __byte_perm(__byte_perm(e[0], e[1], 0x0062), __byte_perm(e[2], e[3], 0x0062), 0x5410) & 0x0F0F0F0Fu;
            mout = __byte_perm((n & 0x000F000Fu) | ((n >> 4) & 0x00F000F0u), 0u, 0x4420);
        } else {
            vout = mout = 0;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const uint32_t h = (((mw[g] & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | mw[g]) & 0x80808080u;      // bit 7 of a byte: kept
                uint32_t keep;                                                    // 0xFF at kept positions
                asm("prmt.b32 %0, %1, %1, 0xBA98;" : "=r"(keep) : "r"(h));
                uint32_t e = table[(h * 0x00204081u) >> 28];                      // bits 7, 15, 23, 31 -> 28 .. 31
                uint32_t two = __byte_perm(cw[g] & keep, 0u, e);                  // bytes: lower, upper
                const bool range = ((two ^ (two >> 1)) & 0x7878u) != 0;           // bits 3 .. 7 of a code are its sign
                if ((int)e < 0 || range) {
                    err |= 1u << ((int)e < 0 ? SLIM_ERR_BAD_MASK : SLIM_ERR_CODE_RANGE);
                    two = 0; e = 4u << 16;
                }
                const uint32_t vb = (two & 0xFu) | ((two >> 4) & 0xF0u);
                vout |= vb << (8 * g);
                mout |= ((e >> 16) & 0xFu) << (4 * g);
            }
        }
        reinterpret_cast<uint32_t*>(vals)[c] = vout;
        reinterpret_cast<uint16_t*>(meta)[c] = (uint16_t)mout;
    }
    if (err && status_dev) atomicOr(status_dev, err);
}

__global__ void __launch_bounds__(256)
unpack_kernel(const uint8_t* __restrict__ vals, const uint8_t* __restrict__ meta,
              long long n_chunks, int8_t* __restrict__ codes, uint8_t* __restrict__ mask)
{
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n_chunks;
         c += (long long)gridDim.x * blockDim.x) {
        const uint32_t vw = __ldg(reinterpret_cast<const uint32_t*>(vals) + c);
        const uint32_t mw = __ldg(reinterpret_cast<const uint16_t*>(meta) + c);
        uint32_t cw[4], kw[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const uint32_t vb = (vw >> (8 * g)) & 0xFFu;
            const uint32_t m = (mw >> (4 * g)) & 0xFu;
            const int p0 = m & 3, p1 = (m >> 2) & 3;
            const int c0 = ((int)((vb & 0xFu) << 28)) >> 28;
            const int c1 = ((int)((vb >> 4) << 28)) >> 28;
            uint32_t cwv = ((uint32_t)c0 & 0xFFu) << (8 * p0);
            cwv = (cwv & ~(0xFFu << (8 * p1))) | (((uint32_t)c1 & 0xFFu) << (8 * p1));
            cw[g] = cwv;
            kw[g] = (1u << (8 * p0)) | (1u << (8 * p1));
        }
        reinterpret_cast<int4*>(codes)[c] = make_int4((int)cw[0], (int)cw[1], (int)cw[2], (int)cw[3]);
        if (mask) reinterpret_cast<int4*>(mask)[c] = make_int4((int)kw[0], (int)kw[1], (int)kw[2], (int)kw[3]);
    }
}

static int grid_for(long long n_chunks, int sm_count) {
    long long blocks = (n_chunks + 255) / 256;
    long long cap = (long long)sm_count * 8;     // grid-stride over a full machine
    return (int)(blocks < cap ? (blocks < 1 ? 1 : blocks) : cap);
}

slim_status_t launch_pack(const int8_t* codes, const uint8_t* mask, int d_out, int d_in,
                          uint8_t* vals, uint8_t* meta, uint32_t* status_dev, cudaStream_t st)
{
    slim_status_t err;
    const DeviceInfo* di = device_info(&err);
    if (!di) return err;
    const long long n_chunks = (long long)d_out * d_in / 16;
    launch_dependent(pack_kernel, dim3((unsigned)grid_for(n_chunks, di->sm_count)), dim3(256), 0, st, codes, mask, n_chunks, vals, meta, status_dev);
    count_launch(1);
    return cudaGetLastError() == cudaSuccess ? SLIM_OK : SLIM_ERR_CUDA;
}

slim_status_t launch_unpack(const uint8_t* vals, const uint8_t* meta, int d_out, int d_in,
                            int8_t* codes, uint8_t* mask, cudaStream_t st)
{
    slim_status_t err;
    const DeviceInfo* di = device_info(&err);
    if (!di) return err;
    const long long n_chunks = (long long)d_out * d_in / 16;
    unpack_kernel<<<grid_for(n_chunks, di->sm_count), 256, 0, st>>>(vals, meta, n_chunks, codes, mask);
    count_launch(1);
    return cudaGetLastError() == cudaSuccess ? SLIM_OK : SLIM_ERR_CUDA;
}

}  // namespace slim
