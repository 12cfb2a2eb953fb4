// Prefill-phase forward (many tokens): tcgen05 tensor cores with the accumulator
// in tensor memory.
//
// Two kernels: persistent CTA pairs on 256-row tiles (prefill_pair_kernel, further down, with what it does otherwise), and, where
// those would be too few, one CTA per 128-row tile.  The text here describes the latter and what they share.
//
// One CTA computes a 128 (output rows) x N (64 tokens; up to 256 in the dense-only launch) tile of
//     out[token][row] = scale * ( sum_k W[row][k] X[token][k]  +  sum_j A2[row][j] B2[token][j] )
// in two chained phases that accumulate into the same TMEM tile:
//   phase 1 (sparse): W is the packed int4 2:4 weight.  TMA brings 128 rows of value
//       bytes and index bytes plus the X tile; eight converter warps (two groups on
//       alternate stages, one thread per weight row) expand nibbles to exact bf16 into the
//       64-byte-swizzled K-major layout the MMA reads, and write the 2:4 index words into
//       tensor memory; one thread issues tcgen05.mma.sp (kind::f16, bf16 x bf16 -> fp32).
//   phase 2 (dense): A2 and B2 are bf16 matrices brought by TMA as they are; the same
//       thread issues tcgen05.mma into the same accumulator.
// The layer forward is two or three launches:
//   T' = (X R^T) / s          phase 2 only (A2 = R, B2 = X, scale 1/s), bf16 into the workspace, in one or two parts
//                             (keeps_T32; two: the main launch's dense stages take a column block of either in turn).
//                             The product has few tiles, so K is split over blockIdx.z; the
//                             slices write fp32 partial tiles and a small kernel adds them in a
//                             fixed order (one slice: bf16 directly, no second launch).
//   Y  = s * (X Q^T + T' L^T) phase 1 then phase 2 (A2 = L, B2 = T', scale s)
// so the adapter product and the scale are fused into the tile loop and the epilogue.
//
// Index words in tensor memory (one 32-bit column per MMA of 32 weight columns): lane
// l holds 16 of the 32 columns (half (l / 8) % 2) of two rows, row l & ~8 in bits
// 0-15 and row l | 8 in bits 16-31; the MMA addresses an even column pair and a
// selector bit of the instruction descriptor picks the column.  A 32-bit word of the
// packed index array is one row's 32 columns, so a converter thread swaps one
// half-word with the thread eight rows away and stores the result.
// Source of the layout: PTX ISA, "tcgen05.mma.sp" -- "Sparse matrices" / "Sparsity selector" for
// kind::f16 (which bits of the metadata columns in tensor memory describe which chunk of A, and
// how the selector picks a column of a pair); the one-hot and exact-integer tests check it.
//
// Pipeline.  A ring of stages {B: token rows x 128 bytes, A: 8 KB (16 KB in the dense-only
// launch)}; a sparse stage is 64 weight columns (two MMAs of K = 32), a dense stage 32 columns
// (two MMAs of K = 16; 64 columns in the dense-only launch).  The packed value and index bytes
// travel separately, 256 columns (4 stages) per TMA tile, through a ring of their own.
// Warps: 0-7 converters, then epilogue; 8 and 10 token tiles of even / odd stages (with the A2
// tile in phase 2); 9 MMA issue; 11 packed tiles.
// mbarriers: b_full / pk_full (TMA bytes landed), conv_done (converters finished a stage),
// empty / pk_empty (tcgen05.commit: the MMAs that read the stage are complete; converters
// done with a packed slot), acc_full.
// Measured on B200 and built into the loops below: a barrier operation is served per thread
// (a warp-wide try_wait or 32 arrivals cost 32 times one); the answer of a try_wait takes about
// 200 cycles even when the phase is long complete, so waits that follow each other are asked
// together; a lane left at a warp barrier while another lane of its warp spins costs some hundred
// nanoseconds per iteration; a lane that walks alone takes 120 cycles to issue an MMA.
// Every wait is bounded; an expired one sets SLIM_ERR_TIMEOUT and the kernel runs on.
#include <atomic>
#include <cuda.h>
#include "common.cuh"
#include "handover.h"
#include "pair_plan.h"
#include "turns.h"

namespace slim {

constexpr int kPM = 128;            // output rows per CTA (MMA M)
constexpr int kPBK = 64;            // columns of a TMA box of bf16 (128 bytes)
constexpr int kPkCols = 256;        // weight columns of one packed tile
constexpr int kConvWarps = 8;       // warps 0-7 converters / epilogue
constexpr int kWarpXEven = 8, kWarpMma = 9, kWarpXOdd = 10, kWarpPk = 11;
constexpr int kPThreads = 32 * 12;
constexpr int kATile = kPM * 128;               // 16 KB: 128 rows x 128 bytes (dense phase)
constexpr int kValsTile = kPM * (kPkCols / 4);  // 8 KB: 64 value bytes per row
constexpr int kMetaTile = kPM * (kPkCols / 8);  // 4 KB: 32 index bytes per row
constexpr int kPkSlotBytes = kValsTile + kMetaTile;
constexpr uint32_t kPSpinLimit = 1u << 21;

// The one-CTA kernel.  PRE = the dense-only launch (T' product): no packed tiles, so the room goes to more stages.
template <int N, bool PRE = false> struct PfCfg {
    static constexpr int kSK = 64;                                          // weight columns of a sparse stage
    static constexpr int kPkStages = kPkCols / kSK;                         // stages covered by one packed tile
    static constexpr int kBTile = N * 128;
    // A region of a stage: the expanded weight tile needs 8 KB.  The main launch's dense stages are 32 columns wide so
    // that their A2 tile fits there too: a smaller stage means more stages in flight, and the loop is bound by the
    // latency of the token tile.  The dense-only launch has no expanded tiles and keeps 64-column stages.
    static constexpr int kARegion = PRE ? kATile : kPM * kSK;
    static constexpr int kDK = PRE ? 64 : 32;                               // columns of a dense stage
    static constexpr int kStages = PRE && N >= 256 ? 4 : 8;
    static constexpr int kPkSlots = PRE ? 1 : 7;                            // packed tiles come from HBM: the ring holds what fits
    static constexpr int kStageBytes = kBTile + kARegion;
    static constexpr int kECol = N;                                         // index words: N + 4 * stage + mma
    static constexpr int kTmemCols = N >= 256 ? 512 : 128;
    static constexpr size_t kSmem = 1024 + (size_t)kStages * kStageBytes + kPkSlots * kPkSlotBytes + 1024;
};

struct alignas(128) PrefillParams {      // (so are the tensor maps behind it in the parameters: none lies across two lines)
    __nv_bfloat16* out;     // [tokens][ldo]
    int ldo;
    int m_total;            // valid output rows
    int b;                  // valid tokens
    int t_parts;            // bf16 matrices [b][r], one behind the other, whose sum is T' (keeps_T32): 1 or 2
    int n1, n2;             // stages of the sparse and of the dense phase
    float scale;
    uint32_t* status;
    // dense-only launch split along K over blockIdx.z: slice z covers `k_per` stages from z * k_per and
    // writes its fp32 partial tile to part[z][token][ldo] (part == nullptr: one slice, bf16 to out)
    float* part;
    int k_per;
    // Index bytes by cp.async where a tensor map cannot describe their rows (d_in / 8 bytes, no 16-byte
    // multiple): the array and its row pitch; nullptr: by TMA.
    const uint8_t* meta;
    int meta_pitch;
    int d_in;
    // pair kernel: pairs of 128-row tiles; tiles of 256 x 256 in all
    int row_pairs, tiles, half;          // half: token rows one CTA loads, half of a tile's tokens
    // T' inside the pair kernel: chunks of t_n columns (of r), tiles of 256 tokens x t_n, 64-column stages of one, pairs that
    // share the work; 1 / s; T' itself, partial tiles, and per (tile, CTA) {arrivals, ready} words that carry the call number
    int r, t_n, t_chunks, t_tiles, t_stages, t_pairs;
    int t_even;             // parts of a T' tile where all have as many, else 0
    float t_scale;
    __nv_bfloat16* t_out;
    float4* t_part;
    unsigned long long* t_sync;
    unsigned long long* departures;
};

// Optional timeline: built with -DSLIM_PREFILL_TRACE, one thread per warp role of the first
// CTAs records the global timer around its waits for the first 48 stages.
#ifdef SLIM_PREFILL_TRACE
#ifndef SLIM_PTRACE_PRE
#define SLIM_PTRACE_PRE 0          // 1: stamp the dense-only launch instead of the main one
#endif
__device__ unsigned long long g_ptrace[8][6][48];
#define PSTAMP(role, it) do { if (PRE == (SLIM_PTRACE_PRE != 0) && blockIdx.z == 0 && blockIdx.x + gridDim.x * blockIdx.y < 8 && (it) < 48) { unsigned long long t_; \
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_)); g_ptrace[blockIdx.x + gridDim.x * blockIdx.y][role][it] = t_; } } while (0)
#else
#define PSTAMP(role, it) do { } while (0)
#endif

namespace pf {

__device__ __forceinline__ uint32_t s32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(s32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(s32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(s32(bar)), "r"(bytes) : "memory");
}
// Bounded wait.  The first wait of a CTA that expires raises `*abort_flag`; every later
// wait of the CTA then gives up at once, so a broken pipeline costs one time-out, not many.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag) {
    const uint32_t addr = s32(bar);
    for (uint32_t it = 0; it < kPSpinLimit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done) : "r"(addr), "r"(parity) : "memory");
        if (done) return true;
        if (*abort_flag) return false;
    }
    *abort_flag = 1u;
    return false;
}
__device__ __forceinline__ void tma_tile(void* dst, const CUtensorMap* tmap, int x, int y, uint64_t* bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 :: "r"(s32(dst)), "l"(tmap), "r"(x), "r"(y), "r"(s32(bar)) : "memory");
}

// Shared-memory matrix descriptor: K-major tile of 128-byte rows, 128-byte swizzle,
// 8-row groups 1024 bytes apart (descriptor version 1).
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// Same with 64-byte rows and 64-byte swizzle (8-row groups 512 bytes apart).
__device__ __forceinline__ uint64_t smem_desc64(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(512 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}
// Instruction descriptor, kind::f16: fp32 accumulate, bf16 A and B, both K-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mma_dense(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        :: "r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// A holds the two kept values of every group of four; e_tmem addresses the index words.
__device__ __forceinline__ void mma_sparse(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t e_tmem,
                                           uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.sp.cta_group::1.kind::f16 [%0], %1, %2, [%3], %4, p;\n\t}"
        :: "r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(e_tmem), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(s32(bar)) : "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) { asm volatile("prefetch.tensormap [%0];" :: "l"(map) : "memory"); }
// A tile into the L2.
__device__ __forceinline__ void prefetch_tile(const CUtensorMap* tmap, int x, int y) {
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" :: "l"(tmap), "r"(x), "r"(y) : "memory");
}
// ---- CTA-pair variants.  The sparse one reads A from tensor memory: lane = row, two stored bf16 per column.  Shared-memory operands are
// given by the low word of their descriptor (128-byte rows; the high word is the same for all): the issuing warp shares its scheduler with the
// converters, and what it spends on a stage is instructions.
constexpr uint32_t kDescHi = (uint32_t)(1024 >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return ((saddr & 0x3FFFFu) >> 4) | (1u << 16); }
__device__ __forceinline__ void mma_dense2(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "mov.b64 a, {%1, %5};\n\tmov.b64 b, {%2, %5};\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, p;\n\t}"
        :: "r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(accumulate), "r"(kDescHi) : "memory");
}
__device__ __forceinline__ void mma_sparse2(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t e_tmem,
                                            uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 b;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 b, {%2, %6};\n\t"
        "tcgen05.mma.sp.cta_group::2.kind::f16 [%0], [%1], b, [%3], %4, p;\n\t}"
        :: "r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(e_tmem), "r"(idesc), "r"(accumulate), "r"(kDescHi) : "memory");
}
// The same for a pair's loads: the bytes are counted on the even CTA's barrier.
__device__ __forceinline__ void tma_tile_pair(void* dst, const CUtensorMap* tmap, int x, int y, uint32_t cluster_bar_addr) {
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 :: "r"(s32(dst)), "l"(tmap), "r"(x), "r"(y), "r"(cluster_bar_addr) : "memory");
}
__device__ __forceinline__ void tma_tile_pair3(void* dst, const CUtensorMap* tmap, int y, int z, uint32_t cluster_bar_addr) {
    asm volatile("cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 :: "r"(s32(dst)), "l"(tmap), "r"(0), "r"(y), "r"(z), "r"(cluster_bar_addr) : "memory");
}
// Address of the same shared-memory object in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(s32(p)), "r"(rank));
    return r;
}
// Completion of this thread's earlier MMAs arrives on the same barrier of both CTAs of the pair.
__device__ __forceinline__ void mma_commit2(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 :: "r"(s32(bar)), "h"((uint16_t)3) : "memory");
}
// Arrival on a barrier of another CTA of the cluster, ordered like a CTA-local arrival.
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_bar_addr) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" :: "r"(cluster_bar_addr) : "memory");
}
__device__ __forceinline__ void mbar_arrive_remote_release(uint32_t cluster_bar_addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" :: "r"(cluster_bar_addr) : "memory");
}
// One try_wait, no loop.  `cluster`: acquire at cluster scope (arrivals came from the other CTA).
__device__ __forceinline__ uint32_t mbar_try(uint64_t* bar, uint32_t parity, bool cluster) {
    uint32_t done;
    if (cluster)
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(s32(bar)), "r"(parity) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(s32(bar)), "r"(parity) : "memory");
    return done;
}
// The same question without waiting (try_wait holds the thread for a while when the answer is no).
__device__ __forceinline__ uint32_t mbar_test(uint64_t* bar, uint32_t parity, bool cluster) {
    uint32_t done;
    if (cluster)
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(s32(bar)), "r"(parity) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(s32(bar)), "r"(parity) : "memory");
    return done;
}
// Bounded wait for several barriers at once.  A try_wait takes about 200 cycles to answer even when
// the phase is long complete, so waits that follow each other are asked together, not in turn.
__device__ __forceinline__ bool mbar_wait_all(uint64_t* b0, uint32_t p0, bool c0, uint64_t* b1, uint32_t p1, bool c1,
                                              uint64_t* b2, uint32_t p2, bool c2, volatile uint32_t* abort_flag) {
    for (uint32_t it = 0; it < kPSpinLimit; ++it) {
        const uint32_t d0 = b0 ? mbar_try(b0, p0, c0) : 1u;
        const uint32_t d1 = b1 ? mbar_try(b1, p1, c1) : 1u;
        const uint32_t d2 = b2 ? mbar_try(b2, p2, c2) : 1u;
        if (d0 & d1 & d2) return true;
        if (*abort_flag) return false;
    }
    *abort_flag = 1u;
    return false;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
    return pred != 0;
}
__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Two int4 codes of byte `T` of w -> exact bf16x2: nibble ^ 8 in the mantissa of 128.0
// is 128 + (v + 8); subtracting 136 leaves v in [-8, 7].
template <int T>
__device__ __forceinline__ uint32_t nib2bf16(uint32_t w, uint32_t w_shr4) {
    uint32_t x, y;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(x) : "r"(w), "r"(w_shr4), "n"(T * 0x1111 + 0x4400));
    asm("lop3.b32 %0, %1, %2, %3, 0x6a;" : "=r"(y) : "r"(x), "r"(0x000F000Fu), "r"(0x43084308u));
    __nv_bfloat162 v = *reinterpret_cast<__nv_bfloat162*>(&y);
    const uint32_t bias_bits = 0x43084308u;
    v = __hsub2(v, *reinterpret_cast<const __nv_bfloat162*>(&bias_bits));
    return *reinterpret_cast<uint32_t*>(&v);
}

// 32 consecutive 32-bit columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 16 consecutive 32-bit columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float4 (&v)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[0].z), "=f"(v[0].w), "=f"(v[1].x), "=f"(v[1].y), "=f"(v[1].z), "=f"(v[1].w),
                   "=f"(v[2].x), "=f"(v[2].y), "=f"(v[2].z), "=f"(v[2].w), "=f"(v[3].x), "=f"(v[3].y), "=f"(v[3].z), "=f"(v[3].w) : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint4 (&a)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
                 "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
                 :: "r"(taddr), "r"(a[0].x), "r"(a[0].y), "r"(a[0].z), "r"(a[0].w), "r"(a[1].x), "r"(a[1].y), "r"(a[1].z), "r"(a[1].w),
                    "r"(a[2].x), "r"(a[2].y), "r"(a[2].z), "r"(a[2].w), "r"(a[3].x), "r"(a[3].y), "r"(a[3].z), "r"(a[3].w),
                    "r"(a[4].x), "r"(a[4].y), "r"(a[4].z), "r"(a[4].w), "r"(a[5].x), "r"(a[5].y), "r"(a[5].z), "r"(a[5].w),
                    "r"(a[6].x), "r"(a[6].y), "r"(a[6].z), "r"(a[6].w), "r"(a[7].x), "r"(a[7].y), "r"(a[7].z), "r"(a[7].w) : "memory");
}
__device__ __forceinline__ void epilogue_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

}  // namespace pf

// One packed tile (128 rows x 256 weight columns, group `kg` along them) into a slot; called by a whole warp.
__device__ __forceinline__ void load_packed(const PrefillParams& p, const CUtensorMap* tmV, const CUtensorMap* tmM, unsigned char* slot,
                                            uint64_t* full, int kg, int m0, int lane)
{
    using namespace pf;
    if (elect_one()) {
        mbar_expect_tx(full, (uint32_t)(p.meta ? kValsTile : kPkSlotBytes));
        tma_tile(slot, tmV, kg * 64, m0, full);
        if (!p.meta) tma_tile(slot + kValsTile, tmM, kg * 32, m0, full);
    }
    if (p.meta) {
        // 128 rows x four 8-byte pieces (64 columns each), stored as the TMA's 32-byte swizzle would: a lane has the rows r0 + 8 i, which all
        // have the same swizzle
        const int q = lane & 3, r0 = lane >> 2;
        const bool col_in = kg * 32 + q * 8 < p.meta_pitch;
        const int rows = col_in ? (p.m_total - m0 - r0 + 7) / 8 : 0;
        const uint8_t* src = p.meta + (rows > 0 ? (size_t)(m0 + r0) * p.meta_pitch + kg * 32 + q * 8 : 0);
        const size_t step = rows > 0 ? (size_t)8 * p.meta_pitch : 0;
        const uint32_t d = s32(slot + kValsTile) + r0 * 32 + ((((q >> 1) ^ (r0 >> 2)) & 1) << 4) + (q & 1) * 8;
#pragma unroll
        for (int i = 0; i < kPM / 8; ++i, src += i < rows ? step : 0)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" :: "r"(d + i * 256), "l"(src), "r"(i < rows ? 8 : 0) : "memory");
        asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" :: "r"(s32(full)) : "memory");
    }
}

// One weight row of a stage of SK (64 or 128) columns, the q-th of its packed tile: 16 value bytes -> 32 bf16 per 64
// columns, and the row's part of the index words of
// the stage's MMAs (layout in the file header).  The packed tiles are stored with the 64-byte (values) and 32-byte
// (indices) TMA swizzles so that a warp's row-strided reads spread over the banks.  Rows past the last (!row_in) and columns
// past it (cols_left) get a legal pair of positions.
template <int SK>
__device__ __forceinline__ void expand_row(const unsigned char* pk, int row, int q, int x, bool row_in, int cols_left, uint4 (&a)[SK / 16], uint32_t (&e)[SK / 32])
{
#pragma unroll
    for (int hh = 0; hh < SK / 64; ++hh) {
        const int qq = q * (SK / 64) + hh;                   // which 64 columns of the packed tile
        const uint4 v = *reinterpret_cast<const uint4*>(pk + row * 64 + (((qq ^ (row >> 1)) & 3) << 4));
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint32_t ws = w[c] >> 4;
            a[hh * 4 + c] = make_uint4(pf::nib2bf16<0>(w[c], ws), pf::nib2bf16<1>(w[c], ws), pf::nib2bf16<2>(w[c], ws), pf::nib2bf16<3>(w[c], ws));
        }
        uint2 mw2 = *reinterpret_cast<const uint2*>(pk + kValsTile + row * 32 + ((((qq >> 1) ^ (row >> 2)) & 1) << 4) + (qq & 1) * 8);
        if (!row_in || hh * 64 >= cols_left) mw2 = make_uint2(0x44444444u, 0x44444444u);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t mw = h ? mw2.y : mw2.x;
            const uint32_t send = x ? (mw & 0xFFFFu) : (mw >> 16);
            const uint32_t recv = __shfl_xor_sync(0xffffffffu, send, 8);
            e[hh * 2 + h] = x ? ((mw & 0xFFFF0000u) | recv) : ((mw & 0xFFFFu) | (recv << 16));
        }
    }
}
// The expanded row of a 64-column stage into the K-major A tile: 64-byte rows, 64-byte swizzle.
__device__ __forceinline__ void store_row(unsigned char* a_tile, int row, const uint4 (&a)[4])
{
#pragma unroll
    for (int c = 0; c < 4; ++c) *reinterpret_cast<uint4*>(a_tile + row * 64 + (((c ^ (row >> 1)) & 3) << 4)) = a[c];
}

template <int N, bool PRE = false>
__global__ void __launch_bounds__(kPThreads, 1)
prefill_kernel(const PrefillParams p, const __grid_constant__ CUtensorMap tmV,
               const __grid_constant__ CUtensorMap tmM, const __grid_constant__ CUtensorMap tmX,
               const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB2)
{
    using namespace pf;
    using Cfg = PfCfg<N, PRE>;
    // The dense-only launch lets the launches behind it start at once (programmatic dependent launch): the
    // main launch's sparse stages do not need T', and it waits (griddepcontrol.wait) just before its first
    // request of a T' tile.
    if (PRE) asm volatile("griddepcontrol.launch_dependents;");
    constexpr int kBTile = Cfg::kBTile, kStageBytes = Cfg::kStageBytes, kECol = Cfg::kECol, kPStages = Cfg::kStages;
    constexpr int kPkSlots = Cfg::kPkSlots, kDK = Cfg::kDK, kSK = Cfg::kSK, kPkStages = Cfg::kPkStages;
    extern __shared__ unsigned char smem_raw[];
    // layout: stages {B | A} | packed slots {value bytes | index bytes} | barriers
    unsigned char* stages = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char* packed = stages + (size_t)kPStages * kStageBytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(packed + kPkSlots * kPkSlotBytes);
    uint64_t* b_full = bars;                         // [kPStages] token tile (and A2 tile) landed
    uint64_t* conv_done = bars + kPStages;           // [kPStages]
    uint64_t* empty = bars + 2 * kPStages;           // [kPStages]
    uint64_t* pk_full = bars + 3 * kPStages;         // [kPkSlots]
    uint64_t* pk_empty = pk_full + kPkSlots;         // [kPkSlots]
    uint64_t* acc_full = pk_empty + kPkSlots;        // [1]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 1);
    volatile uint32_t* abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * kPM, n0 = blockIdx.y * N;
    const int k_first = PRE && p.part ? (int)blockIdx.z * p.k_per : 0;      // first dense stage of this K slice
    const int n_total = PRE && p.part ? min(p.k_per, p.n2 - k_first) : p.n1 + p.n2;
    // CTAs that share token rows start their walk over the weight columns at different places,
    // so that at any moment they ask the L2 for different lines of X rather than all for the same
    // ones.  The walk is rotated by whole 256-column groups.
    const int n_groups = ceil_div(p.n1, kPkStages);
    const int rot_g = (p.d_in % kPkCols == 0 && n_groups > 0)
                          ? (int)((blockIdx.x + 3u * blockIdx.y) % (unsigned)n_groups) : 0;

    if (threadIdx.x == 0) PSTAMP(5, 44);
    if (threadIdx.x == 0) {
        for (int i = 0; i < kPStages; ++i) {
            mbar_init(&b_full[i], 1);
            mbar_init(&conv_done[i], kConvWarps / 2); mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < kPkSlots; ++i) { mbar_init(&pk_full[i], p.meta ? 33 : 1); mbar_init(&pk_empty[i], kConvWarps); }
        mbar_init(acc_full, 1);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kWarpMma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(s32(tmem_slot)), "r"(Cfg::kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(tmem_slot);
    bool ok = true;
    if (threadIdx.x == 0) PSTAMP(5, 45);

    if (warp == kWarpXEven || warp == kWarpXOdd) {
        // ============================ token-tile producers ============================
        // Each of the two warps walks every second stage in order (a waiter that skipped uses of
        // a barrier would mistake an old phase for the one it needs).  Sparse stage: lane 0
        // requests the token tile.  Dense stage: lanes 0 and 1 request the token tile and the A2
        // tile with one instruction.
        bool t_ready = PRE;                                 // main launch: T' (and everything before it) is complete
        for (int it = warp == kWarpXEven ? 0 : 1; it < n_total; it += 2) {
            const int st = it % kPStages;
            const bool sparse = it < p.n1;
            if (!sparse && !t_ready) {
                asm volatile("griddepcontrol.wait;" ::: "memory");
                asm volatile("fence.proxy.async;" ::: "memory");   // the tiles are read by the async proxy
                t_ready = true;
            }
            // The whole warp waits (no lane is left behind at a warp barrier while another
            // spins: that costs some hundred nanoseconds per stage); lane 0 arms the barrier.
            if (it >= kPStages) ok = mbar_wait(&empty[st], ((it / kPStages) & 1) ^ 1, abort_flag) && ok;
            // dense stage: kDK columns of the token rows and of the A2 rows
            // dense stage: kDK columns of the token rows and of the A2 rows
            if (lane == 0) mbar_expect_tx(&b_full[st], (uint32_t)(sparse ? kBTile : (N + kPM) * kDK * 2));
            unsigned char* sbase = stages + (size_t)st * kStageBytes;
            int kb = sparse ? it + rot_g * kPkStages : it - p.n1 + k_first, y = n0;
            if (!PRE && !sparse && p.t_parts == 2) { y += (kb & 1) * p.b; kb >>= 1; }    // a column block of either part in turn
            if (sparse && kb >= p.n1) kb -= p.n1;
            const int k = kb * (sparse ? kSK : kDK);
            // lane 0: the token tile (one box); lane 1, dense stages only: the A2 tile
            if (lane == 0 || (lane == 1 && !sparse))
                tma_tile(lane == 0 ? sbase : sbase + kBTile, lane == 1 ? &tmA2 : (sparse ? &tmX : &tmB2), k, lane == 0 ? y : m0, &b_full[st]);
            if (lane == 0) PSTAMP(0, it);
        }
    } else if (warp == kWarpPk) {
        // ============================ packed-tile producer ============================
        for (int gi = 0; gi < n_groups; ++gi) {
            const int slot = gi % kPkSlots;
            const int g = gi + rot_g < n_groups ? gi + rot_g : gi + rot_g - n_groups;
            if (gi >= kPkSlots) ok = mbar_wait(&pk_empty[slot], ((gi / kPkSlots) & 1) ^ 1, abort_flag) && ok;
            load_packed(p, &tmV, &tmM, packed + slot * kPkSlotBytes, &pk_full[slot], g, m0, lane);
        }
    } else if (warp == kWarpMma) {
        // ============================ MMA issuer ============================
        // One elected lane walks the stages and issues.
        if (elect_one()) {
            constexpr uint32_t idesc = idesc_bf16(kPM, N);
            uint32_t pre = 0;       // the coming stage was found ready by an early test
            for (int it = 0; it < n_total; ++it) {
                const int st = it % kPStages;
                const uint32_t parity = (it / kPStages) & 1;
                const bool sparse = it < p.n1;
                // token tile landed; converters done
                if (!pre)
                    ok = mbar_wait_all(&b_full[st], parity, false, sparse ? &conv_done[st] : nullptr, parity, false,
                                       nullptr, 0, false, abort_flag) && ok;
                fence_after_sync();
                // ask about the next stage now, without waiting: the answer comes back while this stage's
                // MMAs are issued, and in steady state it is yes
                pre = 0;
                if (it + 1 < n_total) {
                    const int st1 = (it + 1) % kPStages;
                    const uint32_t par1 = ((it + 1) / kPStages) & 1;
                    pre = mbar_test(&b_full[st1], par1, false);
                    if (it + 1 < p.n1) pre &= mbar_test(&conv_done[st1], par1, false);
                }
                const uint32_t b_addr = s32(stages + (size_t)st * kStageBytes);
                const uint32_t a_addr = b_addr + kBTile;
                PSTAMP(3, it);
                if (sparse) {
                    // per MMA: A 16 stored bf16 (32 bytes of a row of kSK bytes), B 32 columns (64 bytes)
#pragma unroll
                    for (int j = 0; j < kSK / 32; ++j) {
                        const uint32_t acc = (it > 0 || j > 0) ? 1u : 0u;
                        const uint32_t e_col = tmem_base + kECol + 4 * st;
                        mma_sparse(tmem_base, smem_desc64(a_addr + 32 * j), smem_desc(b_addr + 64 * j), e_col, idesc | (1u << 2) | (uint32_t)j, acc);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < kDK / 16; ++j) {
                        const uint32_t acc = (it > 0 || j > 0) ? 1u : 0u;
                        // 32-column stages: 64-byte rows with the 64-byte swizzle; 64-column stages: 128-byte rows
                        if (kDK == 32) mma_dense(tmem_base, smem_desc64(a_addr + 32 * j), smem_desc64(b_addr + 32 * j), idesc, acc);
                        else           mma_dense(tmem_base, smem_desc(a_addr + 32 * j), smem_desc(b_addr + 32 * j), idesc, acc);
                    }
                }
                mma_commit(&empty[st]);             // the stage is free once these MMAs have read it
                PSTAMP(4, it);
            }
            mma_commit(acc_full);
        }
    } else {
        // ============================ converters, then epilogue ============================
        // Two groups of four warps take every second stage each, so that the latency chain of one
        // stage (load, expand, store, index words into TMEM, fences, arrival) overlaps the next
        // stage's.  Within a group a thread owns one weight row of the tile.
        const int row = threadIdx.x & 127;           // weight row inside the tile = TMEM lane
        const int half = threadIdx.x >> 7;           // converter group; in the epilogue, which half of the columns
        const int x = (row >> 3) & 1;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        for (int it = half; it < p.n1; it += 2) {
            const int st = it % kPStages;
            const int gi = it / kPkStages, q = it % kPkStages, slot = gi % kPkSlots;
            const unsigned char* pk = packed + slot * kPkSlotBytes;
            // the packed tile has landed, and the MMAs of the previous use of this stage are done with
            // its A tile and index words
            ok = mbar_wait_all(&pk_full[slot], (gi / kPkSlots) & 1, false, it >= kPStages ? &empty[st] : nullptr,
                               ((it / kPStages) & 1) ^ 1, false, nullptr, 0, false, abort_flag) && ok;
            if ((threadIdx.x & 127) == 0) PSTAMP(1, it);
            uint4 a[4];
            uint32_t e[2];
            expand_row<64>(pk, row, q, x, m0 + row < p.m_total, 64, a, e);
            store_row(stages + (size_t)st * kStageBytes + kBTile, row, a);
            fence_after_sync();                              // the MMAs have read what is stored over
            asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};"
                         :: "r"(tmem_base + lane_base + kECol + 4 * st), "r"(e[0]), "r"(e[1]) : "memory");
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // A is read by the tensor core
            fence_before_sync();
            // one arrival per warp: arrivals on one barrier are served one after another
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&conv_done[st]);
                // this group's last stage of the packed tile
                if (q + 2 >= kPkStages || it + 2 >= p.n1) mbar_arrive(&pk_empty[slot]);
            }
            if ((threadIdx.x & 127) == 0) PSTAMP(2, it);
        }
        // ---- epilogue: thread = output row, TMEM columns = tokens; the two halves split the columns
        ok = mbar_wait(acc_full, 0, abort_flag) && ok;
        fence_after_sync();
        if (threadIdx.x == 0) PSTAMP(5, 46);
        const int orow = m0 + row;
#pragma unroll 1
        for (int c0 = half * (N / 2); c0 < (half + 1) * (N / 2); c0 += 32) {
            uint32_t r[32];
            tmem_ld32(tmem_base + lane_base + c0, r);
            // what differs between the cases is decided outside the unrolled loops: this code runs once, and its size is its time
            // (the dense-only launch of 512 x 128, 300 tokens, rank 16: 16.7 us with the decisions inside, 10.9 like this)
            const int n = orow < p.m_total ? p.b - n0 - c0 : 0;
            size_t step = (size_t)p.ldo;
            asm volatile("" : "+l"(step));                     // the 32 products of it are not made ahead of the loop over c0
            auto store = [&](auto* to, auto value) {
#pragma unroll
                for (int c = 0; c < 32; ++c, to += step) if (c < n) *to = value(__uint_as_float(r[c]));
            };
            __nv_bfloat16* out = p.out + (size_t)(n0 + c0) * p.ldo + orow;
            if (PRE && p.part) {
                store(p.part + ((size_t)blockIdx.z * p.b + n0 + c0) * p.ldo + orow, [](float v) { return v; });
            } else if (PRE && p.t_parts == 2) {
#pragma unroll 1
                for (int tp = 0; tp < 2; ++tp, out += (size_t)p.b * p.ldo)
                    store(out, [&](float v) { v *= p.scale; return __float2bfloat16_rn(tp ? bf16_tail(v) : bf16_head(v)); });
            } else {
                store(out, [&](float v) { return __float2bfloat16_rn(p.scale * v); });
            }
        }
    }

    if (threadIdx.x == 0) PSTAMP(5, 47);
    if (!ok && lane == 0) flag_error(p.status, SLIM_ERR_TIMEOUT);
    fence_before_sync();
    __syncthreads();
    if (warp == kWarpMma) {
        fence_after_sync();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem_base), "r"(Cfg::kTmemCols) : "memory");
    }
}

// ---------------------------------------------------------------- the wide kernel: persistent CTA pairs
// A cluster of two CTAs computes tiles of 256 output rows x 256 tokens with cta_group::2 MMAs issued by the even CTA: each
// CTA loads and expands its own 128 rows of the weight and loads half of the token tile.  Stages are 128 weight
// columns (four MMAs of K = 32 per commit; 64 columns of the adapters in phase 2).
// The expanded weight goes to tensor memory, not to shared memory: per stage an SM's shared memory carries 76 KB (TMA
// writes 38, converters read 6, tensor core reads 32: 0.31 us at 128 bytes a cycle, as long as the MMAs take) where with
// A in shared memory it was 108 KB and 0.46 us a stage.
// The pairs are persistent: pair c takes tiles c, c + pairs, ..., and all rings run on across tiles, so that the next
// tile's operands are loaded and expanded while this tile ends.  Eight warps of their own read the accumulator out:
// 128 tokens a thread; the next tile's MMAs may start as soon as it is in registers, the stores follow beside
// them.  A CTA per tile spent 4.4 us on start-up and 2.3 us on the epilogue of every tile, with the tensor
// core idle.
// Warps: 0-15 converters (four groups, stages in turn), 16-23 epilogue, 24 and 25 token tiles (sparse stages in turn; in the others one
// requests A, one B), 26 MMA issue, 27 packed tiles.
//
// T' = (X R^T) / s is made by the same pairs first: tiles of 256 tokens x t_n columns of r (the tokens are the MMA's rows), or of 256 ranks x
// the tokens of a narrow tile (t_ranks),
// whose 64-column stages are dealt out evenly in one list, so that every pair gets the same share whatever the number
// of tiles.  Pairs that share a tile leave their parts as fp32 in the workspace; when all are there, each of them adds up a
// share of the columns, in list order, and rounds to bf16.  The main tiles wait for the T' they read just before their
// first adapter stage.  As a launch of its own (and a reduction behind it) T' took 12 us and more of most calls.
//
// N = most tokens of a tile: 256, 128 or 64 (half: half of those that it has).  The sparse MMA of 256 x N x 32 takes N / 2 cycles.  What held
// a stage at 690 cycles whatever N was what stands around it, each worth little without the others:
//   - the issuing thread: a lane walking alone needed 120 cycles an MMA and 400 and more for its barriers; a warp that walks together, asks
//     ahead and adds to the low words of its descriptors 300-400 a stage;
//   - the converters: a group takes 1400 cycles from packed bytes to the arrival, so four groups instead of two;
//   - the packed ring: 48 KB an SM, less than the HBM's latency asks for: a pair's first tile is asked into the L2 ahead.
// With up to 128 tokens a stage is a whole packed tile of 256 columns (the smaller accumulator leaves the tensor memory for it): half the
// barriers and commits a column.  8192 x 8192 without adapters, weights in rotation: 128 tokens 28.5 -> 22.4 us, 333 tokens 32.3 -> 28.3;
// 8192 -> 28672, rank 832, 40 tokens 78 -> 61; 13824 -> 5120, rank 512, 900 tokens 115 -> 110.
// What bounds it now: with 256 tokens 0.36-0.40 us a stage of 128 columns, of which the MMAs take 0.27 (the shared-memory port is busy for 0.31:
// TMA writes 38 KB, converters read 6, tensor core reads 32); with 128 tokens 0.25.  Whose turn a stage is, and why waits by parity are right: turns.h.
// A token-tile warp sees every second phase of an `empty` barrier.  Waiting by parity is still right: before its stage g it has waited
// for the MMAs of stage g - 7, so the phase it did not see (stage g - 10) is over.
constexpr int kTTok = kPairTTok;        // tokens of a T' tile (the rows of its MMA)
constexpr int kPairThreads = 28 * 32;
template <int N> struct PairCfg {
    static constexpr int kGroups = 4, kWarpEpi = 4 * kGroups, kWarpX = kWarpEpi + 8, kWarpMma = kWarpX + 2, kWarpPk = kWarpX + 3;
    static constexpr int kSK = N <= 128 ? 256 : 128, kDK = 64, kStages = 5, kPkSlots = 4, kPkStages = kPkCols / kSK;
    static constexpr int kStageBytes = 32768, kATileAt = kStageBytes / 2;     // dense stages and T': B, then A
    // tensor memory: the accumulator (a T' tile's may be as wide), index words (kSK / 32 columns a stage), expanded weights (kSK / 4
    // columns a stage)
    static constexpr int kECols = kSK / 32, kACols = kSK / 4, kECol = N <= 128 ? 128 : 256, kACol = N <= 128 ? 192 : 288;
    static_assert(kDK == kPairDK && 2 * kPM == kPairRows, "the plan's tiles");      // (a T' tile has up to kECol columns)
    static constexpr size_t kSmem = 1024 + (size_t)kStages * kStageBytes + kPkSlots * kPkSlotBytes + 384 + 8 * 1024;     // .. barriers, epilogue
    static_assert(kECol + kStages * kECols <= kACol && kACol + kStages * kACols <= 512, "tensor memory");
    static_assert(kGroups == kTurnGroups && kStages == kTurnPlaces && kPkSlots == kTurnSlots, "the turns' rings");
};
constexpr size_t kSyncTiles = kSmallTBytes / 16 - 1024;     // T' tiles whose words fit the region beside those of the pairs

__device__ __forceinline__ unsigned long long ld_acquire64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
// Waits (bounded in time) until every lane's word (nullptr: none) is this call's; called by a whole warp.
__device__ __forceinline__ bool wait_words(const unsigned long long* w, uint32_t call, volatile uint32_t* abort_flag) {
    unsigned long long t0 = 0;
    for (uint32_t it = 0;; ++it) {
        const bool there = !w || is_of(ld_acquire64(w), call);
        if (__all_sync(0xffffffffu, there)) return true;
        if (__any_sync(0xffffffffu, *abort_flag != 0)) return false;
        if ((it & 63u) == 63u) {
            unsigned long long now;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
            if (t0 == 0) t0 = now;
            else if (__any_sync(0xffffffffu, now - t0 > 2000000000ull)) { *abort_flag = 1u; return false; }
        }
    }
}

// Four neighbouring values of T', in one part or (`tail`: the way to the second) two.
__device__ __forceinline__ void store_T(__nv_bfloat16* at, size_t tail, float4 v) {
    auto put = [&](float4 q) {
        __nv_bfloat162 lo = __floats2bfloat162_rn(q.x, q.y), hi = __floats2bfloat162_rn(q.z, q.w);
        *reinterpret_cast<uint2*>(at) = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
    };
    if (tail != 0) {
        const float4 h = make_float4(bf16_head(v.x), bf16_head(v.y), bf16_head(v.z), bf16_head(v.w));
        put(h);
        at += tail;
        v = make_float4(v.x - h.x, v.y - h.y, v.z - h.z, v.w - h.w);
        if (!(fabsf(v.x) + fabsf(v.y) + fabsf(v.z) + fabsf(v.w) <= 3.4e38f))        // infinities and NaN are in the head
            v = make_float4(fabsf(v.x) <= 3.4e38f ? v.x : 0.f, fabsf(v.y) <= 3.4e38f ? v.y : 0.f, fabsf(v.z) <= 3.4e38f ? v.z : 0.f, fabsf(v.w) <= 3.4e38f ? v.w : 0.f);
    }
    put(v);
}

// Four neighbouring values of a row of a T' tile: ranks of a token, or (RANKS) tokens of a rank; in two parts where `tail` is not 0.  (Which of the
// two is known when the kernel is compiled: with the question asked at every store, and the rows worked out there, the first pass over the
// longer code made the sums 1-3 us longer: 5120 x 5120, rank 512, 720 tokens 39.6 us a call, 43.0 so; 2304 -> 1568, rank 160, 300 tokens 20.8,
// 22.3.  As a function that is called a first pass took 2 us less, every other 0.7-1 us more where T' is what a call waits for.)
template <bool RANKS>
__device__ __forceinline__ void put_T(__nv_bfloat16* out, int a_row, int b_row, int b, int r, size_t tail, float4 v)
{
    if constexpr (RANKS) {
        if (a_row >= r) return;
        const float t[4] = {v.x, v.y, v.z, v.w};
        __nv_bfloat16* at = out + (size_t)b_row * r + a_row;
#pragma unroll
        for (int i = 0; i < 4; ++i, at += r)
            if (b_row + i < b) {
                *at = __float2bfloat16_rn(tail ? bf16_head(t[i]) : t[i]);
                if (tail) at[tail] = __float2bfloat16_rn(bf16_tail(t[i]));
            }
    } else if (a_row < b && b_row < r) {
        store_T(out + (size_t)a_row * r + b_row, tail, v);
    }
}

template <int N, bool RANKS>
__global__ void __launch_bounds__(kPairThreads, 1)
prefill_pair_kernel(const PrefillParams p, const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmM,
                    const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB2,
                    const __grid_constant__ CUtensorMap tmTA, const __grid_constant__ CUtensorMap tmTB)
{
    using namespace pf;
    using Cfg = PairCfg<N>;
    constexpr int kStages = Cfg::kStages, kPkSlots = Cfg::kPkSlots, kPkStages = Cfg::kPkStages, kSK = Cfg::kSK, kDK = Cfg::kDK;
    constexpr int kStageBytes = Cfg::kStageBytes, kECol = Cfg::kECol;
    const int half_tok = p.half;
    extern __shared__ unsigned char smem_raw[];
    // layout: stages | packed slots {value bytes | index bytes} | barriers
    unsigned char* stages = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char* packed = stages + (size_t)kStages * kStageBytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(packed + kPkSlots * kPkSlotBytes);     // [kStages] even CTA: both CTAs' tiles landed, both CTAs' converters are done
    uint64_t* empty = full + kStages;                // [kStages] the MMAs that read the stage are complete
    uint64_t* pk_full = empty + kStages;             // [kPkSlots]
    uint64_t* pk_empty = pk_full + kPkSlots;         // [kPkSlots]
    uint64_t* acc_full = pk_empty + kPkSlots;        // a tile's MMAs are complete
    uint64_t* acc_empty = acc_full + 1;              // even CTA: both CTAs have read the accumulator
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 1);
    volatile uint32_t* abort_flag = tmem_slot + 1;

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;      // (a shuffle: the same in all lanes, for the compiler too)
    const uint32_t rank = cluster_rank();
    const int pairs = gridDim.x >> 1, first_tile = blockIdx.x >> 1;
    const int n_total = p.n1 + p.n2, n_groups = ceil_div(p.n1, kPkStages);
    // this pair's share of T': the last pairs, which have the fewest tiles, come first
    const int t_units = p.t_tiles * p.t_stages, tq = pairs - 1 - first_tile;
    const int t_begin = tq < p.t_pairs ? share_begin(tq, t_units, p.t_pairs) : 0, t_end = tq < p.t_pairs ? share_begin(tq + 1, t_units, p.t_pairs) : 0;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) { mbar_init(&full[i], 8); mbar_init(&empty[i], 1); }
        for (int i = 0; i < kPkSlots; ++i) { mbar_init(&pk_full[i], p.meta ? 33 : 1); mbar_init(&pk_empty[i], 4 * kPkStages); }
        mbar_init(acc_full, 1);
        mbar_init(acc_empty, 16);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == Cfg::kWarpPk && elect_one()) { prefetch_map(&tmV); if (!p.meta) prefetch_map(&tmM); if (p.r > 0) prefetch_map(&tmA2); }
    if (warp == Cfg::kWarpX && elect_one()) { prefetch_map(&tmX); if (p.r > 0) { prefetch_map(&tmTA); prefetch_map(&tmTB); prefetch_map(&tmB2); } }
    cluster_sync_all();                              // both CTAs' barriers exist before anything crosses
    if (warp == Cfg::kWarpMma) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(s32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t*>(tmem_slot), 0);
    // Launched while the grid before it in the stream still runs (programmatic dependent launch): everything above needs no
    // global memory, everything below comes after that grid.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("fence.proxy.async;" ::: "memory");            // what that grid wrote is read through TMA
    const uint32_t call = p.r > 0 ? call_number(*(volatile unsigned long long*)p.departures) : 0u;
    bool ok = true;
    // The pairs that share a T' tile.  Which 256 rows of its A operand it is made of, and which t_n rows of its B operand.
    auto first_owner = [&](int tile) { return p.t_even > 0 ? tile * p.t_even : share_owner(tile * p.t_stages, t_units, p.t_pairs); };
    auto last_owner = [&](int tile) { return p.t_even > 0 ? (tile + 1) * p.t_even - 1 : share_owner((tile + 1) * p.t_stages - 1, t_units, p.t_pairs); };
    auto t_part_of = [&](int tile, bool a) { return a != RANKS ? tile / p.t_chunks : tile % p.t_chunks; };
    // Tile -> its first row in this CTA, its first token, and where its walk over the weight columns starts: pairs that share
    // token rows start at different places, so that at any moment they ask the L2 for different lines of X.
    struct Tile { int m0, n0, rot; };
    auto tile_of = [&](int t) {
        const int rp = t % p.row_pairs, tt = t / p.row_pairs;
        Tile ti;
        ti.m0 = (2 * rp + (int)rank) * kPM; ti.n0 = tt * 2 * half_tok;
        ti.rot = p.d_in % kPkCols == 0 && n_groups > 0 ? (rp + 3 * tt) % n_groups : 0;       // whole packed tiles
        return ti;
    };

    if (warp == Cfg::kWarpX || warp == Cfg::kWarpX + 1) {
        // ============================ token tiles, A2, B2 ============================
        // Two warps: they take the sparse stages in turn, and in the stages of T' and of the adapters one requests A and the other B.  (So the
        // tiles of L are on their way while T' is waited for.)
        const int odd = warp - Cfg::kWarpX;
        int g = 0;                                          // stages so far
        int t_checked = -1;                                 // the token tile whose T' was found complete
        auto slot_of = [&](int stage) {                     // waits for the stage's place in the ring
            const int st = stage % kStages;
            if (stage >= kStages) ok = mbar_wait(&empty[st], ((stage / kStages) & 1) ^ 1, abort_flag) && ok;
            return st;
        };
        for (int u = t_begin; u < t_end;) {
            // T': 128 rows x 64 columns of X (or R) as A, half of the chunk's rows of R (the tile's tokens of X) as B
            const Run run = run_at(u, t_end, p.t_stages);
            const int a_row = t_part_of(run.tile, true) * kTTok + (int)rank * kPM, b_row = t_part_of(run.tile, false) * p.t_n + (int)rank * (p.t_n / 2);
            for (int it = 0; it < run.len; ++it) {
                const int st = slot_of(g + it);
                unsigned char* sbase = stages + (size_t)st * kStageBytes;
                if (elect_one()) {
                    if (odd) tma_tile_pair(sbase, &tmTB, (run.k0 + it) * kDK, b_row, peer_addr(&full[st], 0));
                    else     tma_tile_pair(sbase + Cfg::kATileAt, &tmTA, (run.k0 + it) * kDK, a_row, peer_addr(&full[st], 0));
                }
            }
            u += run.len; g += run.len;
        }
        for (int t = first_tile; t < p.tiles; t += pairs) {
            const Tile ti = tile_of(t);
            // a sparse stage's token tile: sub-tiles of 64 columns in one box
            for (int it = (g ^ odd) & 1; it < p.n1; it += 2) {
                const int st = slot_of(g + it);
                int kb = it + ti.rot * kPkStages;
                if (kb >= p.n1) kb -= p.n1;
                if (elect_one()) tma_tile_pair3(stages + (size_t)st * kStageBytes, &tmX, ti.n0 + (int)rank * half_tok, kb * (kSK / kPBK), peer_addr(&full[st], 0));
            }
            for (int it = p.n1; it < n_total; ++it) {
                if (odd) {
                    // the T' of this CTA's half of the tokens is complete (a word per part of its tiles, 32 at a time)
                    if (ti.n0 != t_checked) {
                        // T' tiles of 256 tokens: one or two halves of them; T' tiles of this tile's tokens: both halves of the ranks
                        const int tok = ti.n0 + (int)rank * half_tok;
                        const int blk0 = RANKS ? ti.n0 / half_tok : tok / kPM, blk1 = RANKS ? blk0 + 2 : ceil_div(min(tok + half_tok, p.b), kPM);
                        const int per = p.t_chunks * p.t_even;
                        if (per > 0) {                                       // equal parts: the words of a block's chunks follow each other
                            for (int first = 0; first < (blk1 - blk0) * per; first += 32) {
                                const bool in = first + lane < (blk1 - blk0) * per, next = first + lane >= per;
                                const int blk = blk0 + (next ? 1 : 0), i = first + lane - (next ? per : 0), tile0 = (blk / 2) * p.t_chunks;
                                const size_t word = p.t_even == 1 ? tile_word(p.t_pairs, tile0 + i, (uint32_t)blk & 1)
                                                                  : part_word(tile0 * p.t_even + i, i % p.t_even == 0, (uint32_t)blk & 1) + 1;
                                ok = wait_words(in ? p.t_sync + word : nullptr, call, abort_flag) && ok;
                            }
                        } else
                        for (int blk = blk0; blk < blk1; ++blk) {
                            const int tile0 = (blk / 2) * p.t_chunks;
                            const uint32_t t_half = (uint32_t)blk & 1;
                            for (int first = 0, left = 1; left > 0; first += 32) {
                                int i = first + lane;
                                const unsigned long long* w = nullptr;
                                left = -first - 32;
                                for (int c = 0; c < p.t_chunks; ++c) {
                                    const int q0 = first_owner(tile0 + c), q1 = last_owner(tile0 + c);
                                    if (i >= 0 && i <= q1 - q0) w = p.t_sync + (q0 == q1 ? tile_word(p.t_pairs, tile0 + c, t_half) : part_word(q0 + i, i == 0, t_half) + 1);
                                    i -= q1 - q0 + 1; left += q1 - q0 + 1;
                                }
                                ok = wait_words(w, call, abort_flag) && ok;
                            }
                        }
                        t_checked = ti.n0;
                        __syncwarp();
                        asm volatile("fence.proxy.async;" ::: "memory");   // the tiles are read by the async proxy
                    }
                }
                const int st = slot_of(g + it);
                unsigned char* sbase = stages + (size_t)st * kStageBytes;
                int kb = it - p.n1, y = ti.n0 + (int)rank * half_tok;
                if (p.t_parts == 2) { y += (kb & 1) * p.b; kb >>= 1; }       // a column block of either part in turn
                if (elect_one()) {
                    if (odd) tma_tile_pair(sbase, &tmB2, kb * kDK, y, peer_addr(&full[st], 0));
                    else     tma_tile_pair(sbase + Cfg::kATileAt, &tmA2, kb * kDK, ti.m0, peer_addr(&full[st], 0));
                }
            }
            g += n_total;
        }
    } else if (warp == Cfg::kWarpPk) {
        // ============================ packed tiles ============================
        // The ring holds 48 KB, less than what is under way from the HBM to an SM at full rate: a pair's first tile asks its packed tiles into
        // the L2 kAhead before their turn (not where the index bytes keep this warp busy).
        constexpr int kAhead = 6;
        int g = 0;
        for (int t = first_tile; t < p.tiles; t += pairs) {
            const Tile ti = tile_of(t);
            for (int i = 0; i < n_groups; ++i, ++g) {
                const int slot = g % kPkSlots;
                const int kg = i + ti.rot < n_groups ? i + ti.rot : i + ti.rot - n_groups;
                if (g >= kPkSlots) ok = mbar_wait(&pk_empty[slot], ((g / kPkSlots) & 1) ^ 1, abort_flag) && ok;
                load_packed(p, &tmV, &tmM, packed + slot * kPkSlotBytes, &pk_full[slot], kg, ti.m0, lane);
                if (!p.meta && t == first_tile && i + kAhead < n_groups && elect_one()) {
                    const int ka = i + kAhead + ti.rot < n_groups ? i + kAhead + ti.rot : i + kAhead + ti.rot - n_groups;
                    prefetch_tile(&tmV, ka * 64, ti.m0);
                    prefetch_tile(&tmM, ka * 32, ti.m0);
                }
            }
        }
    } else if (warp == Cfg::kWarpMma) {
        // ============================ MMA issue: a warp of the even CTA ============================
        // The whole warp walks the stages together and one elected lane issues a stage's MMAs: what they are given is then known to be
        // the same in all lanes.  (One lane walking alone took 120 cycles for each MMA, 700 and more a stage, whatever N.)  The next
        // stage is asked about before this one's MMAs are issued: the answer of the barrier takes 200 cycles.
        if (rank == 0) {
            const uint32_t idesc = idesc_bf16(2 * kPM, 16) + ((uint32_t)((half_tok - 8) >> 2) << 17);
            int st = 0, nth = 0;
            uint32_t parity = 0, pre = 0;
            auto ready = [&] {
                if (!__all_sync(0xffffffffu, pre)) ok = mbar_wait_all(&full[st], parity, true, nullptr, 0, false, nullptr, 0, false, abort_flag) && ok;
                fence_after_sync();
                const bool wraps = st + 1 == kStages;
                pre = mbar_test(&full[wraps ? 0 : st + 1], wraps ? parity ^ 1 : parity, true);
            };
            auto next = [&] { if (++st == kStages) { st = 0; parity ^= 1; } };
            const uint32_t lo_first = desc_lo(s32(stages)), lo_sub = (uint32_t)half_tok * (128 >> 4);
            constexpr uint32_t kLoStage = kStageBytes >> 4, kLoA = Cfg::kATileAt >> 4;
            auto dense_stage = [&](uint32_t idesc_d, bool adds) {
                const uint32_t lo = lo_first + (uint32_t)st * kLoStage;
                if (elect_one()) {
#pragma unroll
                    for (int j = 0; j < kDK / 16; ++j) mma_dense2(tmem_base, lo + kLoA + 2 * j, lo + 2 * j, idesc_d, j > 0 || adds ? 1u : 0u);
                    mma_commit2(&empty[st]);            // the stage is free, in both CTAs, once these MMAs have read it
                }
            };
            for (int u = t_begin; u < t_end; ++nth) {
                const uint32_t idesc_t = idesc_bf16(2 * kPM, 16) + ((uint32_t)((p.t_n - 16) >> 3) << 17);
                const Run run = run_at(u, t_end, p.t_stages);
                if (nth > 0) ok = mbar_wait_all(acc_empty, (nth & 1) ^ 1, true, nullptr, 0, false, nullptr, 0, false, abort_flag) && ok;
                for (int it = 0; it < run.len; ++it) { ready(); dense_stage(idesc_t, it > 0); next(); }
                if (elect_one()) mma_commit2(acc_full);
                u += run.len;
            }
            for (int t = first_tile; t < p.tiles; t += pairs, ++nth) {
                if (nth > 0) ok = mbar_wait_all(acc_empty, (nth & 1) ^ 1, true, nullptr, 0, false, nullptr, 0, false, abort_flag) && ok;
                for (int it = 0; it < p.n1; ++it) {
                    ready();
                    const uint32_t lo = lo_first + (uint32_t)st * kLoStage, a = tmem_base + Cfg::kACol + Cfg::kACols * st, e = tmem_base + kECol + Cfg::kECols * st;
                    if (elect_one()) {
                        // per MMA: A 16 stored bf16 (8 columns of tensor memory), B 32 columns (64 bytes)
#pragma unroll
                        for (int j = 0; j < kSK / 32; ++j)
                            mma_sparse2(tmem_base, a + 8 * j, lo + (j >> 1) * lo_sub + 4 * (j & 1), e + 2 * (j >> 1), idesc | (1u << 2) | (uint32_t)(j & 1), j > 0 || it > 0 ? 1u : 0u);
                        mma_commit2(&empty[st]);
                    }
                    next();
                }
                for (int it = p.n1; it < n_total; ++it) { ready(); dense_stage(idesc, it > 0); next(); }
                if (elect_one()) mma_commit2(acc_full);
            }
        }
    } else if (warp < Cfg::kWarpEpi) {
        // ============================ converters ============================
        // Within a group of four warps a thread owns one weight row of the tile.
        const int row = threadIdx.x & 127;           // weight row inside the tile = TMEM lane
        constexpr int kGroups = Cfg::kGroups;
        const int group = threadIdx.x >> 7;
        const int x = (row >> 3) & 1;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        // A stage is full when both CTAs' converters have arrived and the bytes have landed that one of the warps announces with its
        // arrival (bytes that land before are counted below zero; the phase cannot end without the arrivals).
        auto arrive = [&](int st, uint32_t bytes) {
            __syncwarp();
            if (lane == 0) {
                if (rank != 0) mbar_arrive_remote(peer_addr(&full[st], 0));
                else if ((warp & 3) == 0) mbar_expect_tx(&full[st], bytes);
                else mbar_arrive(&full[st]);
            }
        };
        // nothing to expand for T' and in phase 2
        auto pass = [&](int g, uint32_t bytes) {
            const int st = g % kStages;
            if (g >= kStages) ok = mbar_wait(&empty[st], ((g / kStages) & 1) ^ 1, abort_flag) && ok;
            arrive(st, bytes);
        };
        // Whether a phase has ended, as lane 0 finds it; the answer is looked at later.  (The shuffle hands the answer over, the barrier behind
        // it what lane 0 has acquired with it.)
        auto ask = [&](uint64_t* bar, uint32_t phase) { return lane == 0 ? mbar_test(bar, phase, false) : 0u; };
        auto yes = [&](uint32_t answer) {
            const bool there = __shfl_sync(0xffffffffu, answer, 0) != 0;
            __syncwarp();
            return there;
        };
        // The groups take the stages in turn (turns.h: why the waits by parity are right).
        int base = t_end - t_begin, nth = 0;         // stages before this tile
        for (int g = first_turn(group, 0); g < base; g += kGroups) pass(g, (uint32_t)(2 * (kPM + p.t_n / 2) * kDK * 2));
        for (int t = first_tile; t < p.tiles; t += pairs, base += n_total, ++nth) {
            const bool row_in = tile_of(t).m0 + row < p.m_total;
            uint32_t pk_there = 0;
            const int seen = seen_from(nth, p.n1, p.n2, kPkStages);
            int it = first_turn(group, base);
            for (; it < p.n1; it += kGroups) {
                const int g = base + it, st = g % kStages;
                // expand into registers as soon as the packed tile is there (and give its slot back), store when the MMAs of
                // the stage's previous use are done: only the stores are between that and the next MMAs.  Both barriers are asked ahead.
                const int gi = nth * n_groups + it / kPkStages, q = it % kPkStages, slot = gi % kPkSlots;
                if (it < seen && g >= kStages) ok = mbar_wait(&empty[st], ((g / kStages) & 1) ^ 1, abort_flag) && ok;
                if (!yes(pk_there)) ok = mbar_wait(&pk_full[slot], (gi / kPkSlots) & 1, abort_flag) && ok;
                const uint32_t free = it >= seen && g >= kStages ? ask(&empty[st], ((g / kStages) & 1) ^ 1) : 1u;
#pragma unroll
                for (int hh = 0; hh < kSK / 128; ++hh) {
                    uint4 a[8];
                    uint32_t e[4];
                    expand_row<128>(packed + slot * kPkSlotBytes, row, kPkStages == 1 ? hh : q, x, row_in, p.d_in - it * kSK - hh * 128, a, e);
#pragma unroll
                    for (int i = 0; i < 8; ++i) asm volatile("" : "+r"(a[i].x), "+r"(a[i].y), "+r"(a[i].z), "+r"(a[i].w));     // here, not after the wait
                    if (hh + 1 == kSK / 128) {
                        __syncwarp();
                        // (half a packed tile at the end: for the other half too)
                        if (lane <= (q + 1 < kPkStages && it + 1 == p.n1 ? 1 : 0)) mbar_arrive(&pk_empty[slot]);
                        // the packed tile of this group's next stage in this tile
                        constexpr int kNext = kGroups / kPkStages;
                        pk_there = it + kGroups < p.n1 && it + kGroups >= seen ? ask(&pk_full[(gi + kNext) % kPkSlots], ((gi + kNext) / kPkSlots) & 1) : 0u;
                    }
                    if (hh == 0) {
                        if (!yes(free)) ok = mbar_wait(&empty[st], ((g / kStages) & 1) ^ 1, abort_flag) && ok;
                        fence_after_sync();                                  // the MMAs have read what is stored over
                    }
                    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};"
                                 :: "r"(tmem_base + lane_base + kECol + Cfg::kECols * st + 4 * hh), "r"(e[0]), "r"(e[1]), "r"(e[2]), "r"(e[3]) : "memory");
                    tmem_st32(tmem_base + lane_base + Cfg::kACol + Cfg::kACols * st + 32 * hh, a);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                fence_before_sync();
                arrive(st, (uint32_t)(2 * half_tok * kSK * 2));
            }
            for (; it < n_total; it += kGroups) pass(base + it, (uint32_t)(2 * (half_tok + kPM) * kDK * 2));
        }
    } else {
        // ============================ epilogue: thread = output row, half of the tokens ============================
        const int half = (warp - Cfg::kWarpEpi) >> 2;
        const int row = (warp & 3) * 32 + lane;
        const uint32_t taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + half * half_tok;
        const uint32_t buf = s32(full) + 384 + (warp - Cfg::kWarpEpi) * 1024;
        int nth = 0;
        // ---- T': thread = token (t_ranks: rank).  Part of pair q: [c / 4][128 tokens] float4; a pair has at most one that starts with its tile and
        // one that does not.
        auto part = [&](int q, bool starts) { return p.t_part + ((size_t)(2 * q + (starts ? 1 : 0)) * 2 + rank) * ((size_t)kPM * p.t_n / 4) + row; };
        const size_t t_tail = p.t_parts == 2 ? (size_t)p.b * p.r : 0;
        int a_row = 0, b_row = 0;                                            // of the run's tile
        auto rows_of = [&](int tile) { a_row = t_part_of(tile, true) * kTTok + (int)rank * kPM + row; b_row = t_part_of(tile, false) * p.t_n; };
        auto store4 = [&](int c, float4 v) {
            put_T<RANKS>(p.t_out, a_row, b_row + c, p.b, p.r, t_tail, make_float4(p.t_scale * v.x, p.t_scale * v.y, p.t_scale * v.z, p.t_scale * v.w));
        };
        auto publish = [&](size_t word) {                                    // the writes of the eight warps, then the word
            epilogue_sync();
            if (threadIdx.x == Cfg::kWarpEpi * 32) {
                __threadfence();
                *(volatile unsigned long long*)(p.t_sync + word) = tagged(call, 0);
            }
        };
        // all of this pair's runs first (nothing here waits for another pair), every second group of 16 columns a thread
        for (int u = t_begin; u < t_end; ++nth) {
            const Run run = run_at(u, t_end, p.t_stages);
            u += run.len;
            const bool whole = run.len == p.t_stages;
            rows_of(run.tile);
            ok = mbar_wait(acc_full, nth & 1, abort_flag) && ok;
            fence_after_sync();
            float4* mine = part(tq, run.k0 == 0);
            const uint32_t t_addr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
            for (int c = half * 16; c < p.t_n; c += 32) {
                float4 v[4];
                tmem_ld16(t_addr + c, v);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (whole) store4(c + 4 * i, v[i]);
                    else __stcg(mine + (size_t)(c / 4 + i) * kPM, v[i]);
                }
            }
            fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_remote_release(peer_addr(acc_empty, 0));
            publish(whole ? tile_word(p.t_pairs, run.tile, rank) : part_word(tq, run.k0 == 0, rank));
        }
        // then its share of the sums: when every part of a tile is there, columns c4 = .. (mod 2 n) for each of its n pairs
        for (int u = t_begin; u < t_end;) {
            const Run run = run_at(u, t_end, p.t_stages);
            u += run.len;
            if (run.len == p.t_stages) continue;
            const int q0 = first_owner(run.tile), q1 = last_owner(run.tile);
            const int n = q1 - q0 + 1;
            rows_of(run.tile);
            for (int q = q0; q <= q1; q += 32)
                ok = wait_words(q + lane <= q1 ? p.t_sync + part_word(q + lane, q + lane == q0, rank) : nullptr, call, abort_flag) && ok;
            if (n == 2) {                                                    // two parts: four columns' loads in flight
                const float4 *f0 = part(q0, true), *f1 = part(q1, false);
                for (int c4 = 2 * (tq - q0) + half; c4 < p.t_n / 4; c4 += 16) {
                    float4 x[4], y[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const size_t at = (size_t)min(c4 + 4 * i, p.t_n / 4 - 1) * kPM;
                        x[i] = __ldcg(f0 + at); y[i] = __ldcg(f1 + at);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (c4 + 4 * i < p.t_n / 4) store4(4 * (c4 + 4 * i), make_float4(x[i].x + y[i].x, x[i].y + y[i].y, x[i].z + y[i].z, x[i].w + y[i].w));
                }
            } else if (n <= 4) {                                             // four parts of two columns
                for (int c4 = 2 * (tq - q0) + half; c4 < p.t_n / 4; c4 += 4 * n) {
                    const int c5 = c4 + 2 * n;
                    float4 x[4], y[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4* from = part(min(q0 + i, q1), i == 0);
                        x[i] = __ldcg(from + (size_t)c4 * kPM); y[i] = __ldcg(from + (size_t)min(c5, p.t_n / 4 - 1) * kPM);
                    }
#pragma unroll
                    for (int i = 1; i < 4; ++i)
                        if (i < n) {
                            x[0].x += x[i].x; x[0].y += x[i].y; x[0].z += x[i].z; x[0].w += x[i].w;
                            y[0].x += y[i].x; y[0].y += y[i].y; y[0].z += y[i].z; y[0].w += y[i].w;
                        }
                    store4(4 * c4, x[0]);
                    if (c5 < p.t_n / 4) store4(4 * c5, y[0]);
                }
            } else {
                constexpr int kParts = 9;
                for (int c4 = 2 * (tq - q0) + half; c4 < p.t_n / 4; c4 += 2 * n) {
                    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
                    for (int qb = q0; qb <= q1; qb += kParts) {
                        float4 v[kParts];
#pragma unroll
                        for (int i = 0; i < kParts; ++i) v[i] = qb + i <= q1 ? __ldcg(part(qb + i, qb + i == q0) + (size_t)c4 * kPM) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int i = 0; i < kParts; ++i) { s.x += v[i].x; s.y += v[i].y; s.z += v[i].z; s.w += v[i].w; }
                    }
                    store4(4 * c4, s);
                }
            }
            publish(part_word(tq, run.k0 == 0, rank) + 1);
        }
        for (int t = first_tile; t < p.tiles; t += pairs, ++nth) {
            const Tile ti = tile_of(t);
            ok = mbar_wait(acc_full, nth & 1, abort_flag) && ok;
            fence_after_sync();
            // 16 tokens at a time, through the warp's kilobyte of shared memory, [token][32 rows] bf16: a thread then stores 16 bytes,
            // eight rows of a token (direct two-byte stores took 5.6 us a tile).  Two passes of 64 tokens (what fits in
            // registers): the accumulator is free before the second pass's stores.
            const int tok0 = ti.n0 + half * half_tok, row8 = ti.m0 + (warp & 3) * 32 + (lane & 3) * 8;
            const int toks = min(half_tok, p.b - tok0), n_tok = row8 < p.m_total ? toks : 0;
            __nv_bfloat16* out = p.out + (size_t)(tok0 + (lane >> 2)) * p.ldo + row8;
            constexpr int kPass = N < 128 ? N / 2 : 64;
            bool held = true;                                                // the accumulator, by this warp
#pragma unroll
            for (int c0 = 0; c0 < N / 2; c0 += kPass) {
                uint32_t y[kPass / 2];                                       // bf16 pairs of neighbouring tokens
                if (c0 < half_tok) {
#pragma unroll
                    for (int c1 = 0; c1 < kPass; c1 += 32) {
                        uint32_t r[32];
                        tmem_ld32(taddr + c0 + c1, r);
#pragma unroll
                        for (int c = 0; c < 32; c += 2) {
                            __nv_bfloat162 v = __floats2bfloat162_rn(p.scale * __uint_as_float(r[c]), p.scale * __uint_as_float(r[c + 1]));
                            y[(c1 + c) / 2] = *reinterpret_cast<uint32_t*>(&v);
                        }
                    }
                }
                if (held && c0 + kPass >= half_tok) {
                    held = false;
                    fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_remote_release(peer_addr(acc_empty, 0));
                }
#pragma unroll
                for (int c1 = 0; c1 < kPass; c1 += 16) {
                    if (c0 + c1 >= toks) break;
#pragma unroll
                    for (int c = 0; c < 16; ++c)
                        asm volatile("st.shared.u16 [%0], %1;" :: "r"(buf + c * 64 + lane * 2), "h"((unsigned short)(c & 1 ? y[(c1 + c) / 2] >> 16 : y[(c1 + c) / 2] & 0xFFFFu)) : "memory");
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 2; ++i) {                            // tokens 8 i + lane / 4
                        uint4 v;
                        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(buf + i * 512 + lane * 16) : "memory");
                        if (c0 + c1 + i * 8 + (lane >> 2) < n_tok) *reinterpret_cast<uint4*>(out + (size_t)(c0 + c1 + i * 8) * p.ldo) = v;
                    }
                    __syncwarp();
                }
            }
        }
    }

    if (!ok && lane == 0) flag_error(p.status, SLIM_ERR_TIMEOUT);
    fence_before_sync();
    __syncthreads();
    cluster_sync_all();                              // neither CTA leaves while the other may still use its shared memory
    if (warp == Cfg::kWarpMma) {
        fence_after_sync();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" :: "r"(tmem_base), "r"(512) : "memory");
    }
    if (threadIdx.x == 0) atomicAdd(p.departures, departure(blockIdx.x, gridDim.x));
}

// Sum of the K slices' partial tiles, scaled and rounded to bf16 (fixed order: deterministic).
__global__ void pre_reduce_kernel(const float* part, int slices, size_t n, float scale, int t_parts, __nv_bfloat16* out)
{
    // lets the main launch start, then waits for the dense-only launch whose partial tiles it adds
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (size_t i = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * 4; i < n; i += (size_t)gridDim.x * blockDim.x * 4) {
        float4 acc = *reinterpret_cast<const float4*>(part + i);
        for (int z = 1; z < slices; ++z) {
            const float4 v = *reinterpret_cast<const float4*>(part + (size_t)z * n + i);
            acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
        }
        store_T(out + i, t_parts == 2 ? n : 0, make_float4(scale * acc.x, scale * acc.y, scale * acc.z, scale * acc.w));
    }
}

// ------------------------------------------------------------------ host side
// Shape of the dense-only launch T' = X R^T: token tile, K slices, stages per slice.  The product
// has few tiles (r / 128 x tokens / tile), so K is split until they about fill the machine.
struct PrePlan { int n_tok; int slices; int k_per; };
// `overlapped`: the main launch has sparse stages to run meanwhile.  A short product with few tiles is then
// better left whole on few SMs -- no partial tiles, no reduction, and the other SMs go to the main launch at
// once -- than split over the machine (measured: 4096 columns and 32 tiles gain 2-6 %; longer or wider
// products lose, their T' arrives after the main launch's first CTAs want it).
static PrePlan pre_plan(int b, int d_in, int r, int sm_count, bool overlapped = false) {
    PrePlan pl;
    pl.n_tok = b >= 192 ? 256 : 64;
    const int tiles = ceil_div(r, kPM) * ceil_div(b, pl.n_tok);
    const int n2 = d_in / kPBK;
    int ks = overlapped && n2 <= 64 && tiles <= sm_count / 4 ? 1 : sm_count / (tiles > 0 ? tiles : 1);
    ks = ks < 1 ? 1 : (ks > 8 ? 8 : ks);
    if (ks > n2) ks = n2 > 0 ? n2 : 1;
    pl.k_per = ceil_div(n2, ks);
    pl.slices = ceil_div(n2, pl.k_per);          // every slice has at least one stage
    return pl;
}
static int pre_sm_count() {
    slim_status_t err = SLIM_OK;
    const DeviceInfo* di = device_info(&err);
    return di && di->sm_count > 0 ? di->sm_count : 148;
}

typedef CUresult (*PfEncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                    const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Row-major 2-D tensor [rows][row_elems]; box of box_rows x box_elems elements.
static bool pf_map(CUtensorMap* map, const void* base, CUtensorMapDataType type, int esize, uint64_t row_elems,
                   uint64_t rows, int box_elems, int box_rows, int swizzle_bytes) {
    PfEncodeTiledFn fn = reinterpret_cast<PfEncodeTiledFn>(tensor_map_encoder());
    if (!fn) return false;
    cuuint64_t dims[2] = {row_elems, rows};
    cuuint64_t strides[1] = {row_elems * (uint64_t)esize};
    cuuint32_t box[2] = {(cuuint32_t)box_elems, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, type, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              swizzle_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : swizzle_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : swizzle_bytes == 32 ? CU_TENSOR_MAP_SWIZZLE_32B : CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// bf16 rows as 64-column sub-tiles: one box of box_rows rows x sub_tiles of 128 bytes, in that order.
static bool pf_map3(CUtensorMap* map, const void* base, uint64_t cols, uint64_t rows, int box_rows, int sub_tiles) {
    PfEncodeTiledFn fn = reinterpret_cast<PfEncodeTiledFn>(tensor_map_encoder());
    if (!fn) return false;
    cuuint64_t dims[3] = {64, rows, cols / 64};
    cuuint64_t strides[2] = {cols * 2, 128};
    cuuint32_t box[3] = {64, (cuuint32_t)box_rows, (cuuint32_t)sub_tiles};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool prefill_supports(int b, int d_out, int d_in, int r) {
    // (when the rows of the index-byte array, d_in / 8 bytes, are no 16-byte multiples they come by cp.async)
    return b >= 1 && d_out % 16 == 0 && d_in % kPBK == 0 && r % 16 == 0 && r >= 0;
}

static size_t pair_part_bytes(int r, int sm_count) { return (size_t)(sm_count / 2) * 2 * kPairTTok * t_width(r, ceil_div(r, 256)) * sizeof(float); }

// The pair kernel, asked for by the kernel family's name: when its 128 x 256 tiles would give a quarter of the SMs or more a tile.
// The dispatcher (`automatic`) takes it unless the 128 x 64 tiles of the one-CTA kernel have an SM each and rows are short: the pairs'
// stage of 128 columns costs less, but they make T' in a cooperative launch that takes 10 us however short it is.  The two meet
//   without adapters at 768 columns (512 -> 4096, 200 tokens: one CTA 8 % faster; 1024 -> 4096: the same; 1536 columns: 8 % slower);
//   on shapes that come out even at 2048 columns up to 191 tokens (768 -> 8192, 100 tokens, rank 208 11.0 us against 22.8; 2048 -> 8192 15.4
//   against 20.7), at 1024 where tiles are up to two an SM and the rank above 128 (1024 -> 8192, 160 tokens, rank 208 20.0 against 22.2,
//   rank 64 18.3 against 15.6), at 1024 above (1536 -> 2048, 300 tokens, rank 16 18.0 against 13.4; 1024 -> 256, rank 208 16.2 against 20.5);
//   on others, whose T' has two parts, at 2048 up to 191 tokens and few tiles; above the pairs are always faster (2048 -> 48, 200 tokens,
//   rank 16 13.6 us against 32).
static bool runs_wide(int b, int d_out, int d_in, int r, int sm_count, bool automatic) {
    const bool many = (long long)ceil_div(d_out, kPM) * ceil_div(b, 256) * 4 >= (long long)sm_count;
    if (!automatic) return many;
    const long long tiles = (long long)ceil_div(d_out, kPM) * ceil_div(b, 64);
    const bool even = d_out % kPM == 0 && d_in % 128 == 0;
    if (tiles > sm_count) return !(even && r > 128 && b < 192 && d_in <= 1024 && tiles <= 2 * sm_count);
    if (r == 0) return d_in > 768;
    if (!even) return many || b >= 192 || d_in >= 2048;
    return d_in > (b < 192 ? 2048 : 1024);
}

// T' in the workspace; the partial sums follow it.
static size_t t_bytes(int b, int r, int parts) { return ((size_t)b * (size_t)r * parts * sizeof(__nv_bfloat16) + 255) / 256 * 256; }

size_t prefill_workspace_bytes(int b, int d_out, int d_in, int r) {
    if (!prefill_supports(b, d_out, d_in, r)) return 0;
    const size_t tq = t_bytes(b, r, keeps_T32(b, d_out, d_in, r) ? 2 : 1);
    if (r == 0) return tq;
    const PrePlan pl = pre_plan(b, d_in, r, pre_sm_count());
    const size_t narrow = pl.slices > 1 ? (size_t)pl.slices * b * r * sizeof(float) : 0, wide = pair_part_bytes(r, pre_sm_count());
    return tq + (wide > narrow ? wide : narrow);           // (either kernel may be asked for by name)
}

static std::atomic<int> g_pairs[64];               // pairs resident at once
static std::atomic<bool> g_prefill_attr_set[64];   // attributes set once per device (setting them twice is harmless)

// `after_dense_only`: may start while the launch before it (the dense-only launch or its reduction) still runs.
template <int N, bool PRE>
static slim_status_t launch_tile_kernel(const PrefillParams& q, int m_rows, const CUtensorMap& tmV, const CUtensorMap& tmM, const CUtensorMap& tmX,
                                        const CUtensorMap& tmA2, const CUtensorMap& tmB2, cudaStream_t st, int slices = 1, bool after_dense_only = false) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ceil_div(m_rows, kPM), ceil_div(q.b, N), slices); cfg.blockDim = dim3(kPThreads);
    cfg.dynamicSmemBytes = PfCfg<N, PRE>::kSmem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = after_dense_only ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, prefill_kernel<N, PRE>, q, tmV, tmM, tmX, tmA2, tmB2);
    count_launch(1);
    return e == cudaSuccess ? SLIM_OK : SLIM_ERR_CUDA;
}

template <int N, bool RANKS>
static slim_status_t launch_pair(const PrefillParams& p, const CUtensorMap& tmV, const CUtensorMap& tmM, const CUtensorMap& tmX, const CUtensorMap& tmA2,
                                 const CUtensorMap& tmB2, const CUtensorMap& tmTA, const CUtensorMap& tmTB, int pairs, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * pairs); cfg.blockDim = dim3(kPairThreads); cfg.dynamicSmemBytes = PairCfg<N>::kSmem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    if (p.t_pairs > 0) {
        // the pairs wait for one another's T': all of them are resident together (two such calls on different streams could
        // otherwise each hold half of the SMs and wait for their other half)
        attr[1].id = cudaLaunchAttributeCooperative;
        attr[1].val.cooperative = 1;
    } else {
        // set up while the grid before it ends (8192 x 8192, 333 tokens, weight in the L2 32.9 -> 31.8 us; no gain beside a cooperative launch)
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
    }
    cfg.attrs = attr; cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, prefill_pair_kernel<N, RANKS>, p, tmV, tmM, tmX, tmA2, tmB2, tmTA, tmTB);
    count_launch(1);
    return e == cudaSuccess ? SLIM_OK : SLIM_ERR_CUDA;
}

slim_status_t launch_prefill(const __nv_bfloat16* X, int b, const uint8_t* vals, const uint8_t* meta,
                             float s, const __nv_bfloat16* L, const __nv_bfloat16* R, int r,
                             int d_out, int d_in, __nv_bfloat16* Y, void* ws, uint32_t* status_dev,
                             cudaStream_t st, bool force_pair, bool automatic)
{
    slim_status_t err;
    const DeviceInfo* di = device_info(&err);
    if (!di) return err;
    if (!prefill_supports(b, d_out, d_in, r)) return SLIM_ERR_UNSUPPORTED_SHAPE;
    // The words of T' tiles have a region of fixed size (8.1 million tokens of up to 256 ranks): more go in equal parts, one behind
    // the other on the stream and the workspace.
    const long long most = r > 0 ? (long long)(kSyncTiles / ceil_div(r, 256)) * kTTok : b;
    if (b > most) {
        const int n = ceil_div(ceil_div(b, (int)((b + most - 1) / most)), kTTok) * kTTok;
        slim_status_t rc = SLIM_OK;
        for (long long t = 0; t < b && rc == SLIM_OK; t += n)
            rc = launch_prefill(X + t * d_in, (int)(b - t < n ? b - t : n), vals, meta, s, L, R, r, d_out, d_in, Y + t * d_out, ws, status_dev, st, force_pair, automatic);
        return rc;
    }
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return SLIM_ERR_CUDA;
    if (!g_prefill_attr_set[dev].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(prefill_pair_kernel<256, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PairCfg<256>::kSmem) != cudaSuccess ||
            cudaFuncSetAttribute(prefill_pair_kernel<128, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PairCfg<128>::kSmem) != cudaSuccess ||
            cudaFuncSetAttribute(prefill_pair_kernel<128, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PairCfg<128>::kSmem) != cudaSuccess ||
            cudaFuncSetAttribute(prefill_pair_kernel<64, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PairCfg<64>::kSmem) != cudaSuccess ||
            cudaFuncSetAttribute(prefill_pair_kernel<64, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PairCfg<64>::kSmem) != cudaSuccess ||
            cudaFuncSetAttribute(prefill_kernel<64, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PfCfg<64, false>::kSmem) != cudaSuccess ||
            cudaFuncSetAttribute(prefill_kernel<64, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PfCfg<64, true>::kSmem) != cudaSuccess ||
            cudaFuncSetAttribute(prefill_kernel<256, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PfCfg<256, true>::kSmem) != cudaSuccess)
            return SLIM_ERR_CUDA;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2); cfg.blockDim = dim3(kPairThreads); cfg.dynamicSmemBytes = PairCfg<256>::kSmem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, prefill_pair_kernel<256, false>, &cfg) != cudaSuccess || n < 1) return SLIM_ERR_CUDA;
        g_pairs[dev].store(n < di->sm_count / 2 ? n : di->sm_count / 2, std::memory_order_relaxed);
        g_prefill_attr_set[dev].store(true, std::memory_order_release);
    }
    __nv_bfloat16* Tq = reinterpret_cast<__nv_bfloat16*>(reinterpret_cast<char*>(ws) + SLIM_WORKSPACE_SYNC_BYTES + kSmallTBytes);
    const float s_eff = s != 0.f ? s : 1.f;       // with s == 0 only the adapter term remains
    const int t_parts = keeps_T32(b, d_out, d_in, r) ? 2 : 1;
    const bool wide = force_pair || runs_wide(b, d_out, d_in, r, di->sm_count, automatic);
    if (force_pair && ceil_div(d_out, kPM) % 2 != 0) return SLIM_ERR_UNSUPPORTED_SHAPE;
    const int n_pairs = g_pairs[dev].load(std::memory_order_relaxed);
    const PairPlan plan = wide ? pair_plan(b, d_out, d_in, r, n_pairs) : PairPlan{};
    const int tile_n = wide ? plan.tile_n : 64;
    const int xbox = wide ? tile_n / 2 : 64;              // token rows one CTA loads per stage = one TMA box
    const bool narrow = tile_n <= 128;
    const int dk = wide ? PairCfg<256>::kDK : PfCfg<64>::kDK;      // columns of a dense stage of the main kernel
    CUtensorMap tmV, tmM, tmX, tmXpre, tmA2, tmB2, tmTA, tmTB;
    bool ok = pf_map(&tmV, vals, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)d_in / 4, (uint64_t)d_out, kPkCols / 4, kPM, 64) &&
              (d_in % 128 != 0 || pf_map(&tmM, meta, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)d_in / 8, (uint64_t)d_out, kPkCols / 8, kPM, 32)) &&
              (wide ? pf_map3(&tmX, X, (uint64_t)d_in, (uint64_t)b, xbox, (narrow ? PairCfg<128>::kSK : PairCfg<256>::kSK) / 64)
                    : pf_map(&tmX, X, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)d_in, (uint64_t)b, 64, xbox, 128));
    if (!ok) return SLIM_ERR_CUDA;
    if (d_in % 128 != 0) tmM = tmV;              // not used
    tmA2 = tmX; tmB2 = tmX; tmTA = tmX; tmTB = tmX;    // not used when r == 0
    if (r > 0 && wide) {
        ok = pf_map(&tmTA, plan.t_ranks ? R : X, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)d_in, (uint64_t)(plan.t_ranks ? r : b), 64, kPM, 128) &&
             pf_map(&tmTB, plan.t_ranks ? X : R, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)d_in, (uint64_t)(plan.t_ranks ? b : r), 64, plan.t_n / 2, 128);
        if (!ok) return SLIM_ERR_CUDA;
    } else if (r > 0) {
        // T' = (X R^T) / s : dense phase only, output rows = adapter index
        const PrePlan pl = pre_plan(b, d_in, r, di->sm_count, s != 0.f);
        ok = pf_map(&tmA2, R, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)d_in, (uint64_t)r, 64, kPM, 128) &&
             pf_map(&tmXpre, X, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)d_in, (uint64_t)b, 64, pl.n_tok, 128);
        if (!ok) return SLIM_ERR_CUDA;
        PrefillParams q = {};
        q.out = Tq; q.ldo = r; q.m_total = r; q.b = b; q.t_parts = t_parts; q.n1 = 0; q.n2 = d_in / kPBK; q.scale = 1.f / s_eff; q.status = status_dev;
        q.k_per = pl.k_per; q.meta = nullptr; q.meta_pitch = 0; q.d_in = d_in;
        // partial tiles of the K slices follow T' in the workspace
        q.part = pl.slices > 1 ? reinterpret_cast<float*>(reinterpret_cast<char*>(Tq) + t_bytes(b, r, t_parts)) : nullptr;
        slim_status_t rc = pl.n_tok == 256 ? launch_tile_kernel<256, true>(q, r, tmV, tmM, tmXpre, tmA2, tmXpre, st, pl.slices)
                                           : launch_tile_kernel<64, true>(q, r, tmV, tmM, tmXpre, tmA2, tmXpre, st, pl.slices);
        if (rc != SLIM_OK) return rc;
        if (q.part) {
            const size_t n = (size_t)b * r;
            // a small grid: its blocks wait beside the dense-only launch's and must leave room for the main launch's
            cudaLaunchConfig_t rc_cfg = {};
            const unsigned want = (unsigned)((n / 4 + 255) / 256), cap = (unsigned)(2 * di->sm_count);
            rc_cfg.gridDim = dim3(want < cap ? want : cap); rc_cfg.blockDim = dim3(256); rc_cfg.dynamicSmemBytes = 0; rc_cfg.stream = st;
            cudaLaunchAttribute rc_attr[1];
            rc_attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            rc_attr[0].val.programmaticStreamSerializationAllowed = 1;
            rc_cfg.attrs = rc_attr; rc_cfg.numAttrs = 1;
            const cudaError_t re = cudaLaunchKernelEx(&rc_cfg, pre_reduce_kernel, (const float*)q.part, pl.slices, n, q.scale, t_parts, Tq);
            count_launch(1);
            if (re != cudaSuccess) return SLIM_ERR_CUDA;
        }
    }
    if (r > 0) {
        // dense stages of the main kernel: 64 columns (128-byte rows) in the pair kernel, else 32 (64-byte rows)
        ok = pf_map(&tmA2, L, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)r, (uint64_t)d_out, dk, kPM, dk == 64 ? 128 : 64) &&
             pf_map(&tmB2, Tq, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)r, (uint64_t)b * t_parts, dk, xbox, dk == 64 ? 128 : 64);
        if (!ok) return SLIM_ERR_CUDA;
    }
    PrefillParams p = {};
    p.out = Y; p.ldo = d_out; p.m_total = d_out; p.b = b; p.t_parts = t_parts;
    p.n1 = s != 0.f ? ceil_div(d_in, !wide ? PfCfg<64>::kSK : narrow ? PairCfg<128>::kSK : PairCfg<256>::kSK) : 0;
    p.n2 = r > 0 ? ceil_div(r, dk) * t_parts : 0;
    p.scale = s_eff; p.status = status_dev; p.part = nullptr; p.k_per = 0;
    p.meta = d_in % 128 != 0 ? meta : nullptr; p.meta_pitch = d_in / 8; p.d_in = d_in;
    if (p.n1 + p.n2 == 0)             // s == 0 and no adapters: the result is zero
        return cudaMemsetAsync(Y, 0, (size_t)b * d_out * 2, st) == cudaSuccess ? SLIM_OK : SLIM_ERR_CUDA;
    note_token_tile(tile_n > 128 ? 256 : tile_n > 64 ? 128 : 64);
    slim_status_t rc;
    const bool dep = r > 0 && p.n1 > 0;               // sparse stages to run while T' is being made
    p.row_pairs = ceil_div(d_out, 2 * kPM); p.tiles = plan.tiles; p.half = tile_n / 2;
    if (!wide) {
        rc = launch_tile_kernel<64, false>(p, d_out, tmV, tmM, tmX, tmA2, tmB2, st, 1, dep);
    } else {
        const int pairs = n_pairs;
        p.departures = reinterpret_cast<unsigned long long*>(ws);
        p.t_sync = reinterpret_cast<unsigned long long*>(reinterpret_cast<char*>(ws) + SLIM_WORKSPACE_SYNC_BYTES);
        p.r = r;
        int grid = p.tiles < pairs ? p.tiles : pairs;
        if (r > 0) {
            p.t_n = plan.t_n; p.t_chunks = plan.t_chunks; p.t_tiles = plan.t_tiles; p.t_stages = d_in / PairCfg<256>::kDK;
            p.t_scale = 1.f / s_eff; p.t_out = Tq;
            p.t_part = reinterpret_cast<float4*>(reinterpret_cast<char*>(Tq) + t_bytes(b, r, t_parts));
            p.t_pairs = t_share(p.t_tiles, p.t_stages, pairs, pairs - grid, s != 0.f ? ceil_div(d_in, 128) : 0);
            p.t_even = p.t_pairs % p.t_tiles == 0 ? p.t_pairs / p.t_tiles : 0;
            grid = grid + p.t_pairs < pairs ? grid + p.t_pairs : pairs;      // the last pairs make T'
        }
        auto* launch = tile_n > 128 ? launch_pair<256, false>
                     : tile_n > 64  ? (plan.t_ranks ? launch_pair<128, true> : launch_pair<128, false>)
                                    : (plan.t_ranks ? launch_pair<64, true> : launch_pair<64, false>);
        rc = launch(p, tmV, tmM, tmX, tmA2, tmB2, tmTA, tmTB, grid, st);
    }
    if (rc != SLIM_OK) return rc;
    return SLIM_OK;
}

}  // namespace slim

#ifdef SLIM_PREFILL_TRACE
extern "C" int slim_debug_read_ptrace(unsigned long long* out) {
    return (int)cudaMemcpyFromSymbol(out, slim::g_ptrace, sizeof(slim::g_ptrace));
}
#endif
