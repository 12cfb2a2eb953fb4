// Small-batch forward (b <= 64): one launch of thread-block clusters that streams the weight and the
// adapters exactly once.
//
// Work split.  A tile is 256 output rows (up to 16 tokens of layers with fewer rows: 128 or 64); the C CTAs of a cluster
// (C = 1, 2, 4 or 8) cut d_in into C ranges of whole 256-column units.  In a CTA eight consumer warps are 4 row blocks x 2
// halves of every unit: a warp keeps the fp32 accumulators of its 64 (32, 16) rows x b tokens in registers
// through the whole range (from 33 tokens on the two halves are token halves instead), so nothing is
// summed across warps inside the stream; the partial tiles meet once, at the end: each CTA sends its own, a share of the
// rows to every CTA of the cluster, by asynchronous remote stores.  With 256-row tiles C is the largest with which the clusters of
// all tiles are resident at once (two CTAs per SM up to 16 tokens), so that a tile's stream is spread as widely as it can be; with
// lower ones see narrow_tiles.
//   The first clusters make T = X R^T instead: 32 rows of R each, the same cut of d_in; their
// CTAs exchange partial sums with asynchronous remote stores, round to bf16 (TP = 2: to two bf16 numbers, keeps_T32) and publish T as
// 8-byte words {two columns, call number}.
//   A tile's cluster streams the packed weight and the activations through a ring of stages by TMA
// (256 rows x 64 value bytes, x 32 index bytes, b tokens x 512 bytes; two requesting warps, since the engine takes about
// one 32-64 byte row a cycle and a request made on a lane's number took its warp 220 cycles),
// then the columns of L (32 of bf16, or 64 int4 codes a row and stage: codes by plain loads of the consumers, one step ahead,
// cost 8192 -> 28672 with 16 tokens 58.7 us instead of 47.6), waiting for just the words of T it multiplies, then writes
// Y = s X Q^T + T L^T.
//
// Fragments of the sparse MMA.  Inside a 256-column unit the four 64-column regions are q = 2 a + h; step
// j = 0..7 multiplies groups 2 j and 2 j + 1 of every region: thread t of a quad owns byte 2 j + (t & 1)
// of region a = t / 2 (h = 0: registers 0 and 1, h = 1: registers 2 and 3).  Then
//   - a row's 16 value bytes of a region are one thread pair's operand of eight steps: one 8-byte read
//     per row and half serves four steps, and a register costs half a shift, one prmt, one lop3 and one
//     bf16 subtraction;
//   - the index bits a lane has to supply for a step are byte j of two regions of two rows: two prmt;
//   - the activations of a step are 16 contiguous bytes per token and region: one ldmatrix.x4.
// The decode-tiled copy holds registers and index words in the instruction's natural column order instead.
// Registers: 96 a thread up to 16 tokens (two CTAs an SM), 168 above.  256-row tiles at 9 to 16 tokens spill 32 bytes there (80 with
// int4 adapters; up to 140 with T in two parts), 33 to 64 tokens 72 (up to 88 with int4).
// Alone on an SM (16 warps) a 16-row x 32-column step takes a scheduler 33 cycles at 8 tokens, 41 at 16
// (20 of them the ALU pipe's), and 24 / 33 on the tiled copy.
//
// The hand-over of T is the only wait between clusters.  It goes from lower to higher cluster numbers only:
// clusters that make T wait for nobody and are started first, so the wait ends whether or not the whole grid is
// resident.  Every poll is bounded in time, and the first to run out ends all others of the call.  An entry carries the number of the call that wrote it, so
// nothing has to be cleared between calls; the call number is (departures >> 16) + 1, and every call adds
// 1 << 16 to that counter in all.
// Reductions have a fixed order: results are bit-identical from run to run.
#include <atomic>
#include <mutex>
#include <cuda.h>
#include "decode_tile.cuh"
#include "handover.h"

namespace slim {

namespace {

using namespace dt;

constexpr int kCW = 8;                          // consumer warps
constexpr int kConsumers = kCW * 32;
constexpr int kProdW = kCW, kProdX = kCW + 1;   // requests of the weight, R and L; of the activations and the index bytes
constexpr int kFetchT = kCW + 2;                // from 17 tokens on: two warps that bring T into shared memory
constexpr int kUnit = 256;                      // columns of a stage
constexpr int kGroup = 32;                      // rows of R in one piece of the T product
constexpr unsigned long long kWaitNs = 500ull * 1000 * 1000;

enum { FMT_PACKED = 0, FMT_PACKED_LD = 1, FMT_TILED = 2 };   // LD: index bytes by cp.async (rows no 16-byte multiples)

// (A multiple of 128 bytes, as the tensor maps behind it in the parameters are: a map across two lines of 128 takes two fetches.  8192 -> 1024,
// int4 adapters, 16 tokens 8.4 us a call, with the maps 64 bytes further 8.8.)
struct alignas(128) SmallParams {
    const __nv_bfloat16* X; const uint8_t* vals; const uint8_t* meta; const uint8_t* tiled;
    const void* L; const void* R;                             // bf16, or int4 codes
    const __nv_bfloat16* Ls; const __nv_bfloat16* Rs;         // scales of quantized adapters
    __nv_bfloat16* Y;
    unsigned long long* T;                                    // [TP][b][r / 2] {bf16 pair, call number}
    unsigned long long* departures;
    uint32_t* status;
    float s;
    int b, r, d_out, d_in;
    int units, groups;                                        // of 256 columns, 32 rows of R
    int ahead;                                                // so many CTAs ask their first lines into the L2 while the grid before ends
};

// NT tiles of 8 tokens; a warp's MT tiles of 16 rows (four warps: 64 MT rows of the layer).
template <int NT, int MT> struct Cfg {
    static constexpr int kTok = NT * 8, kRows = 64 * MT;
    static constexpr int kThreads = (kCW + (NT >= 4 ? 4 : 2)) * 32;
    static constexpr int kNW = NT < 4 ? NT : 4;               // n-tiles of a warp: with eight, two warps share the tokens of a row block
    static constexpr int kTSlots = NT == 8 ? 6 : 8, kTSlot = kTok * 64;        // steps of T in shared memory: 32 columns in bf16
    static constexpr int kValsBytes = kRows * 64, kMetaBytes = kRows * 32;     // MT = 4: 24 KB, = four 6144-byte pieces of the tiled copy
    static constexpr int kXOff = MT == 4 ? kValsBytes + kMetaBytes : 16384;    // a stage of R: 16 KB
    static constexpr int kXBytes = kTok * 512;                // activations of a unit
    static constexpr int kStage = kXOff + kXBytes;
    static constexpr int kStages = NT == 4 || MT < 4 ? 4 : 3;
    static constexpr int kPiece = kTok * kGroup * 4;          // bytes of a piece of T
    static constexpr int kPitch = kRows + 4;                  // floats per token of a partial tile (conflict-free writes)
    static constexpr int kHalves = NT == 8 ? 1 : 2;
    // after the ring: in the CTAs that make T, [4][kNW * 8][kGroup] floats and the piece as the cluster sends it; in the others,
    // the steps of T, and the partial tiles that the cluster sends (eight n-tiles: these in the ring, when all CTAs are done with it)
    static constexpr int kOffPart = kStages * kStage;
    static constexpr int kOffRecv = kOffPart + 4 * kNW * 8 * kGroup * 4;
    static constexpr int kOffY = NT == 8 ? 72 * 1024 : kOffPart + (NT >= 4 ? kTSlots * kTSlot : 0), kYBytes = kTok * kRows * 4;
    static constexpr int kEndT = kOffRecv + kPiece, kEndY = NT == 8 ? kOffPart + kTSlots * kTSlot : kOffY + kYBytes;
    static constexpr int kOffBars = kEndT > kEndY ? kEndT : kEndY;
    static constexpr int kSmem = kOffBars + 256;
    static constexpr int kCtasPerSm = NT <= 2 ? 2 : 1;
    static_assert(kHalves * kTok * kPitch * 4 <= (NT == 8 ? kOffY : kOffPart) && (NT < 8 || kOffY + kYBytes <= kOffPart), "partial tiles do not fit the ring");
    static_assert(kSmem <= (NT <= 2 ? 113 : 227) * 1024, "shared memory");
};

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint32_t peer(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void mbar_arrive_peer(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" :: "r"(bar) : "memory");
}
__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// An entry of T is one 64-bit access: value and call number are seen together.
__device__ __forceinline__ unsigned long long ld_gpu64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_gpu64(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" :: "l"(p), "l"(v) : "memory");
}
// Whether a wait that began at *t0 (0: it starts now) is to be given up: it has taken kWaitNs, or another wait of this call, in whatever
// CTA, has.  The first to expire leaves the call's number in the word behind the departures, so a broken call costs one such
// time, not one a step and CTA (3072 ranks in one CTA: 96 steps to wait for).
__device__ __forceinline__ bool give_up(unsigned long long* sync, unsigned long long* t0) {
    const unsigned long long now = now_ns();
    if (*t0 == 0) *t0 = now;
    const uint32_t call = call_number(ld_gpu64(sync));
    if (is_of(ld_gpu64(sync + 1), call)) return true;
    if (now - *t0 <= kWaitNs) return false;
    st_gpu64(sync + 1, tagged(call, 0));
    return true;
}
// Waits for a phase, for kWaitNs at most (a try may suspend the thread, so the bound is on time).
template <bool CLUSTER = false>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, unsigned long long* sync) {
    unsigned long long t0 = 0;
    for (uint32_t it = 0;; ++it) {
        uint32_t done;
        if (CLUSTER)
            asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                         : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        else
            asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                         : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        if (done) return true;
        if ((it & 63u) == 63u && give_up(sync, &t0)) return false;
    }
}
__device__ __forceinline__ void tma_tile(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 :: "r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void tma_tile3(uint32_t dst, const CUtensorMap* map, int y, int z, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 :: "r"(dst), "l"(map), "r"(0), "r"(y), "r"(z), "r"(bar) : "memory");
}
// One lane of a warp whose lanes have all come here.  Requests are made in such a branch, from operands that are the same in all lanes: a
// branch on the lane's number took longer (4096 -> 11008, rank 416, 16 tokens 17.1 us a call, 15.7 so; 28672 -> 8192, 16 tokens 48.9,
// 46.6; 8192 -> 8192, rank 832, one token 18.6, 18.0).
__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
    return pred != 0;
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) { asm volatile("prefetch.tensormap [%0];" :: "l"(map) : "memory"); }
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// Eight bytes, or (not `in`) eight zero bytes.
__device__ __forceinline__ void cp_async8(uint32_t dst, const void* src, bool in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" :: "r"(dst), "l"(src), "r"(in ? 8 : 0) : "memory");
}
__device__ __forceinline__ void consumer_sync() { asm volatile("bar.sync 1, %0;" :: "n"(kConsumers) : "memory"); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Eight or sixteen bytes into a peer's shared memory; its barrier counts them.
__device__ __forceinline__ void st_peer4(uint32_t addr, float4 v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                 :: "r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_peer2(uint32_t addr, float x, float y, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" :: "r"(addr), "f"(x), "f"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void sts_f(uint32_t addr, float v) { asm volatile("st.shared.f32 [%0], %1;" :: "r"(addr), "f"(v) : "memory"); }
__device__ __forceinline__ void sts32(uint32_t addr, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" :: "r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ float2 lds_f2(uint32_t addr) { float2 v; asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr)); return v; }
__device__ __forceinline__ float4 lds_f4(uint32_t addr) { float4 v; asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr)); return v; }
__device__ __forceinline__ uint2 lds64(uint32_t addr) {
    return *reinterpret_cast<const uint2*>(__cvta_shared_to_generic(addr));
}
// Two entries, each seen whole (the vector form is two 64-bit accesses).
__device__ __forceinline__ void ld_gpu64x2(const unsigned long long* p, unsigned long long& x, unsigned long long& y) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(p) : "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t addr, uint4& v) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
}
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}
// Eight int4 codes of a word give, shifted by 4 i, the pair (c_i, c_{i+4}); the other operand's eight
// consecutive bf16 values are put in the same order.
__device__ __forceinline__ uint4 pair_four_apart(const uint4& v) {
    return make_uint4(prmt(v.x, v.z, 0x5410), prmt(v.x, v.z, 0x7632), prmt(v.y, v.w, 0x5410), prmt(v.y, v.w, 0x7632));
}

static_assert(sizeof(SmallParams) == 128, "the tensor maps' place in the parameters");

// ---------------------------------------------------------------- one stage of the weight
struct Lane { int lane, g, t; };

// Rows past d_out and columns past d_in arrive as zero bytes.  Zero values are what they should be, but zero index
// bits name one position twice: before a ragged stage is multiplied every lane completes the index words it will
// read itself (0x4: positions 0 and 1).
template <int MT>
__device__ __forceinline__ void complete_index(uint32_t stage, int rb, int kk, int mts, int cols_left, const Lane& ln)
{
    const int h = ln.t & 1, g = ln.g;
    const uint32_t mrow = stage + MT * 4096 + (uint32_t)(rb * 16 * MT + g) * 32 + h * 8 + kk * 4, mx = (uint32_t)(g >> 2) & 1;
    for (int i = 0; i < 2 * MT; ++i)                              // rows g + 8 i; regions h and 2 + h
#pragma unroll
        for (int a = 0; a < 2; ++a)
            if ((i >> 1) >= mts || 64 * (2 * a + h) >= cols_left) sts32(mrow + i * 256 + (((uint32_t)a ^ mx) << 4), 0x44444444u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the next use of the stage is written by TMA
    __syncwarp();
}

// This warp's 16 MT rows x half a unit (four steps) of a packed-format stage, NB n-tiles from tile n0 on.
// KS steps' activations are held at a time: four where the registers allow it, else two.
template <int NT, int NB, int MT>
__device__ __forceinline__ void weight_stage(float (&acc)[MT][NB][4], uint32_t stage, int rb, int kk, int n0, const Lane& ln)
{
    constexpr int KS = NB <= 2 ? 4 : 2;
    const int a = ln.t >> 1, h = ln.t & 1, g = ln.g;
    // value bytes: 64-byte rows, 64-byte swizzle; index bytes: 32-byte rows, 32-byte swizzle
    const uint32_t vrow = stage + (uint32_t)(rb * 16 * MT + g) * 64 + kk * 8, vx = (uint32_t)(g >> 1) & 3;
    const uint32_t v0 = vrow + (((uint32_t)(2 * a) ^ vx) << 4), v1 = vrow + (((uint32_t)(2 * a + 1) ^ vx) << 4);
    const uint32_t mrow = stage + MT * 4096 + (uint32_t)(rb * 16 * MT + g) * 32 + h * 8 + kk * 4, mx = (uint32_t)(g >> 2) & 1;
    const uint32_t m0 = mrow + (mx << 4), m1 = mrow + ((mx ^ 1) << 4);
    // activations: 64-column sub-tiles of 128-byte token rows, 128-byte swizzle; lane l addresses row l & 7 of matrix l / 8
    const int mat = ln.lane >> 3, tok = ln.lane & 7, q = 2 * (mat & 1) + (mat >> 1);
    const uint32_t xrow = stage + Cfg<NT, MT>::kXOff + (uint32_t)q * (NT * 1024) + (uint32_t)(n0 * 8 + tok) * 128;
    const uint32_t sel_e = 0x4400u + (uint32_t)h * 0x1111u, sel_o = sel_e + 0x2222u;     // byte h (+ 2) of w and of w >> 4
#pragma unroll
    for (int s0 = 0; s0 < 4; s0 += KS) {
        uint4 xb[KS][NB];
#pragma unroll
        for (int s = 0; s < KS; ++s)
#pragma unroll
            for (int n = 0; n < NB; ++n)
                ldsm4(xrow + n * 1024 + ((((uint32_t)(kk * 4 + s0 + s)) ^ (uint32_t)tok) << 4), xb[s][n]);
        // which two steps' index words this lane supplies: with four steps a quad's lanes share the work
        const uint32_t S = KS == 4 ? (uint32_t)a : (uint32_t)(s0 >> 1);
        const uint32_t msel = (2 * S) | ((4 + 2 * S) << 4) | ((2 * S + 1) << 8) | ((5 + 2 * S) << 12);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            const uint32_t vo = mt * 1024, mo = mt * 512;
            uint32_t w[4][KS / 2];                            // (row g, h 0), (row g + 8, h 0), (row g, h 1), (row g + 8, h 1)
            if (KS == 4) {
                const uint2 x0 = lds64(v0 + vo), x1 = lds64(v0 + vo + 512), x2 = lds64(v1 + vo), x3 = lds64(v1 + vo + 512);
                w[0][0] = x0.x; w[1][0] = x1.x; w[2][0] = x2.x; w[3][0] = x3.x;
                w[0][KS / 2 - 1] = x0.y; w[1][KS / 2 - 1] = x1.y; w[2][KS / 2 - 1] = x2.y; w[3][KS / 2 - 1] = x3.y;
            } else {
                w[0][0] = lds32(v0 + vo + s0 * 2); w[1][0] = lds32(v0 + vo + 512 + s0 * 2);
                w[2][0] = lds32(v1 + vo + s0 * 2); w[3][0] = lds32(v1 + vo + 512 + s0 * 2);
            }
            const uint32_t u = prmt(lds32(m0 + mo), lds32(m1 + mo), msel), v = prmt(lds32(m0 + mo + 256), lds32(m1 + mo + 256), msel);
            const uint32_t e0 = prmt(u, v, 0x5410), e1 = prmt(u, v, 0x7632);
#pragma unroll
            for (int s = 0; s < KS; ++s) {
                uint32_t ar[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t ww = w[i][s >> 1];
                    ar[i] = nibbles_to_bf16x2(prmt(ww, ww >> 4, (s & 1) ? sel_o : sel_e));
                }
#pragma unroll
                for (int n = 0; n < NB; ++n) {
                    if (s < 2) mma_sp_16832<0>(acc[mt][n], ar, xb[s][n], (s & 1) ? e1 : e0);
                    else       mma_sp_16832<1>(acc[mt][n], ar, xb[s][n], (s & 1) ? e1 : e0);
                }
            }
        }
    }
}

// The same for a stage of the decode-tiled copy (its row groups are complete): registers and index words in the
// instruction's column order.
template <int NT>
__device__ __forceinline__ void weight_stage_tiled(float (&acc)[4][NT][4], uint32_t stage, int rb, int kk, const Lane& ln)
{
    const int mat = ln.lane >> 3, tok = ln.lane & 7;
    const uint32_t xrow = stage + Cfg<NT, 4>::kXOff + (uint32_t)tok * 128;
    const uint32_t piece0 = stage + (uint32_t)rb * 6144;
    const uint32_t idx_lane = (uint32_t)(ln.g * 4 + 2 * kk + (ln.t & 1));       // the lane that holds this half's index words
#pragma unroll
    for (int s0 = 0; s0 < 4; s0 += 2) {
        uint4 xb[2][NT];
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int n = 0; n < NT; ++n)   // step j = 4 kk + s0 + s: columns 32 j + 8 mat, sub-tile j / 2
                ldsm4(xrow + (uint32_t)(2 * kk + (s0 >> 1)) * (NT * 1024) + n * 1024 + ((uint32_t)((s * 4 + mat) ^ tok) << 4), xb[s][n]);
        uint2 w[4], e[4];
#pragma unroll
        for (int mt = 0; mt < 4; ++mt) {
            w[mt] = lds64(piece0 + mt * 1536 + kk * 512 + ln.lane * 16 + s0 * 4);
            e[mt] = lds64(piece0 + mt * 1536 + 1024 + idx_lane * 16 + s0 * 4);
        }
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int mt = 0; mt < 4; ++mt) {
                const uint32_t ww = s ? w[mt].y : w[mt].x;
                uint32_t ar[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) ar[i] = nibbles_to_bf16x2(ww >> (4 * i));
#pragma unroll
                for (int n = 0; n < NT; ++n) mma_sp_16832<0>(acc[mt][n], ar, xb[s][n], s ? e[mt].y : e[mt].x);
            }
    }
}

// ---------------------------------------------------------------- one stage of R
// 32 rows of R x 256 columns: warp = (16-row tile m, 64-column sub-tile kq).
template <int NT, int MT>
__device__ __forceinline__ void adapter_stage(float (&acc)[NT][4], uint32_t stage, int m, int kq, const Lane& ln)
{
    const int mat = ln.lane >> 3, r8 = ln.lane & 7;
    const uint32_t arow = stage + (uint32_t)kq * 4096 + (uint32_t)(m * 16 + (mat & 1) * 8 + r8) * 128;
    const uint32_t xrow = stage + Cfg<NT, MT>::kXOff + (uint32_t)kq * (NT * 1024) + (uint32_t)r8 * 128;
#pragma unroll
    for (int s = 0; s < 2; ++s) {                  // 32 columns
        uint4 a0, a1;
        ldsm4(arow + ((uint32_t)((4 * s + (mat >> 1)) ^ r8) << 4), a0);
        ldsm4(arow + ((uint32_t)((4 * s + 2 + (mat >> 1)) ^ r8) << 4), a1);
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            uint4 x;
            ldsm4(xrow + n * 1024 + ((uint32_t)((4 * s + mat) ^ r8) << 4), x);
            mma_16816(acc[n], a0.x, a0.y, a0.z, a0.w, x.x, x.y);
            mma_16816(acc[n], a1.x, a1.y, a1.z, a1.w, x.z, x.w);
        }
    }
}
// The same on int4 codes.  A word of a row is eight columns; the activations of a step are read as the thread's
// own eight columns and paired four apart.  The 64 columns lie in one group: the integer products are scaled once.
template <int NT, int MT>
__device__ __forceinline__ void adapter_stage_q(float (&acc)[NT][4], uint32_t stage, int m, int kq, float sc0, float sc1, const Lane& ln)
{
    const uint32_t arow = stage + (uint32_t)(m * 16 + ln.g) * 128 + ln.t * 4;
    const uint32_t xrow = stage + Cfg<NT, MT>::kXOff + (uint32_t)kq * (NT * 1024) + (uint32_t)ln.g * 128;
    float part[NT][4];
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) part[n][e] = 0.f;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const uint32_t lo = lds32(arow + ((uint32_t)((2 * kq + s) ^ ln.g) << 4)), hi = lds32(arow + 1024 + ((uint32_t)((2 * kq + s) ^ ln.g) << 4));
        uint32_t a[4], c[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) { a[i] = nibbles_to_bf16x2(lo >> (4 * i)); c[i] = nibbles_to_bf16x2(hi >> (4 * i)); }
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            const uint4 x = pair_four_apart(lds128(xrow + n * 1024 + ((uint32_t)((4 * s + ln.t) ^ ln.g) << 4)));
            mma_16816(part[n], a[0], c[0], a[1], c[1], x.x, x.y);
            mma_16816(part[n], a[2], c[2], a[3], c[3], x.z, x.w);
        }
    }
#pragma unroll
    for (int n = 0; n < NT; ++n) {
        acc[n][0] = fmaf(part[n][0], sc0, acc[n][0]); acc[n][1] = fmaf(part[n][1], sc0, acc[n][1]);
        acc[n][2] = fmaf(part[n][2], sc1, acc[n][2]); acc[n][3] = fmaf(part[n][3], sc1, acc[n][3]);
    }
}

// The words of T that B fragments need (two columns each), asked for by `ask` (a padding token or column is there at once, zero)
// and waited for.
// Where words are missing, one lane polls one of them, and all are asked for again when it has come: the tiles of a layer
// wait for the same words, and with every lane polling its own (1024 warps on a few lines of the L2) the words
// themselves came 1-3 us later (2048 -> 2048, rank 208, 6 tokens: 6.8 us a call instead of 7.5).
template <int NE, typename A, typename W>
__device__ __forceinline__ bool wait_words(unsigned long long (&v)[NE], uint32_t call, unsigned long long* sync, A ask, W word)
{
    for (int round = 0; round < 64; ++round) {
        const unsigned long long* w = nullptr;
#pragma unroll
        for (int n = 0; n < NE; ++n) if (!w && !is_of(v[n], call)) w = word(n);
        const uint32_t missing = __ballot_sync(0xffffffffu, w != nullptr);
        if (!missing) return true;
        bool late = false;
        if ((int)(threadIdx.x & 31) == __ffs(missing) - 1) {
            unsigned long long t0 = 0;
            for (uint32_t spin = 0; !late && !is_of(ld_gpu64(w), call); ++spin) {
                if ((spin & 63u) == 63u) late = give_up(sync, &t0);
                __nanosleep(20);
            }
        }
        if (__any_sync(0xffffffffu, late)) return false;
        ask();
    }
    return false;
}
// The words of eight codes of rows g and g + 8 of a 16-row tile, step h of a stage of L's codes (32-byte rows, 32-byte
// swizzle), and their product with T.  Integer products are scaled once.
template <int MT>
__device__ __forceinline__ uint2 l_codes(uint32_t stage, int rb, int m, int h, const Lane& ln) {
    const uint32_t at = stage + (uint32_t)((rb * MT + m) * 16 + ln.g) * 32 + ((uint32_t)(h ^ (ln.g >> 2)) << 4) + ln.t * 4;
    return make_uint2(lds32(at), lds32(at + 256));
}
template <int NW>
__device__ __forceinline__ void code_tile(float (&acc)[NW][4], uint2 w, float sc0, float sc1, const uint4 (&tb)[NW])
{
    uint32_t a[4], d[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) { a[q] = nibbles_to_bf16x2(w.x >> (4 * q)); d[q] = nibbles_to_bf16x2(w.y >> (4 * q)); }
#pragma unroll
    for (int n = 0; n < NW; ++n) {
        float pt[4] = {0.f, 0.f, 0.f, 0.f};
        mma_16816(pt, a[0], d[0], a[1], d[1], tb[n].x, tb[n].y);
        mma_16816(pt, a[2], d[2], a[3], d[3], tb[n].z, tb[n].w);
        acc[n][0] = fmaf(pt[0], sc0, acc[n][0]); acc[n][1] = fmaf(pt[1], sc0, acc[n][1]);
        acc[n][2] = fmaf(pt[2], sc1, acc[n][2]); acc[n][3] = fmaf(pt[3], sc1, acc[n][3]);
    }
}

// The tile of a CTA, its two halves (eight n-tiles: one) added up, goes to the CTAs of the cluster, a share of the rows to
// each: four rows of a token at a time, [sender][token][rows of the share].  (The CTAs reading the partial tiles out of each
// other's shared memory, both halves, took 2 us longer for 16 tokens and 0.5 us for one.)
template <int NT, int MT>
__device__ __forceinline__ void send(const SmallParams& p, uint32_t smem, uint32_t red_full, int logC, int rank)
{
    using C_ = Cfg<NT, MT>;
    constexpr int kQuads = C_::kRows / 4;
    const int share = kQuads >> logC;
    for (int e = threadIdx.x; e < p.b * kQuads; e += kConsumers) {
        const int tok = e / kQuads, q = e % kQuads, owner = q / share;
        const uint32_t at = smem + (uint32_t)(tok * C_::kPitch + 4 * q) * 4;
        float4 v = lds_f4(at);
        if (C_::kHalves == 2) {
            const float4 w = lds_f4(at + C_::kTok * C_::kPitch * 4);
            v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
        }
        st_peer4(peer(smem + C_::kOffY + (uint32_t)((rank * p.b + tok) * share + (q & (share - 1))) * 16, owner), v, peer(red_full, owner));
    }
}
// Y of the rows of this CTA's share: the senders' sums in a fixed order.
template <int NT, int MT>
__device__ __forceinline__ void finish(const SmallParams& p, uint32_t smem, int tile, int logC, int rank)
{
    using C_ = Cfg<NT, MT>;
    const int share = (C_::kRows / 4) >> logC, items = p.b * share, C = 1 << logC;
    for (int e = threadIdx.x; e < items; e += kConsumers) {
        const uint32_t at = smem + C_::kOffY + (uint32_t)e * 16;
        float4 v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) if (c < C) v[c] = lds_f4(at + (uint32_t)(c * items) * 16);
        float4 y = v[0];
#pragma unroll
        for (int c = 1; c < 8; ++c) if (c < C) { y.x += v[c].x; y.y += v[c].y; y.z += v[c].z; y.w += v[c].w; }
        const int tok = e / share, n = tile * C_::kRows + 4 * (rank * share + (e & (share - 1)));
        if (n < p.d_out) {
            __nv_bfloat162 lo = __floats2bfloat162_rn(y.x, y.y), hi = __floats2bfloat162_rn(y.z, y.w);
            *reinterpret_cast<uint2*>(p.Y + (size_t)tok * p.d_out + n) = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
        }
    }
}

// Asks bytes [from, to) of `rows` rows from row0 on into the L2, up to eight lines a consumer: ROWS rows side by side, then the next lines
// of each.  (Where rows are whole lines, one that begins before `from` is asked for with the bytes that it begins with; where they are not, bytes
// of two CTAs share lines that neither need see whole, and both ask: 5504 -> 4096, rank 416, 4 tokens 8.95 us, 8.83 so.)
template <int ROWS>
__device__ __forceinline__ void lines_ahead(const void* base, size_t pitch, int row0, int rows, size_t from, size_t to)
{
    constexpr size_t kLine = 128, kBeside = kConsumers / ROWS;
    const int row = threadIdx.x % ROWS;
    if (row >= rows) return;
    const char* at_row = static_cast<const char*>(base) + (size_t)(row0 + row) * pitch;
    size_t at = (from + (from > 0 && pitch % kLine == 0 ? kLine - 1 : 0)) / kLine * kLine + threadIdx.x / ROWS * kLine;
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (at + i * (kBeside * kLine) < to) asm volatile("prefetch.global.L2 [%0];" :: "l"(at_row + at + i * (kBeside * kLine)));
}

// ---------------------------------------------------------------- the kernel
template <int NT, int FMT, bool QA, int MT, int TP>
__global__ void __launch_bounds__(Cfg<NT, MT>::kThreads, Cfg<NT, MT>::kCtasPerSm)
small_kernel(const SmallParams p, const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmM,
             const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmR, const __grid_constant__ CUtensorMap tmL)
{
    using C_ = Cfg<NT, MT>;
    static_assert(MT == 4 || (NT <= 2 && FMT != FMT_TILED), "narrow tiles: up to 16 tokens, packed format");
    static_assert(TP == 1 || FMT != FMT_TILED, "T in two parts: packed format");
    const int t_tail = TP == 2 ? p.b * (p.r / 2) : 0;          // from T's first part to the second
    constexpr int kTok = C_::kTok, kNW = C_::kNW, kStages = C_::kStages, kStage = C_::kStage, kRows = C_::kRows;
    constexpr int kValsBytes = C_::kValsBytes, kMetaBytes = C_::kMetaBytes, kXOff = C_::kXOff;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t smem = smem_u32(smem_raw);
    const uint32_t part = smem + C_::kOffPart, recv = smem + C_::kOffRecv, bars = smem + C_::kOffBars;
    const uint32_t full = bars, empty = bars + 32, piece_bar = bars + 64, red_full = bars + 72, t_full = bars + 80, t_empty = bars + 144, gone = bars + 208;

    const int lane = threadIdx.x & 31;
    // (role, a shuffle: the same in all lanes, for the compiler too.  Not so the consumers' warp: see `release`.)
    const int warp = threadIdx.x >> 5, role = QA ? warp : __shfl_sync(0xffffffffu, warp, 0);
    // The lane that requests.  (Beside int4 adapters the branch on the lane's number, two lanes' requests with one instruction, is the faster one:
    // 5120 x 5120, rank 512, 7 tokens 8.1 us against 8.5, 4096 x 4096, rank 208, 6 tokens 6.5 against 7.1, weights in the L2.)
    auto asks = [&] { return QA ? lane == 0 : elect_one(); };
    Lane ln; ln.lane = lane; ln.g = lane >> 2; ln.t = lane & 3;
    uint32_t C, rank;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int logC = 31 - __clz((int)C);
    // the first clusters make T, a piece each, and wait for nobody; the others wait for them
    const int cluster = blockIdx.x >> logC;
    const bool makes_T = cluster < p.groups;
    const int piece = cluster, tile = cluster - p.groups;
    const int u0 = (int)(rank * (unsigned)p.units) >> logC, u1 = (int)((rank + 1) * (unsigned)p.units) >> logC;
    const int u_end = p.s != 0.f ? u1 : u0;                    // s == 0: the adapter term alone
    const int l_steps = ceil_div(p.r, 32), l_chunks = ceil_div(p.r, QA ? 64 : 32);      // steps of 32 columns; stages of L

    if (threadIdx.x == 0) {
        // a stage's barrier counts both producers (and, with index bytes by cp.async, the lanes of one of them)
        for (int i = 0; i < kStages; ++i) { mbar_init(full + 8 * i, FMT == FMT_PACKED_LD ? 34 : 2); mbar_init(empty + 8 * i, kCW); }
        mbar_init(piece_bar, 1); mbar_init(red_full, 1); mbar_init(gone, C);
        if (NT >= 4) for (int i = 0; i < C_::kTSlots; ++i) { mbar_init(t_full + 8 * i, 2); mbar_init(t_empty + 8 * i, kCW); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // every CTA of the cluster sends this one its share of the piece: 16 / C column pairs per token
        mbar_expect(piece_bar, (uint32_t)p.b * 16 * 8);
        // and its share of the rows of the tile, four bytes per token and row
        mbar_expect(red_full, (uint32_t)p.b * kRows * 4);
    }
    __syncthreads();
    cluster_arrive();                                          // waited for before the first access to a peer
    // Launched while the grid before it in the stream still runs (programmatic dependent launch): everything above needs
    // no global memory, everything below comes after that grid.  The next grid may be set up as soon as all CTAs are here.
    if (role == kProdW && lane == 0) { prefetch_map(FMT == FMT_TILED ? &tmX : &tmV); prefetch_map(&tmR); prefetch_map(&tmL); }
    if (role == kProdX && lane == 0) { prefetch_map(&tmX); prefetch_map(&tmM); }
    // The first lines of this CTA's part of the weight or of R go into the L2 meanwhile.  Nothing is read by that: what the grid before still
    // writes is what the loads behind the wait find there.
    if (NT <= 2 && FMT != FMT_TILED && !QA && (int)blockIdx.x < p.ahead && warp < kCW) {
        const size_t c0 = (size_t)u0 * kUnit, c1 = min((size_t)(makes_T ? u1 : u_end) * kUnit, (size_t)p.d_in);
        if (makes_T) {
            lines_ahead<kGroup>(p.R, (size_t)p.d_in * 2, piece * kGroup, min(kGroup, p.r - piece * kGroup), c0 * 2, c1 * 2);
        } else {
            const int row0 = tile * kRows, rows = min(kRows, p.d_out - row0);
            lines_ahead<kRows>(p.vals, (size_t)p.d_in / 4, row0, rows, c0 / 4, c1 / 4);
            lines_ahead<kRows>(p.meta, (size_t)p.d_in / 8, row0, rows, c0 / 8, c1 / 8);
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (role == kProdW || role == kProdX) asm volatile("fence.proxy.async;" ::: "memory");      // what that grid wrote is read through TMA
    bool ok = true;

    int p_it = 0;                                              // producers: next stage
    auto acquire = [&]() -> int {
        const int st = p_it % kStages, use = p_it / kStages;
        if (use > 0) ok = mbar_wait(empty + 8 * st, (use - 1) & 1, p.departures) && ok;
        ++p_it;
        return st;
    };
    // L's codes where rows of r / 2 bytes are no 16-byte multiples, half of the tile by either producer: 8-byte pieces, stored
    // as the TMA's 32-byte swizzle would.  Each lane's pieces are one more arrival that the barrier waits for.
    const bool l_by_lanes = QA && p.r % 32 != 0;
    auto codes_of_L = [&](int lc, uint32_t dst, uint32_t bar, int first) {
        const int q = lane & 3, row0 = tile * kRows;
        const bool col_in = lc * 64 + q * 16 < p.r;
#pragma unroll 4
        for (int r = first + (lane >> 2); r < first + kRows / 2; r += 8) {
            const bool in = col_in && row0 + r < p.d_out;
            const uint8_t* src = static_cast<const uint8_t*>(p.L) + (in ? (size_t)(row0 + r) * (p.r / 2) + lc * 32 + q * 8 : 0);
            cp_async8(dst + r * 32 + (((q >> 1) ^ ((r >> 2) & 1)) << 4) + (q & 1) * 8, src, in);
        }
        asm volatile("cp.async.mbarrier.arrive.shared::cta.b64 [%0];" :: "r"(bar) : "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(bar);
    };
    if (role == kProdW) {
        // ============================ the weight, R, L ============================
        const int row0 = tile * kRows;
        if (makes_T) {
            for (int u = u0; u < u1; ++u) {
                const int st = acquire();
                const uint32_t bar = full + 8 * st;
                if (asks()) {
                    mbar_expect(bar, QA ? 4096 : 16384);
                    if (QA) tma_tile(smem + st * kStage, &tmR, u * 128, piece * kGroup, bar);
                    else tma_tile3(smem + st * kStage, &tmR, piece * kGroup, u * 4, bar);
                }
            }
        } else {
            const int groups = FMT == FMT_TILED ? min(4, ceil_div(p.d_out - row0, 64)) : 0;
            for (int u = u0; u < u_end; ++u) {
                const int st = acquire();
                const uint32_t dst = smem + st * kStage, bar = full + 8 * st;
                if (asks()) {
                    mbar_expect(bar, FMT == FMT_TILED ? groups * 6144 : kValsBytes);
                    if (FMT == FMT_TILED) {
                        for (int i = 0; i < groups; ++i) bulk_copy(dst + i * 6144, p.tiled + ((size_t)(tile * 4 + i) * p.units + u) * 6144, 6144, bar);
                    } else {
                        tma_tile(dst, &tmV, u * 64, row0, bar);
                    }
                }
            }
            // 32 columns of L in bf16, or 64 codes a row
            for (int lc = (int)rank; lc < l_chunks; lc += (int)C) {
                const int st = acquire();
                const uint32_t dst = smem + st * kStage, bar = full + 8 * st;
                if (l_by_lanes) {
                    codes_of_L(lc, dst, bar, 0);
                } else if (asks()) {
                    mbar_expect(bar, kRows * (QA ? 32 : 64));
                    mbar_arrive(bar);                           // in place of the other producer
                    tma_tile(dst, &tmL, lc * 32, row0, bar);
                }
                if (FMT == FMT_PACKED_LD) mbar_arrive(bar);
            }
        }
        cluster_wait();
    } else if (role == kProdX) {
        // ============================ activations, index bytes ============================
        const int row0 = tile * kRows;
        if (makes_T) {
            for (int u = u0; u < u1; ++u) {
                const int st = acquire();
                const uint32_t bar = full + 8 * st;
                if (asks()) {
                    mbar_expect(bar, C_::kXBytes);
                    tma_tile3(smem + st * kStage + kXOff, &tmX, 0, u * 4, bar);
                }
                if (FMT == FMT_PACKED_LD) mbar_arrive(bar);
            }
            // this CTA's share of the piece, once every CTA of the cluster has sent its sums
            const uint32_t call = call_number(ld_gpu64(p.departures));
            const int per = 16 >> logC;                        // column pairs of a token that this CTA adds up
            ok = mbar_wait<true>(piece_bar, 0, p.departures) && ok;
            for (int e = lane; e < p.b * per; e += 32) {
                const int tok = e / per, j = piece * kGroup + 2 * ((int)rank * per + e % per);
                float2 s = lds_f2(recv + e * 8);
#pragma unroll
                for (int c = 1; c < 8; ++c)
                    if (c < (int)C) {
                        const float2 v = lds_f2(recv + (c * p.b * per + e) * 8);
                        s.x += v.x; s.y += v.y;
                    }
                if (j < p.r)
#pragma unroll
                    for (int part = 0; part < TP; ++part) {
                        __nv_bfloat162 pr = TP == 1    ? __floats2bfloat162_rn(s.x, s.y)
                                            : part == 0 ? __floats2bfloat162_rn(bf16_head(s.x), bf16_head(s.y))
                                                        : __floats2bfloat162_rn(bf16_tail(s.x), bf16_tail(s.y));
                        st_gpu64(p.T + part * t_tail + (size_t)tok * (p.r / 2) + (j >> 1), tagged(call, *reinterpret_cast<uint32_t*>(&pr)));
                    }
            }
        } else {
            for (int u = u0; u < u_end; ++u) {
                const int st = acquire();
                const uint32_t dst = smem + st * kStage, bar = full + 8 * st;
                if (QA) {                                       // (both requests with one instruction)
                    if (lane == 0) mbar_expect(bar, C_::kXBytes + (FMT == FMT_PACKED ? kMetaBytes : 0));
                    __syncwarp();
                    if (lane == 0) tma_tile3(dst + kXOff, &tmX, 0, u * 4, bar);
                    if (FMT == FMT_PACKED && lane == 1) tma_tile(dst + kValsBytes, &tmM, u * 32, row0, bar);
                } else if (elect_one()) {
                    mbar_expect(bar, C_::kXBytes + (FMT == FMT_PACKED ? kMetaBytes : 0));
                    if (FMT == FMT_PACKED) tma_tile(dst + kValsBytes, &tmM, u * 32, row0, bar);
                    tma_tile3(dst + kXOff, &tmX, 0, u * 4, bar);
                }
                if (FMT == FMT_PACKED_LD) {
                    // 256 rows x four 8-byte pieces (64 columns), stored as the TMA's 32-byte swizzle would
                    const size_t pitch = (size_t)p.d_in / 8;
                    const int q = lane & 3;
                    const bool col_in = u * kUnit + q * 64 < p.d_in;
#pragma unroll 4
                    for (int r = lane >> 2; r < kRows; r += 8) {
                        const bool in = col_in && row0 + r < p.d_out;
                        const uint8_t* src = p.meta + (in ? (size_t)(row0 + r) * pitch + (size_t)u * 32 + q * 8 : 0);
                        const uint32_t d = dst + kValsBytes + r * 32 + (((q >> 1) ^ ((r >> 2) & 1)) << 4) + (q & 1) * 8;
                        cp_async8(d, src, in);
                    }
                    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" :: "r"(bar) : "memory");
                }
            }
            if (l_by_lanes)
                for (int lc = (int)rank; lc < l_chunks; lc += (int)C) {
                    const int st = acquire();
                    codes_of_L(lc, smem + st * kStage, full + 8 * st, kRows / 2);
                }
        }
        cluster_wait();
    } else if (NT >= 4 && warp >= kFetchT) {
        // ============================ T into shared memory, step by step ============================
        // [token][32 columns] bf16, 64-byte rows stored with the 64-byte swizzle; each of the two warps half of the tokens
        if (!makes_T && p.r > 0) {
            const uint32_t call = call_number(ld_gpu64(p.departures));
            constexpr int kPer = NT * 2;                       // words a lane fetches
            const int steps = (l_chunks - (int)rank + (int)C - 1) / (int)C * (QA ? 2 : 1);
            for (int it = 0; it < steps; ++it) {
                const int ls = QA ? 2 * ((int)rank + (it >> 1) * (int)C) + (it & 1) : (int)rank + it * (int)C;
                unsigned long long v[TP * kPer];               // both parts of T are under way together
                const int pr = lane & 15, tok0 = (warp - kFetchT) * (kTok / 2) + (lane >> 4);
                const unsigned long long* at = p.T + (size_t)tok0 * (p.r / 2) + ls * 16 + pr;
                const int toks = ls * 32 + 2 * pr < p.r ? p.b - tok0 : 0;
                auto ask = [&] {
#pragma unroll
                    for (int n = 0; n < TP * kPer; ++n) {
                        const int i = n % kPer;
                        v[n] = 2 * i < toks ? ld_gpu64(at + (n / kPer) * t_tail + i * p.r) : tagged(call, 0);
                    }
                };
                ask();
                ok = wait_words(v, call, p.departures, ask, [&](int n) { return at + (n / kPer) * t_tail + (n % kPer) * p.r; }) && ok;
#pragma unroll
                for (int tp = 0; tp < TP; ++tp) {
                    const int slot = it * TP + tp, st = slot % C_::kTSlots, use = slot / C_::kTSlots;
                    if (use > 0) ok = mbar_wait(t_empty + 8 * st, (use - 1) & 1, p.departures) && ok;
#pragma unroll
                    for (int i = 0; i < kPer; ++i) {
                        const int tok = tok0 + 2 * i;
                        sts32(part + st * C_::kTSlot + tok * 64 + (((pr >> 2) ^ ((tok >> 1) & 3)) << 4) + (pr & 3) * 4, (uint32_t)v[tp * kPer + i]);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(t_full + 8 * st);
                }
            }
        }
        cluster_wait();
    } else {
        // ============================ consumer warps ============================
        uint32_t call = 0;
        if (p.r > 0) call = call_number(ld_gpu64(p.departures));
        int it = 0;
        auto wait_stage = [&]() -> uint32_t {
            const int st = it % kStages;
            ok = mbar_wait(full + 8 * st, (it / kStages) & 1, p.departures) && ok;
            __syncwarp();                                      // lanes find the phase ended one by one, and what follows takes the whole warp (ldmatrix, mma)
            return smem + st * kStage;
        };
        // The stage's reads are over before TMA, another proxy, writes it again: an arrival does not say so by itself.  (With addresses that the compiler
        // knew to be the same in all lanes arrivals overtook ldmatrix: with more steps of L than places in the ring rows came out wrong.)
        auto release = [&]() {
            __syncwarp();
            if (lane == 0) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_arrive(empty + 8 * (it % kStages));
            }
            ++it;
        };
        if (makes_T) {
            // ---------------- a piece of T
            const int m = warp & 1, kq = warp >> 1;
            const bool valid = piece * kGroup + m * 16 < p.r;
            float acc[NT][4];
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[n][e] = 0.f;
            for (int u = u0; u < u1; ++u) {
                float sc0 = 0.f, sc1 = 0.f;
                if (QA && valid && u * kUnit + 64 * kq < p.d_in) {
                    const size_t per_row = (size_t)((p.d_in + 127) >> 7);
                    const __nv_bfloat16* s = p.Rs + (size_t)(piece * kGroup + m * 16 + ln.g) * per_row + 2 * u + (kq >> 1);
                    sc0 = __bfloat162float(s[0]); sc1 = __bfloat162float(s[8 * per_row]);
                }
                const uint32_t stage = wait_stage();
                if (valid) {
                    if (QA) adapter_stage_q<NT, MT>(acc, stage, m, kq, sc0, sc1, ln);
                    else adapter_stage<NT, MT>(acc, stage, m, kq, ln);
                }
                release();
            }
            // four partial sums per element: added up in shared memory and sent to the CTA that owns the column pair.
            // Element (token, column j) sits at token * 32 + (j ^ 8 * (token / 2 % 4)): conflict-free both ways.
            const int per = 16 >> logC;
#pragma unroll
            for (int n0 = 0; n0 < NT; n0 += kNW) {
                if (n0 > 0) consumer_sync();
#pragma unroll
                for (int n = 0; n < kNW; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        sts_f(part + (uint32_t)((kq * kNW * 8 + n * 8 + 2 * ln.t + (e & 1)) * kGroup + ((m * 16 + ln.g + 8 * (e >> 1)) ^ (8 * ln.t))) * 4, acc[n0 + n][e]);
                consumer_sync();
                if (n0 == 0) cluster_wait();
                for (int e = threadIdx.x; e < kNW * 8 * 16; e += kConsumers) {
                    const int tok = e >> 4, pr = e & 15;
                    const uint32_t at = part + (uint32_t)(tok * kGroup + ((2 * pr) ^ (8 * ((tok >> 1) & 3)))) * 4;
                    float2 s = lds_f2(at);
#pragma unroll
                    for (int w = 1; w < 4; ++w) {
                        const float2 v = lds_f2(at + w * kNW * 8 * kGroup * 4);
                        s.x += v.x; s.y += v.y;
                    }
                    const int gt = n0 * 8 + tok, owner = pr >> (4 - logC);
                    if (gt < p.b) {
                        const uint32_t dst = recv + (uint32_t)(((int)rank * p.b + gt) * per + (pr & (per - 1))) * 8;
                        st_peer2(peer(dst, owner), s.x, s.y, peer(piece_bar, owner));
                    }
                }
            }
        } else {
            const int rb = warp & 3, kk = warp >> 2;
            const int n_first = NT == 8 ? 4 * kk : 0;           // with eight n-tiles kk picks tokens, not columns
            const int row0 = tile * kRows + rb * 16 * MT;
            const int mts = max(0, min(MT, (p.d_out - row0) / 16));         // valid 16-row tiles of this warp
            float acc[MT][kNW][4];
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int n = 0; n < kNW; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[m][n][e] = 0.f;
            cluster_wait();                                    // every CTA has started (they all have by the time the first stage arrives)
            // ---------------- the weight
            for (int u = u0; u < u_end; ++u) {
                const uint32_t stage = wait_stage();
                if (mts > 0) {
                    const int left = p.d_in - u * kUnit;
                    if constexpr (FMT == FMT_TILED) {
                        weight_stage_tiled<NT>(acc, stage, rb, kk, ln);
                    } else if constexpr (NT == 8) {
#pragma unroll 1
                        for (int h = 0; h < 2; ++h) {
                            if (mts < MT || left < kUnit) complete_index<MT>(stage, rb, h, mts, left, ln);
                            weight_stage<NT, kNW, MT>(acc, stage, rb, h, n_first, ln);
                        }
                    } else {
                        if (mts < MT || left < kUnit) complete_index<MT>(stage, rb, kk, mts, left, ln);
                        weight_stage<NT, kNW, MT>(acc, stage, rb, kk, 0, ln);
                    }
                }
                release();
            }
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int n = 0; n < kNW; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[m][n][e] *= p.s;
            // ---------------- T L^T
            if constexpr (NT >= 4) {
                // T from shared memory.  With four n-tiles kk picks the step's MMA depth (bf16)
                int lt = 0;
                for (int lc = (int)rank; lc < l_chunks; lc += (int)C) {
                    const uint32_t stage = wait_stage();
                    if constexpr (QA) {
                        // codes: four n-tiles, kk picks the row tiles of both steps of the stage
                        float sc[8];
#pragma unroll
                        for (int m = 0; m < 8; ++m)
                            sc[m] = (m >> 1) < mts && (NT == 8 || (m >> 2) == kk) ? __bfloat162float(p.Ls[(size_t)(row0 + ln.g + 8 * m) * ((p.r + 127) >> 7) + (lc >> 1)]) : 0.f;
#pragma unroll 1
                        for (int ht = 0; ht < 2 * TP; ++ht, ++lt) {             // steps, T's parts inside them
                            const int h = ht / TP, ts = lt % C_::kTSlots;
                            const uint32_t tslot = part + ts * C_::kTSlot;
                            ok = mbar_wait(t_full + 8 * ts, (lt / C_::kTSlots) & 1, p.departures) && ok;
                            __syncwarp();
                            if (mts > 0 && 2 * lc + h < l_steps) {
                                uint4 tb[kNW];
#pragma unroll
                                for (int n = 0; n < kNW; ++n)
                                    tb[n] = pair_four_apart(lds128(tslot + ((n_first + n) * 8 + ln.g) * 64 + ((ln.t ^ ((ln.g >> 1) & 3)) << 4)));
#pragma unroll
                                for (int m = 0; m < 4; ++m)
                                    if (NT == 8 || (m >> 1) == kk) code_tile<kNW>(acc[m], l_codes<MT>(stage, rb, m, h, ln), sc[2 * m], sc[2 * m + 1], tb);
                            }
                            __syncwarp();
                            if (lane == 0) mbar_arrive(t_empty + 8 * ts);
                        }
                    } else
#pragma unroll 1
                    for (int tp = 0; tp < TP; ++tp, ++lt) {
                        const int ls = lc, ts = lt % C_::kTSlots;
                        const uint32_t tslot = part + ts * C_::kTSlot;
                        ok = mbar_wait(t_full + 8 * ts, (lt / C_::kTSlots) & 1, p.departures) && ok;
                        __syncwarp();
                        if (mts > 0) {
                            const int mat = lane >> 3, r8 = lane & 7;
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                if ((NT == 8 || h == kk) && ls * 32 + 16 * h < p.r) {
                                    uint4 tb[kNW / 2];              // two n-tiles of 8 tokens x two chunks of 8 columns
#pragma unroll
                                    for (int n = 0; n < kNW / 2; ++n)
                                        ldsm4(tslot + ((n_first + 2 * n + (mat >> 1)) * 8 + r8) * 64 + ((uint32_t)((2 * h + (mat & 1)) ^ ((r8 >> 1) & 3)) << 4), tb[n]);
#pragma unroll
                                    for (int m = 0; m < 4; ++m) {
                                        uint4 a;                    // 64-byte rows, 64-byte swizzle
                                        ldsm4(stage + (rb * 64 + m * 16 + (mat & 1) * 8 + r8) * 64 + ((uint32_t)((2 * h + (mat >> 1)) ^ ((r8 >> 1) & 3)) << 4), a);
#pragma unroll
                                        for (int n = 0; n < kNW / 2; ++n) {
                                            mma_16816(acc[m][2 * n], a.x, a.y, a.z, a.w, tb[n].x, tb[n].y);
                                            mma_16816(acc[m][2 * n + 1], a.x, a.y, a.z, a.w, tb[n].z, tb[n].w);
                                        }
                                    }
                                }
                            }
                        }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(t_empty + 8 * ts);
                    }
                    release();
                }
            } else if constexpr (!QA) {
                // kk picks the MMA depth of 16 of a 32-column step; the words of T (of both its parts) are asked for one step ahead
                constexpr int kWords = 2 * kNW;
                const int mat = lane >> 3, r8 = lane & 7;
                unsigned long long v[TP * kWords];
                auto word = [&](int ls, int q) {
                    const int n = q % kWords;
                    return p.T + (q / kWords) * t_tail + (size_t)((n >> 1) * 8 + ln.g) * (p.r / 2) + ls * 16 + 8 * kk + ln.t + 4 * (n & 1);
                };
                auto ask = [&](int ls) {
#pragma unroll
                    for (int q = 0; q < TP * kWords; ++q)
                        v[q] = (q % kWords >> 1) * 8 + ln.g < p.b && ls * 32 + 16 * kk < p.r ? ld_gpu64(word(ls, q)) : tagged(call, 0);
                };
                ask((int)rank);
                for (int ls = (int)rank; ls < l_steps; ls += (int)C) {
                    ok = wait_words(v, call, p.departures, [&] { ask(ls); }, [&](int q) { return word(ls, q); }) && ok;
                    uint32_t tb[TP * kWords];
#pragma unroll
                    for (int q = 0; q < TP * kWords; ++q) tb[q] = (uint32_t)v[q];
                    ask(ls + (int)C);
                    const uint32_t stage = wait_stage();
                    if (ls * 32 + 16 * kk < p.r && mts > 0) {
#pragma unroll
                        for (int m = 0; m < MT; ++m) {
                            uint4 a;                                // 64-byte rows, 64-byte swizzle
                            const int row = (rb * MT + m) * 16 + (mat & 1) * 8 + r8;
                            ldsm4(stage + row * 64 + ((uint32_t)((2 * kk + (mat >> 1)) ^ ((r8 >> 1) & 3)) << 4), a);
#pragma unroll
                            for (int tp = 0; tp < TP; ++tp)
#pragma unroll
                                for (int n = 0; n < kNW; ++n) mma_16816(acc[m][n], a.x, a.y, a.z, a.w, tb[tp * kWords + 2 * n], tb[tp * kWords + 2 * n + 1]);
                        }
                    }
                    release();
                }
            } else {
                // codes: kk picks the step of a stage of 64; scales and words of T are asked for one stage ahead, sixteen words after the
                // products of this one (with them in registers beside the products these spilled: 1728 -> 20480, 16 tokens 21.9 us, 19.2 so)
                constexpr int kWords = 4 * kNW;
                constexpr bool kAhead = TP * kWords <= 8;
                const uint32_t per_row = (uint32_t)((p.r + 127) >> 7);
                __nv_bfloat16 next[2 * MT];
                unsigned long long v[TP * kWords];
                auto word = [&](int ls, int q) {
                    const int n = q % kWords;
                    return p.T + (q / kWords) * t_tail + (size_t)((n >> 2) * 8 + ln.g) * (p.r / 2) + 4 * ln.t + 16 * ls + (n & 3);
                };
                auto ask = [&](int ls) {
#pragma unroll
                    for (int q = 0; q < TP * kWords; q += 2) {
                        v[q] = v[q + 1] = tagged(call, 0);
                        // r is a multiple of 16: a thread's 8 columns exist or not
                        if (ls * 32 + 8 * ln.t < p.r && (q % kWords >> 2) * 8 + ln.g < p.b) ld_gpu64x2(word(ls, q), v[q], v[q + 1]);
                    }
                };
                auto scales = [&](int lc) {
#pragma unroll
                    for (int m = 0; m < 2 * MT; ++m)                     // rows g + 8 m of the warp's
                        next[m] = lc < l_chunks && (m >> 1) < mts ? p.Ls[(size_t)(row0 + ln.g + 8 * m) * per_row + (lc >> 1)] : __ushort_as_bfloat16(0);
                };
                scales((int)rank);
                ask(2 * (int)rank + kk);
                for (int lc = (int)rank; lc < l_chunks; lc += (int)C) {
                    const int ls = 2 * lc + kk;
                    ok = wait_words(v, call, p.departures, [&] { ask(ls); }, [&](int q) { return word(ls, q); }) && ok;
                    uint4 tb[TP][kNW];
#pragma unroll
                    for (int q = 0; q < TP * kNW; ++q)
                        tb[q / kNW][q % kNW] = pair_four_apart(make_uint4((uint32_t)v[4 * q], (uint32_t)v[4 * q + 1], (uint32_t)v[4 * q + 2], (uint32_t)v[4 * q + 3]));
                    if (kAhead) ask(ls + 2 * (int)C);
                    float sc[2 * MT];
#pragma unroll
                    for (int m = 0; m < 2 * MT; ++m) sc[m] = __bfloat162float(next[m]);
                    scales(lc + (int)C);
                    const uint32_t stage = wait_stage();
                    if (ls < l_steps && mts > 0)
#pragma unroll
                        for (int m = 0; m < MT; ++m)
#pragma unroll
                            for (int tp = 0; tp < TP; ++tp) code_tile<kNW>(acc[m], l_codes<MT>(stage, rb, m, kk, ln), sc[2 * m], sc[2 * m + 1], tb[tp]);
                    release();
                    if (!kAhead) ask(ls + 2 * (int)C);
                }
            }
            // ---------------- partial tiles -> Y
            consumer_sync();                                   // every warp is done with the ring
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int n = 0; n < kNW; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        sts_f(smem + (uint32_t)(((NT == 8 ? 0 : kk * kTok) + (n_first + n) * 8 + 2 * ln.t + (e & 1)) * C_::kPitch + (rb * MT + m) * 16 + ln.g + 8 * (e >> 1)) * 4, acc[m][n][e]);
            consumer_sync();
            if (NT == 8) {                                     // the receivers' ring is free
                if (warp == 0 && lane < (int)C) mbar_arrive_peer(peer(gone, lane));
                ok = mbar_wait<true>(gone, 0, p.departures) && ok;
            }
            send<NT, MT>(p, smem, red_full, logC, (int)rank);
            ok = mbar_wait<true>(red_full, 0, p.departures) && ok;
            finish<NT, MT>(p, smem, tile, logC, (int)rank);
        }
    }
    if (!ok && lane == 0) flag_error(p.status, SLIM_ERR_TIMEOUT);
    __syncwarp();
    // nobody leaves while a peer may still read its shared memory (the reads are over: no memory ordering is asked for)
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    cluster_wait();
    if (threadIdx.x == 0) atomicAdd(p.departures, departure(blockIdx.x, gridDim.x));
}

// ------------------------------------------------------------------ host side
using KernelFn = void (*)(const SmallParams, const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap);

template <int NT, int FMT, int MT, int TP> KernelFn pick_q(bool qa) { return qa ? small_kernel<NT, FMT, true, MT, TP> : small_kernel<NT, FMT, false, MT, TP>; }
template <int NT, int FMT, int TP> KernelFn pick_m(int mt, bool qa) {
    return mt == 1 ? pick_q<NT, FMT, 1, TP>(qa) : mt == 2 ? pick_q<NT, FMT, 2, TP>(qa) : pick_q<NT, FMT, 4, TP>(qa);
}
template <int FMT, int TP> KernelFn pick_n(int nt, int mt, bool qa) {
    return nt == 1 ? pick_m<1, FMT, TP>(mt, qa) : nt == 2 ? pick_m<2, FMT, TP>(mt, qa) : nt == 4 ? pick_q<4, FMT, 4, TP>(qa) : pick_q<8, FMT, 4, TP>(qa);
}
// Rows of index bytes that no tensor map describes (FMT_PACKED_LD) belong to shapes whose T has two parts.
KernelFn pick(int nt, int fmt, bool qa, int mt, int tp) {
    if (fmt == FMT_TILED) return nt == 1 ? small_kernel<1, FMT_TILED, false, 4, 1> : small_kernel<2, FMT_TILED, false, 4, 1>;
    return fmt == FMT_PACKED_LD ? pick_n<FMT_PACKED_LD, 2>(nt, mt, qa) : tp == 2 ? pick_n<FMT_PACKED, 2>(nt, mt, qa) : pick_n<FMT_PACKED, 1>(nt, mt, qa);
}
int smem_bytes(int nt, int mt) {
    if (mt == 1) return nt == 1 ? Cfg<1, 1>::kSmem : Cfg<2, 1>::kSmem;
    if (mt == 2) return nt == 1 ? Cfg<1, 2>::kSmem : Cfg<2, 2>::kSmem;
    return nt == 1 ? Cfg<1, 4>::kSmem : nt == 2 ? Cfg<2, 4>::kSmem : nt == 4 ? Cfg<4, 4>::kSmem : Cfg<8, 4>::kSmem;
}
int threads_of(int nt) { return nt >= 4 ? Cfg<4, 4>::kThreads : Cfg<1, 4>::kThreads; }
int tiles_of(int b) { return b <= 8 ? 1 : b <= 16 ? 2 : b <= 32 ? 4 : 8; }

// Clusters of 1, 2, 4, 8 CTAs of one kernel that the device holds at once; asked once per device and kernel.
struct Residency { std::atomic<int> ready{0}; int clusters[4]; };
Residency g_res[64][4][3][2][3][2];
std::mutex g_res_mutex;

const int* residency(int dev, int nt, int fmt, bool qa, int mt, int tp) {
    const int ni = nt == 1 ? 0 : nt == 2 ? 1 : nt == 4 ? 2 : 3;
    Residency& rs = g_res[dev][ni][fmt][qa ? 1 : 0][mt >> 1][tp - 1];
    if (rs.ready.load(std::memory_order_acquire)) return rs.clusters;
    std::lock_guard<std::mutex> lock(g_res_mutex);
    if (rs.ready.load(std::memory_order_relaxed)) return rs.clusters;
    const void* fn = (const void*)pick(nt, fmt, qa, mt, tp);
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(nt, mt)) != cudaSuccess) return nullptr;
    for (int i = 0; i < 4; ++i) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1u << i); cfg.blockDim = dim3(threads_of(nt)); cfg.dynamicSmemBytes = smem_bytes(nt, mt);
        cudaLaunchAttribute a[1];
        a[0].id = cudaLaunchAttributeClusterDimension;
        a[0].val.clusterDim.x = 1u << i; a[0].val.clusterDim.y = 1; a[0].val.clusterDim.z = 1;
        cfg.attrs = a; cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
        rs.clusters[i] = n;
    }
    rs.ready.store(1, std::memory_order_release);
    return rs.clusters;
}

typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

bool make_map(CUtensorMap* map, const void* base, CUtensorMapDataType type, int esize, uint64_t cols, uint64_t rows,
              int box_cols, int box_rows, CUtensorMapSwizzle swz) {
    EncodeFn fn = reinterpret_cast<EncodeFn>(tensor_map_encoder());
    if (!fn) return false;
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {cols * (uint64_t)esize};
    cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, type, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
              CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// bf16 rows as 64-column sub-tiles: one box of box_rows rows x 4 sub-tiles of 128 bytes, in that order.
bool make_map3(CUtensorMap* map, const void* base, uint64_t cols, uint64_t rows, int box_rows) {
    EncodeFn fn = reinterpret_cast<EncodeFn>(tensor_map_encoder());
    if (!fn) return false;
    cuuint64_t dims[3] = {64, rows, cols / 64};
    cuuint64_t strides[2] = {cols * 2, 128};
    cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 4};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// CTAs per cluster: the most (up to 8, and no more than there are units) with which the clusters of all tiles fit the
// device at once, so that the stream of a tile is spread as widely as it can be; with more tiles than that, one.  (The clusters of T
// are not counted here, unlike for narrow tiles: they are done first and leave their places; 28672 -> 8192, 16 tokens has 464 CTAs on 296
// places this way.  Four CTAs a cluster, with which all would be resident, have not been measured.)
int cluster_size(const int* res, int tiles, int units) {
    for (int i = 3; i > 0; --i)
        if ((1 << i) <= units && tiles <= res[i]) return 1 << i;
    return 1;
}

// Up to 16 tokens, tiles of 128 rows where all clusters (tiles, and pieces of T) of four CTAs are then resident at once.  They
// have eight CTAs if there is no more than one CTA per SM even so: the words of T take 1-2 us longer to reach tiles that
// share their SMs with others and are done with the weight before T is there (2048 -> 2048, rank 208, 6 tokens:
// 23 clusters of four 4.8 us, of eight 6.8).  Tiles of 64 rows pay without adapters (4096 x 4096, 16 tokens: 5.1 us against 5.9)
// and for long rows that leave a CTA of a 128-row tile eight stages or more (8192 -> 3584, rank 368, 16 tokens: 9.9 us
// against 12.5), else not (4096 x 4096, rank 208: 9.1 us against 8.3).  With 256-row tiles only: 8192 -> 1024, rank 112, 16
// tokens 9.3 us instead of 6.6; 5120 x 5120, rank 512, 8 tokens 11.1 instead of 8.6; larger layers are better off with them
// (28672 -> 8192, 16 tokens 48 us against 65).
//   Without adapters clusters of two CTAs do (they start and exchange less) where rows are short and four would put more than a CTA on every SM.
// Clusters of four against two, us a call in a graph, weights in the L2 / from the HBM: tiles of 64 rows up to 8 units (1024 -> 4096, 16 tokens
// 3.07 / 3.08, 2.77 / 2.81; 2048 -> 4096 3.52 / 3.80, 3.37 / 3.72; but 4096 -> 4096, one token 3.89 / 4.75, 4.15 / 4.93; 2048 -> 2048, a CTA an SM
// either way, 2.62 / 2.65, 2.86 / 2.90), of 128 rows up to 20 (2304 -> 6784, 2 tokens 4.71 / 5.47, 4.11 / 5.06; 3072 -> 8192, one token 4.81 / 5.98,
// 4.63 / 5.62; 5120 -> 8192 6.05 / 7.63, 6.15 / 7.22).  And with them tiles of 128 rows fit more layers (16 tokens, 256 rows against 128: 5120 ->
// 13824 13.52 / 14.72, 12.23 / 13.14; 4096 -> 11008 10.69 / 12.20, 10.06 / 11.10; one token 7.64 / 9.16, 7.78 / 8.80).
void narrow_tiles(int dev, int nt, int fmt, bool qa, int tp, int sm_count, int d_out, int units, int groups, int* mt, int* C) {
    auto fits = [&](int m, int c) {
        const int* res = residency(dev, nt, fmt, qa, m, tp);
        return res && ceil_div(d_out, 64 * m) + groups <= res[c];
    };
    if (!fits(2, 2)) {
        if (groups == 0 && units >= 2 && fits(2, 1)) { *mt = 2; *C = 2; }
        return;
    }
    const bool spread = 8 * (ceil_div(d_out, 128) + groups) <= sm_count;
    *mt = fits(1, 2) && (groups == 0 || (!spread && units >= 32)) ? 1 : 2;
    const int widest = 8 * (ceil_div(d_out, 64 * *mt) + groups) <= sm_count ? 8 : 4;
    for (*C = widest; *C > units; *C /= 2) {}
    if (groups == 0 && *C == 4 && (*mt == 1 ? units <= 8 && 4 * ceil_div(d_out, 64) > sm_count : units <= 20 && d_out >= 6144)) *C = 2;
}

}  // namespace

// Limits of the kernel: the region of the workspace that T lives in (and r <= 3072), and the call counter, which
// takes 65536 CTAs.
bool small_supports(int b, int d_out, int d_in, int r) {
    return b >= 1 && b <= 64 && d_out >= 16 && d_out % 16 == 0 && d_in >= 64 && d_in % 64 == 0 && r >= 0 && r % 16 == 0 &&
           r <= kSmallMaxRank && (size_t)b * r * (keeps_T32(b, d_out, d_in, r) ? 8 : 4) <= kSmallTBytes && ceil_div(d_out, 256) < 32768;
}

slim_status_t launch_small(const __nv_bfloat16* X, int b, const uint8_t* vals, const uint8_t* meta, const uint8_t* tiled, float s,
                           const void* L, const void* R, const __nv_bfloat16* Ls, const __nv_bfloat16* Rs, int r, int d_out, int d_in,
                           __nv_bfloat16* Y, void* ws, uint32_t* status_dev, cudaStream_t st)
{
    slim_status_t err;
    const DeviceInfo* di = device_info(&err);
    if (!di) return err;
    if (!small_supports(b, d_out, d_in, r) || (tiled && (b > 16 || d_in % 256 != 0 || Ls))) return SLIM_ERR_UNSUPPORTED_SHAPE;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SLIM_ERR_CUDA;
    const int nt = tiles_of(b), fmt = tiled ? FMT_TILED : d_in % 128 == 0 ? FMT_PACKED : FMT_PACKED_LD;
    const bool qa = Ls != nullptr;
    const int tp = !tiled && (fmt == FMT_PACKED_LD || (r > 0 && keeps_T32(b, d_out, d_in, r))) ? 2 : 1;
    const int units = ceil_div(d_in, kUnit), groups = ceil_div(r, kGroup);
    int mt = 4, C = 0;
    if (nt <= 2 && !tiled) narrow_tiles(dev, nt, fmt, qa, tp, di->sm_count, d_out, units, groups, &mt, &C);
    const int rows = 64 * mt;
    const int* res = residency(dev, nt, fmt, qa, mt, tp);
    if (!res) return SLIM_ERR_CUDA;
    if (mt == 4) C = cluster_size(res, ceil_div(d_out, rows), units);
    SmallParams p;
    p.X = X; p.vals = vals; p.meta = meta; p.tiled = tiled; p.L = L; p.R = R; p.Ls = Ls; p.Rs = Rs; p.Y = Y;
    p.departures = reinterpret_cast<unsigned long long*>(ws);
    p.T = reinterpret_cast<unsigned long long*>(reinterpret_cast<char*>(ws) + SLIM_WORKSPACE_SYNC_BYTES);
    p.status = status_dev; p.s = s; p.b = b; p.r = r; p.d_out = d_out; p.d_in = d_in;
    // With adapters the HBM is idle for much of a call (start, hand-over of T, exchange), and the lines asked for ahead come for little: us a call
    // in a graph, weights in the L2 / from the HBM, without and with them: 4096 x 4096, rank 416, one token 6.82 / 7.92, 6.81 / 7.37; 4096 ->
    // 11008, rank 416 10.23 / 11.79, 10.38 / 11.14; 3584 -> 8192, rank 368, 4 tokens 10.95 / 12.68, 11.08 / 12.09; over 200 such calls 0.7 % more from
    // the L2, 3-4 % less from the HBM.  Not where that is not so: without adapters (4096 x 4096, one token 3.83 / 4.75, 4.46 / 4.81; 3072 -> 13824,
    // 16 tokens 8.14 / 9.44, 8.89 / 9.35), beside int4 adapters (4096 -> 11008, rank 416 10.54 / 12.36, 11.30 / 11.85), from 17 tokens on (8192 x 8192,
    // rank 832, 25 tokens 23.9, 25.3), under 2 MB of weight, beyond 40 MB (the HBM is busy throughout: 28672 -> 8192, 16 tokens 49, 53), and in CTAs
    // that find no place at first: those start in the middle of the call (3584 -> 8192 11.08 / 12.09 without them, 12.16 / 12.70).
    const size_t weight = (size_t)d_out * (size_t)d_in * 3 / 8;
    int log_c = 0;
    while ((2 << log_c) <= C) ++log_c;
    p.ahead = r > 0 && !qa && b <= 16 && weight >= (size_t)2 << 20 && weight <= (size_t)40 << 20 ? res[log_c] * C : 0;
    p.units = units; p.groups = groups;
    CUtensorMap tmV, tmM, tmX, tmR, tmL;
    bool ok = make_map3(&tmX, X, (uint64_t)d_in, (uint64_t)b, nt * 8);
    if (!tiled) ok = ok && make_map(&tmV, vals, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)d_in / 4, (uint64_t)d_out, 64, rows, CU_TENSOR_MAP_SWIZZLE_64B);
    else tmV = tmX;
    if (fmt == FMT_PACKED) ok = ok && make_map(&tmM, meta, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)d_in / 8, (uint64_t)d_out, 32, rows, CU_TENSOR_MAP_SWIZZLE_32B);
    else tmM = tmX;
    if (r > 0) ok = ok && (qa ? make_map(&tmR, R, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)d_in / 2, (uint64_t)r, 128, kGroup, CU_TENSOR_MAP_SWIZZLE_128B)
                              : make_map3(&tmR, R, (uint64_t)d_in, (uint64_t)r, kGroup));
    else tmR = tmX;
    if (r > 0 && !qa) ok = ok && make_map(&tmL, L, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)r, (uint64_t)d_out, 32, rows, CU_TENSOR_MAP_SWIZZLE_64B);
    else if (r > 0 && r % 32 == 0) ok = ok && make_map(&tmL, L, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)r / 2, (uint64_t)d_out, 32, rows, CU_TENSOR_MAP_SWIZZLE_32B);
    else tmL = tmX;
    if (!ok) return SLIM_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(C * (ceil_div(d_out, rows) + groups))); cfg.blockDim = dim3(threads_of(nt)); cfg.dynamicSmemBytes = smem_bytes(nt, mt); cfg.stream = st;
    cudaLaunchAttribute a[2];
    a[0].id = cudaLaunchAttributeClusterDimension;
    a[0].val.clusterDim.x = (unsigned)C; a[0].val.clusterDim.y = 1; a[0].val.clusterDim.z = 1;
    a[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = a; cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, pick(nt, fmt, qa, mt, tp), p, tmV, tmM, tmX, tmR, tmL);
    count_launch(1);
    return e == cudaSuccess ? SLIM_OK : SLIM_ERR_CUDA;
}

}  // namespace slim
