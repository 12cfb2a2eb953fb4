// SLiM-Quant: the per-tensor scale search and the quantization step (Sec. 3.1, Eq. 2-7, Algorithm 1;
// number of histogram bins: App. "Settings and Hyperparameters").  The steps and the precision of every
// decision are those include/slim.h states for slim_quant: the bin of a weight in binary32, the error
// of a candidate in binary64 with the bins added in ascending order and no fused multiply-add, the
// codes in binary32.  Four launches: largest magnitude, histogram, search, codes.
//
// (The weights themselves are complete before the first launch, which is no dependent one: they are read through the read-only path;
// what the launches hand to one another is not.)
//
// The three passes over the weights are bound by memory: 16-byte loads, and the histogram walks the array backwards,
// so that it starts with what the largest-magnitude pass left in the L2 (the codes pass, forwards again, finds the
// histogram's end there).  Measured on 4096 x 11008 (180 MB): see the figure at each kernel.
#include <atomic>
#include "common.cuh"

namespace slim {

namespace {

constexpr int kQsTable = 29;          // candidates: ten coarse, nineteen fine

struct QsHeader {                     // first 256 bytes of the workspace
    unsigned int max_bits;            // bit pattern of the largest |w| (non-negative floats order like unsigned integers)
    unsigned int bad;                 // a NaN or an infinity was seen
    unsigned int done;                // blocks of the search that have finished
};

constexpr int kVec = 4;               // float4 loads a thread has in flight

// The array as float4s i = first, first + stride, ..: kVec loads at a time (AHEAD: asked for while `f` works on those before), then `f` on each.  `tail` elements (n % 4)
// go to the first threads.
template <bool BACKWARDS, bool AHEAD, typename F>
__device__ __forceinline__ void for_weights(const float* __restrict__ W, size_t n, F f)
{
    const size_t n4 = n / 4, stride = (size_t)gridDim.x * blockDim.x, me = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const float4* W4 = reinterpret_cast<const float4*>(W);
    size_t i = me;
    float4 v[kVec];
    auto load = [&](float4 (&to)[kVec]) {
#pragma unroll
        for (int k = 0; k < kVec; ++k) to[k] = __ldg(W4 + (BACKWARDS ? n4 - 1 - (i + k * stride) : i + k * stride));
    };
    auto use = [&] {
#pragma unroll
        for (int k = 0; k < kVec; ++k) { f(v[k].x); f(v[k].y); f(v[k].z); f(v[k].w); }
    };
    if constexpr (AHEAD) {
        float4 w[kVec];
        bool some = i + (kVec - 1) * stride < n4;
        if (some) load(v);
        while (some) {
            i += kVec * stride;
            some = i + (kVec - 1) * stride < n4;
            if (some) load(w);
            use();
#pragma unroll
            for (int k = 0; k < kVec; ++k) v[k] = w[k];
        }
    } else {
        for (; i + (kVec - 1) * stride < n4; i += kVec * stride) { load(v); use(); }
    }
    for (; i < n4; i += stride) {
        const float4 v = __ldg(W4 + (BACKWARDS ? n4 - 1 - i : i));
        f(v.x); f(v.y); f(v.z); f(v.w);
    }
    if (me < n - 4 * n4) f(W[4 * n4 + me]);
}

__global__ void __launch_bounds__(512)
qs_absmax_kernel(const float* __restrict__ W, size_t n, QsHeader* hdr)
{
    __shared__ unsigned int sm[16], sb[16];
    after_previous_grid();
    unsigned int m = 0, bad = 0;
    for_weights<false, false>(W, n, [&](float w) {
        const float a = fabsf(w);
        if (!(a <= 3.0e38f)) bad = 1;
        m = max(m, __float_as_uint(a));
    });
    m = __reduce_max_sync(0xffffffffu, m);
    bad = __reduce_or_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0) { sm[threadIdx.x >> 5] = m; sb[threadIdx.x >> 5] = bad; }
    __syncthreads();
    if (threadIdx.x < 16) {
        m = __reduce_max_sync(0xffffu, sm[threadIdx.x]);
        bad = __reduce_or_sync(0xffffu, sb[threadIdx.x]);
        if (threadIdx.x == 0) {
            if (bad) atomicOr(&hdr->bad, 1u);
            else atomicMax(&hdr->max_bits, m);
        }
    }
}

// Histogram of |w| / M over `bins` uniform bins, per block in shared memory, then added to the global one.
__global__ void __launch_bounds__(1024)
qs_hist_kernel(const float* __restrict__ W, size_t n, const QsHeader* hdr, int bins, unsigned int* hist)
{
    extern __shared__ unsigned int sh[];
    for (int i = threadIdx.x; i < bins; i += blockDim.x) sh[i] = 0;
    after_previous_grid();
    __syncthreads();
    const float M = __uint_as_float(hdr->max_bits);
    if (M > 0.f && !hdr->bad) {
        const float fb = (float)bins;
        const Divisor by(M);
        for_weights<true, true>(W, n, [&](float w) { atomicAdd(&sh[min((int)__fmul_rn(by.of(fabsf(w)), fb), bins - 1)], 1u); });
    }
    __syncthreads();
    for (int i = threadIdx.x; i < bins; i += blockDim.x)
        if (sh[i]) atomicAdd(&hist[i], sh[i]);
}

// ---------------------------------------------------------------- E(alpha) on the bin centres
// The error is defined as a sum taken bin by bin, each addition rounded: a chain of 20000 dependent additions for each
// of the 29 candidates.  Two observations shorten it without changing a bit.
//   - While the sum e stays in one binade [2^k, 2^(k+1)), whose spacing is u, adding t >= 0 gives e + q with q = t
//     rounded to a multiple of u, unless t lies exactly half-way between two multiples (then the parity of e
//     decides).  The q of many bins can be found side by side and added in any order: all are multiples of u
//     and the sums stay below 2^53 u, so every addition is exact.  Sixteen warps work out the terms of a block of 256 bins
//     each; a lane guesses from an ordinary sum of the terms before it which binade e will be in at its eight bins, and
//     adds up their q.  Lanes where e seems to leave its binade, or that hold a half-way case, are "crossings": between them
//     the warp adds up the lanes' sums.  Then e walks over the blocks: a segment's sum, a crossing's eight terms one by one, and
//     so on; where a guess proves wrong, the block is gone through by parts (add_block).
//   - The fine candidates depend on the best coarse one only through ten possible values: all 10 + 10 x 19
//     candidates are evaluated at once, a block each, and the last block to finish takes the minima.
// Bound by the walk of one warp over the blocks' sums, the first of them a term at a time (41 cycles each). A warp of its own walks
// over a round of blocks while the other sixteen work out the next: their guesses start from ordinary sums, not from the walk's result.
// 20000 bins: 400 us with a warp per candidate and the bins in sequence, 54 with one adding warp per candidate that every
// block of bins passed through, 39 with one of the sixteen warps walking between the rounds, now 36.
constexpr int kSearchWarps = 16, kTermThreads = 32 * kSearchWarps, kSearchThreads = kTermThreads + 32, kCoarse = 10, kFine = 19, kCandidates = kCoarse + kCoarse * kFine;

// x / b correctly rounded in binary64, for many x and one b: as Divisor does it in binary32.
struct Divisor64 {
    double b, y;
    bool plain;
    __device__ __forceinline__ explicit Divisor64(double d) : b(d) {
        y = __drcp_rn(d);
        const unsigned long long bits = (unsigned long long)__double_as_longlong(d);
        plain = (bits & 0xFFFFFFFFFFFFFull) == 0xFFFFFFFFFFFFFull || !(d >= 0x1p-300 && d <= 0x1p300);
    }
    __device__ __forceinline__ double of(double x) const {
        if (plain) return __ddiv_rn(x, b);
        double q = __dmul_rn(x, y);
        q = __fma_rn(__fma_rn(-q, b, x), y, q);
        return __fma_rn(__fma_rn(-q, b, x), y, q);
    }
};

// One bin's term: every operation rounded on its own; an empty bin adds +0, which changes nothing.
__device__ __forceinline__ double qs_term(unsigned int c, int i, double width, const Divisor64& by_n, const Divisor64& by_alpha)
{
    if (!c) return 0.0;
    // i + 1/2 and c as binary64 (2^52 + i and 2^52 + c less 2^52, exact), and below the nearest integer of a number up to 8:
    // one or two additions each instead of conversions, which have a quarter of the rate
    const double alpha = by_alpha.b, x = __dmul_rn(__dadd_rn(__hiloint2double(0x43300000, i), -(0x1p52 - 0.5)), width);
    const double p = by_n.of(__dadd_rn(__hiloint2double(0x43300000, (int)c), -0x1p52));
    double d;
    if (x <= alpha) {
        const double level = __dadd_rn(__dadd_rn(by_alpha.of(__dmul_rn(x, 8.0)), 0x1.8p52), -0x1.8p52);
        d = __dsub_rn(__dmul_rn(__dmul_rn(alpha, 0.125), level), x);
    } else {
        d = __dsub_rn(alpha, x);
    }
    return __dmul_rn(p, __dmul_rn(d, d));
}

__device__ __forceinline__ int exponent(double e) { return (int)((__double_as_longlong(e) >> 52) & 0x7FF); }
// The binade of e > 2^-900: its end, half its start (terms below that are rounded by adding `magic`), half its spacing.
struct Binade {
    double end, half, magic, tie;
    int k;                                                    // biased exponent
    bool valid;
    __device__ __forceinline__ explicit Binade(double e) {
        k = exponent(e);
        valid = k > 123 && k < 2000;
        end = __longlong_as_double((long long)(k + 1) << 52);
        half = __longlong_as_double((long long)(valid ? k - 1 : 1) << 52);
        magic = __longlong_as_double(((long long)k << 52) | (1ll << 51));
        tie = __longlong_as_double((long long)(valid ? k - 53 : 1) << 52);
    }
    // t as a multiple of the spacing; *bad: t is too large for that, or half-way
    __device__ __forceinline__ double round(double t, bool* bad) const {
        const double q = __dsub_rn(__dadd_rn(t, magic), magic);
        *bad = !(t < half) || fabs(__dsub_rn(t, q)) == tie;
        return q;
    }
};

// The terms of 256 bins in shared memory: lane l has bins 8 l .. 8 l + 7 (pitch: no bank conflicts either way).
constexpr int kPitch = 36, kBlockTerms = 8 * kPitch;
__host__ __device__ __forceinline__ constexpr int term_at(int i) { return (i & 7) * kPitch + (i >> 3); }

constexpr size_t kSearchSmem = 2 * kSearchWarps * kBlockTerms * sizeof(double);
constexpr int kCross = 3;                                     // crossings of a block that are walked one by one
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ void named_sync(int id, int threads) { asm volatile("bar.sync %0, %1;" :: "r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void named_arrive(int id, int threads) { asm volatile("bar.arrive %0, %1;" :: "r"(id), "r"(threads) : "memory"); }

// e + the first 256 terms, one by one (every lane does it).  They grow from nothing: e leaves a binade every few of them.
__device__ double add_first(double e, const double* terms)
{
#pragma unroll 32
    for (int i = 0; i < 256; ++i) e = __dadd_rn(e, terms[term_at(i)]);
    return e;
}

// e + 256 terms in order.
__device__ double add_block(double e, const double* terms, int lane)
{
    double t[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) t[j] = terms[j * kPitch + lane];
    int at = 0;                                               // the terms of lanes before `at` are in e
    while (at < 32) {
        const Binade bn(e);
        bool bad = !bn.valid, b1;
        double q[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) { q[j] = bn.round(t[j], &b1); bad |= b1; }
        double s = __dadd_rn(__dadd_rn(__dadd_rn(q[0], q[1]), __dadd_rn(q[2], q[3])), __dadd_rn(__dadd_rn(q[4], q[5]), __dadd_rn(q[6], q[7])));
        if (lane < at) s = 0.0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double v = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s = __dadd_rn(s, v);
        }
        const double after = __dadd_rn(e, s);
        const unsigned stop = __ballot_sync(0xffffffffu, lane >= at && (bad || !(after < bn.end)));
        if (!stop) return __shfl_sync(0xffffffffu, after, 31);
        const int f = __ffs(stop) - 1;                        // this lane's eight terms go one by one
        const double before = __shfl_sync(0xffffffffu, after, f > 0 ? f - 1 : 0);
        if (f > at) e = before;
#pragma unroll
        for (int j = 0; j < 8; ++j) e = __dadd_rn(e, terms[j * kPitch + f]);
        at = f + 1;
    }
    return e;
}

__global__ void __launch_bounds__(kSearchThreads, 2)
qs_search_kernel(QsHeader* hdr, const unsigned int* hist, int bins, double n_total, float* scale_alpha, double* table,
                 double* errors, uint32_t* status)
{
    extern __shared__ double all_terms[];                     // of two rounds: [2][kSearchWarps][kBlockTerms]
    __shared__ double plain_sum[2][kSearchWarps], seg_sum[2][kSearchWarps][kCross + 1];
    __shared__ int seg_k[2][kSearchWarps][kCross + 1];        // a segment's binade, -1: it is empty
    __shared__ uint32_t crossings[2][kSearchWarps];           // lanes
    __shared__ bool last;
    after_previous_grid();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float Mf = __uint_as_float(hdr->max_bits);
    if (hdr->bad || !(Mf > 0.f)) {
        if (blockIdx.x != 0) return;
        if (threadIdx.x == 0) {
            scale_alpha[0] = 0.f; scale_alpha[1] = 0.f;
            if (hdr->bad) flag_error(status, SLIM_ERR_INVALID_ARG);
        }
        for (int i = threadIdx.x; i < 2 * kQsTable + 1; i += blockDim.x) table[i] = 0.0;
        return;
    }
    const double M = (double)Mf, eta_low = __ddiv_rn(M, 10.0), eta_high = __ddiv_rn(eta_low, 10.0);
    auto coarse = [&](int k) { return __ddiv_rn(__dmul_rn(M, (double)(k + 1)), 10.0); };
    auto fine = [&](int k, int j) {
        const double a = __dadd_rn(__dsub_rn(coarse(k), eta_low), __dmul_rn((double)(j + 1), eta_high));
        return a > M ? M : a;
    };
    const int cand = blockIdx.x;
    const double alpha = cand < kCoarse ? coarse(cand) : fine((cand - kCoarse) / kFine, (cand - kCoarse) % kFine);
    const double width = __ddiv_rn(M, (double)bins);
    double e = alpha > 0.0 ? 0.0 : -1.0;
    const int blocks = ceil_div(bins, 256), rounds = alpha > 0.0 ? ceil_div(blocks, kSearchWarps) : 0;
    auto round_terms = [&](int buf, int w) { return all_terms + (buf * kSearchWarps + w) * kBlockTerms; };
    if (warp < kSearchWarps) {
        const Divisor64 by_n(n_total), by_alpha(alpha);
        double sum_before = 0.0;                              // of the rounds before, an ordinary sum: for the guesses
        for (int r = 0; r < rounds; ++r) {
            const int buf = r & 1, first = r * kSearchWarps;
            double* terms = round_terms(buf, warp);
            const int i0 = (first + warp) * 256 + lane * 8;
            unsigned int c[8];
            if (i0 + 8 <= bins) {
                const uint4 lo = reinterpret_cast<const uint4*>(hist + i0)[0], hi = reinterpret_cast<const uint4*>(hist + i0)[1];
                c[0] = lo.x; c[1] = lo.y; c[2] = lo.z; c[3] = lo.w; c[4] = hi.x; c[5] = hi.y; c[6] = hi.z; c[7] = hi.w;
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) c[j] = i0 + j < bins ? hist[i0 + j] : 0u;
            }
            if (r >= 2) named_sync(4 + buf, kSearchThreads);  // the walk is done with this half of the buffers
            double v[8], sum = 0.0;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                v[j] = qs_term(c[j], i0 + j, width, by_n, by_alpha);
                terms[j * kPitch + lane] = v[j];
                sum = __dadd_rn(sum, v[j]);
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const double w = __shfl_up_sync(0xffffffffu, sum, o);
                if (lane >= o) sum = __dadd_rn(sum, w);
            }
            if (lane == 31) plain_sum[buf][warp] = sum;
            named_sync(1, kTermThreads);
            // guesses: e at the first of this lane's bins and after the last (the next lane's first)
            const double plain = lane < kSearchWarps ? plain_sum[buf][lane] : 0.0;
            const double before = __dadd_rn(sum_before, warp_sum(lane < warp ? plain : 0.0)), end = __dadd_rn(before, sum);
            sum_before = __dadd_rn(sum_before, warp_sum(plain));
            double start = __shfl_up_sync(0xffffffffu, end, 1);
            if (lane == 0) start = before;
            const Binade bn(start);
            bool bad = !bn.valid || exponent(end) != bn.k, b1;
            double q = 0.0;
#pragma unroll
            for (int j = 0; j < 8; ++j) { q = __dadd_rn(q, bn.round(v[j], &b1)); bad |= b1; }
            const uint32_t cross = __ballot_sync(0xffffffffu, bad);
            const int n_cross = __popc(cross), segment = bad ? -1 : __popc(cross & ((1u << lane) - 1));
            for (int i = 0; i <= min(n_cross, kCross); ++i) {
                const uint32_t in = __ballot_sync(0xffffffffu, segment == i);
                const double s = warp_sum(segment == i ? q : 0.0);
                const int k = __shfl_sync(0xffffffffu, bn.k, in ? __ffs(in) - 1 : 0);
                if (lane == 0) { seg_sum[buf][warp][i] = s; seg_k[buf][warp][i] = in ? k : -1; }
            }
            if (lane == 0) crossings[buf][warp] = cross;
            named_arrive(2 + buf, kSearchThreads);
        }
    } else {
        for (int r = 0; r < rounds; ++r) {
            const int buf = r & 1, first = r * kSearchWarps, n = min(kSearchWarps, blocks - first);
            named_sync(2 + buf, kSearchThreads);
            int b = 0;
            if (first == 0) { e = add_first(e, round_terms(0, 0)); b = 1; }
            const uint32_t cross_l = lane < n ? crossings[buf][lane] : 1u;
            const double s_l = lane < n ? seg_sum[buf][lane][0] : 0.0;
            const int k_l = cross_l == 0 ? seg_k[buf][lane][0] : -1;
            for (; b < n; ++b) {
                // blocks from b on without a crossing, as far as e stays in its binade
                double after = lane >= b ? s_l : 0.0;
#pragma unroll
                for (int o = 1; o < kSearchWarps; o <<= 1) {
                    const double w = __shfl_up_sync(0xffffffffu, after, o);
                    if (lane >= o) after = __dadd_rn(after, w);
                }
                after = __dadd_rn(e, after);
                const uint32_t stop = __ballot_sync(0xffffffffu, lane >= b && !(k_l == exponent(e) && exponent(after) == k_l));
                const int upto = __ffs(stop) - 1;             // lane n at the latest
                if (upto > b) { e = __shfl_sync(0xffffffffu, after, upto - 1); b = upto; }
                if (b >= n) break;
                const double* terms = round_terms(buf, b);
                uint32_t left = crossings[buf][b];
                const int nc = __popc(left);
                bool good = nc <= kCross;
                double f = e;
                for (int i = 0; good; ++i) {
                    const int k = seg_k[buf][b][i];
                    if (k >= 0) {
                        const double to = __dadd_rn(f, seg_sum[buf][b][i]);
                        good = exponent(f) == k && exponent(to) == k;
                        f = to;
                    }
                    if (i == nc) break;
                    const int l = __ffs(left) - 1;
                    left &= left - 1;
#pragma unroll
                    for (int j = 0; j < 8; ++j) f = __dadd_rn(f, terms[j * kPitch + l]);
                }
                e = good ? f : add_block(e, terms, lane);
            }
            if (r + 2 < rounds) named_arrive(4 + buf, kSearchThreads);
        }
    }
    if (threadIdx.x == kTermThreads) {
        errors[cand] = e;
        __threadfence();
        last = atomicAdd(&hdr->done, 1u) == gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    if (!last) return;
    // the minima, in the order the algorithm visits the candidates (one thread; the errors are fetched by all, since one
    // after the other they took 15 us)
    double* er = all_terms;
    for (int i = threadIdx.x; i < kCandidates; i += kSearchThreads) er[i] = __ldcg(errors + i);
    __syncthreads();
    if (threadIdx.x != 0) return;
    int best = 0;
    for (int k = 1; k < kCoarse; ++k) if (er[k] < er[best]) best = k;
    double best_a = coarse(best), best_e = er[best];
    for (int k = 0; k < kCoarse; ++k) { table[2 * k] = coarse(k); table[2 * k + 1] = er[k]; }
    for (int j = 0; j < kFine; ++j) {
        const double a = fine(best, j);
        double ej = er[kCoarse + best * kFine + j];
        if (!(a > 0.0)) ej = __dadd_rn(best_e, 1.0);                              // not a candidate; listed like this
        else if (ej < best_e || (ej == best_e && a < best_a)) { best_a = a; best_e = ej; }
        table[2 * (kCoarse + j)] = a; table[2 * (kCoarse + j) + 1] = ej;
    }
    const float a32 = (float)best_a;
    scale_alpha[0] = __fmul_rn(a32, 0.125f);
    scale_alpha[1] = a32;
    table[2 * kQsTable] = best_a;
}

// Four float4 loads of a thread under way, a warp's side by side (512 bytes; four neighbouring ones a thread, for a 16-byte store, touch
// sixteen lines a load), four codes stored together.
__global__ void __launch_bounds__(256)
qs_codes_kernel(const float* __restrict__ W, size_t n, const float* scale_alpha, int8_t* codes)
{
    after_previous_grid();
    const float a32 = scale_alpha[1];
    const Divisor by(a32 > 0.f ? a32 : 1.f);
    auto code = [&](float w) -> uint32_t {
        return a32 > 0.f ? (uint32_t)max(-8, min(7, __float2int_rn(__fmul_rn(by.of(w), 8.0f)))) & 0xFFu : 0u;
    };
    const size_t n4 = n / 4;
    for (size_t i = (size_t)blockIdx.x * 1024 + threadIdx.x; i < n4; i += (size_t)gridDim.x * 1024) {
        float4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) if (i + k * 256 < n4) v[k] = __ldg(reinterpret_cast<const float4*>(W) + i + k * 256);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i + k * 256 < n4) reinterpret_cast<uint32_t*>(codes)[i + k * 256] = code(v[k].x) | code(v[k].y) << 8 | code(v[k].z) << 16 | code(v[k].w) << 24;
    }
    const size_t me = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (me < n - 4 * n4) codes[4 * n4 + me] = (int8_t)code(W[4 * n4 + me]);
}

}  // namespace

int quant_bins(int d_out, int d_in) {
    long long b = (long long)d_out * (long long)d_in / 1000;
    if (b > 20000) b = 20000;
    if (b < 512) b = 512;
    return (int)b;
}

size_t quant_workspace_bytes(int d_out, int d_in) {
    return 256 + (size_t)quant_bins(d_out, d_in) * 4 + 256 + (2 * kQsTable + 1 + kCandidates) * sizeof(double);
}

slim_status_t launch_quant(const float* W, int d_out, int d_in, int8_t* codes, float* scale_alpha, void* ws,
                           uint32_t* status_dev, cudaStream_t st)
{
    slim_status_t err;
    const DeviceInfo* di = device_info(&err);
    if (!di) return err;
    const size_t n = (size_t)d_out * (size_t)d_in;
    const int bins = quant_bins(d_out, d_in);
    char* base = static_cast<char*>(ws);
    QsHeader* hdr = reinterpret_cast<QsHeader*>(base);
    unsigned int* hist = reinterpret_cast<unsigned int*>(base + 256);
    double* table = reinterpret_cast<double*>(base + 256 + ((size_t)bins * 4 + 255) / 256 * 256);
    if (cudaMemsetAsync(ws, 0, 256 + (size_t)bins * 4, st) != cudaSuccess) return SLIM_ERR_CUDA;
    qs_absmax_kernel<<<(unsigned)(di->sm_count * 4), 512, 0, st>>>(W, n, hdr);
    const size_t hist_smem = (size_t)bins * 4;
    int dev = 0;
    cudaGetDevice(&dev);
    static std::atomic<bool> attr_set[64];
    if (dev < 0 || dev >= 64) return SLIM_ERR_CUDA;
    if (!attr_set[dev].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(qs_hist_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 20000 * 4) != cudaSuccess ||
            cudaFuncSetAttribute(qs_search_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSearchSmem) != cudaSuccess) return SLIM_ERR_CUDA;
        attr_set[dev].store(true, std::memory_order_release);
    }
    // a block per SM: two would find no more work in flight and double the additions to the global histogram
    launch_dependent(qs_hist_kernel, dim3((unsigned)di->sm_count), dim3(1024), hist_smem, st, W, n, hdr, bins, hist);
    launch_dependent(qs_search_kernel, dim3(kCandidates), dim3(kSearchThreads), kSearchSmem, st, hdr, hist, bins, (double)n, scale_alpha, table,
                     table + 2 * kQsTable + 1, status_dev);
    launch_dependent(qs_codes_kernel, dim3((unsigned)(di->sm_count * 8)), dim3(256), 0, st, W, n, scale_alpha, codes);
    count_launch(4);
    return cudaGetLastError() == cudaSuccess ? SLIM_OK : SLIM_ERR_CUDA;
}

}  // namespace slim
