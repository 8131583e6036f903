// Gamma builder: per-block importance and selection of the n_zero lowest blocks.
// Eq. (1), Eq. (2) and Section "Predetermined Sparsity ratio and Full Training Ahead" of the paper.
#include <type_traits>
#include "bsp_internal.cuh"
#include "bsp_span.cuh"

namespace bsp {
namespace {

constexpr int kScoreThreads = 256;
constexpr int kRankThreads = 512;        // of the kernels that score and select in one launch
constexpr int kSelectThreads = 1024;

// One 4-byte word of W holds 1 fp32, 2 bf16 or 4 int8 values, lowest channel in the lowest bytes.
template <int DT> struct Acc;
template <> struct Acc<BSP_F32> { using type = double; };
template <> struct Acc<BSP_BF16> { using type = double; };
template <> struct Acc<BSP_I8> { using type = long long; };

// Measures of one weight: BSP_NORM_L2 (w^2), BSP_NORM_L1 (|w|), and for the variance two passes over the block:
// kNormSum (w, for the block mean) and BSP_NORM_VAR ((w - mean)^2, with the subtraction, the product and the addition
// each rounded on its own, never fused: the float64 result must not depend on what the compiler contracts).
constexpr int kNormSum = 3;

template <int NORM>
__device__ __forceinline__ void add_value(double v, double &acc, double mean)
{
    if constexpr (NORM == BSP_NORM_L2) acc += v * v;
    else if constexpr (NORM == BSP_NORM_L1) acc += fabs(v);
    else if constexpr (NORM == kNormSum) acc += v;
    else { const double d = __dsub_rn(v, mean); acc = __dadd_rn(acc, __dmul_rn(d, d)); }
}

template <int DT, int NORM>
__device__ __forceinline__ void add_word(uint32_t w, typename Acc<DT>::type &acc, double mean)
{
    if constexpr (DT == BSP_F32) {
        add_value<NORM>((double)__uint_as_float(w), acc, mean);
    } else if constexpr (DT == BSP_BF16) {
        add_value<NORM>((double)__uint_as_float(w << 16), acc, mean);
        add_value<NORM>((double)__uint_as_float(w & 0xFFFF0000u), acc, mean);
    } else {
        // (four exact products at once; one at a time in 64 bits the integer unit bounded large layers)
        if constexpr (NORM == BSP_NORM_L2) acc += (long long)__dp4a((int)w, (int)w, 0);
        else acc += (long long)__dp4a(__vabs4(w), 0x01010101u, 0u);      // (|-128| is 128 as an unsigned byte)
    }
}

// One thread sums one output row r of one block over (h, k, c) in that order; the thread with r = 0 then
// adds the b_o row sums in order of r.  The order is part of the definition of the float score: it makes
// the float64 result, and so Gamma, independent of the launch shape.  (Each square of a float or bf16 value
// is exact in float64, so a fused multiply-add rounds like a multiply followed by an add.)
// Threads are laid out with consecutive blocks of one block row on consecutive lanes, so that for a fixed
// (r, h, k) a warp reads one contiguous stretch of input channels.
// Sum of one output row r of block B over (h, k, c) in that order, for a block of WORDS 32-bit words per tap.
// Loads of up to nine taps (a whole 3x3 kernel) are issued together, as 16-byte loads when `vec` says that the
// rows are 16-byte aligned; the adds keep the (h, k, c) order.
template <int DT, int NORM, int WORDS, int kBatch>
__device__ __forceinline__ typename Acc<DT>::type row_sum_w(const uint32_t *src, size_t row_words, int HK, bool vec,
                                                            double mean)
{
    using acc_t = typename Acc<DT>::type;
    acc_t pr = 0;
    for (int t = 0; t < HK; t += kBatch) {
        uint32_t w[kBatch][WORDS];
        if constexpr (WORDS % 4 == 0) {
            if (vec) {
#pragma unroll
                for (int u = 0; u < kBatch; ++u)
#pragma unroll
                    for (int j = 0; j < WORDS; j += 4)
                        if (t + u < HK) {
                            const uint4 q = load_free((const uint4 *)(src + (size_t)u * row_words + j));
                            w[u][j] = q.x; w[u][j + 1] = q.y; w[u][j + 2] = q.z; w[u][j + 3] = q.w;
                        }
            } else {
#pragma unroll
                for (int u = 0; u < kBatch; ++u)
#pragma unroll
                    for (int j = 0; j < WORDS; ++j)
                        if (t + u < HK) w[u][j] = load_free(src + (size_t)u * row_words + j);
            }
        } else {
#pragma unroll
            for (int u = 0; u < kBatch; ++u)
#pragma unroll
                for (int j = 0; j < WORDS; ++j)
                    if (t + u < HK) w[u][j] = load_free(src + (size_t)u * row_words + j);
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u)
#pragma unroll
            for (int j = 0; j < WORDS; ++j)
                if (t + u < HK) add_word<DT, NORM>(w[u][j], pr, mean);
        src += (size_t)kBatch * row_words;
    }
    return pr;
}

// kBatch = taps whose loads are in flight together: 9 (a 3x3 kernel at once), or 1 in the kernels compiled for
// one-tap layers, which then need few registers and keep many CTAs resident.
template <int DT, int NORM, int kBatch>
__device__ __forceinline__ typename Acc<DT>::type row_sum(const uint32_t *W, int I, int HK, int bo, int bi,
                                                          int NBi, long long B, int r, double mean = 0.0)
{
    constexpr int per_word = (DT == BSP_F32) ? 1 : (DT == BSP_BF16 ? 2 : 4);
    const int l = B < (1ll << 31) ? (int)((unsigned)B / (unsigned)NBi) : (int)(B / NBi);     // (64-bit divisions are slow)
    const int iota = (int)(B - (long long)l * NBi);
    const int words = bi / per_word;
    const size_t row_words = (size_t)I / per_word;
    const uint32_t *src = W + ((size_t)(l * bo + r) * HK) * row_words + (size_t)iota * words;
    const bool vec = (((uintptr_t)W) & 15u) == 0 && row_words % 4 == 0;
    // (rows of 8 and 16 words take fewer taps at a time: nine of 16 words did not fit the registers, and the spills made the
    // variance of a 512x512 3x3 layer cost 45 us)
    switch (words) {
        case 1: return row_sum_w<DT, NORM, 1, kBatch>(src, row_words, HK, vec, mean);
        case 2: return row_sum_w<DT, NORM, 2, kBatch>(src, row_words, HK, vec, mean);
        case 4: return row_sum_w<DT, NORM, 4, kBatch>(src, row_words, HK, vec, mean);
        case 8: return row_sum_w<DT, NORM, 8, (kBatch > 4 ? 4 : kBatch)>(src, row_words, HK, vec, mean);
        default: return row_sum_w<DT, NORM, 16, (kBatch > 2 ? 2 : kBatch)>(src, row_words, HK, vec, mean);
    }
}

// One-tap layers (H K = 1) with the L2 or L1 measure: one thread per block (consecutive threads take consecutive blocks of
// a block row, so a warp's load of one row r is one contiguous stretch of input channels).  The rows of a block are
// WORDS words each; kRows rows (eight, or four when b_o = 4 or the rows are long) are loaded at a time, every row is summed over its channels in order and the row sums
// are added in order of r: the same order of additions as row_sum followed by the sum over r.
template <int DT, int WORDS, int kRows>
__device__ __forceinline__ void one_tap_load(const uint32_t *W, int I, int bo, int NBi, long long B, int r0, uint32_t (&w)[kRows][WORDS])
{
    constexpr int per_word = (DT == BSP_F32) ? 1 : (DT == BSP_BF16 ? 2 : 4);
    constexpr int kVec = WORDS % 4 == 0 ? 4 : (WORDS % 2 == 0 ? 2 : 1);       // words per load
    const size_t row_words = (size_t)I / per_word;
    const bool vec = kVec > 1 && (((uintptr_t)W) & (4u * kVec - 1u)) == 0 && row_words % kVec == 0;
    // (a 64-bit division costs an order of magnitude more than a 32-bit one: taken only by blocks that need it)
    const int l = B < (1ll << 31) ? (int)((unsigned)B / (unsigned)NBi) : (int)(B / NBi);
    const int iota = (int)(B - (long long)l * NBi);
    const uint32_t *src = W + ((size_t)l * bo + r0) * row_words + (size_t)iota * WORDS;
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
        const uint32_t *row = src + (size_t)u * row_words;
        if (vec && kVec == 4) {
#pragma unroll
            for (int j = 0; j + 3 < WORDS; j += 4) {
                const uint4 q = load_free((const uint4 *)(row + j));
                w[u][j] = q.x; w[u][j + 1] = q.y; w[u][j + 2] = q.z; w[u][j + 3] = q.w;
            }
        } else if (vec && kVec == 2) {
#pragma unroll
            for (int j = 0; j + 1 < WORDS; j += 2) {
                const uint2 q = load_free((const uint2 *)(row + j));
                w[u][j] = q.x; w[u][j + 1] = q.y;
            }
        } else {
#pragma unroll
            for (int j = 0; j < WORDS; ++j) w[u][j] = load_free(row + j);
        }
    }
}
template <int DT, int NORM, int WORDS, int kRows>
__device__ __forceinline__ typename Acc<DT>::type one_tap_add(const uint32_t (&w)[kRows][WORDS], typename Acc<DT>::type total)
{
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
        typename Acc<DT>::type pr = 0;
#pragma unroll
        for (int j = 0; j < WORDS; ++j) add_word<DT, NORM>(w[u][j], pr, 0.0);
        total += pr;
    }
    return total;
}
// Calls f with the template arguments WORDS and kRows of the layer's block shape as integral constants.
template <int DT, typename F>
__device__ __forceinline__ void one_tap_form(int bo, int bi, F f)
{
    constexpr int per_word = (DT == BSP_F32) ? 1 : (DT == BSP_BF16 ? 2 : 4);
    using std::integral_constant;
    const bool eight = bo % 8 == 0;
    switch (bi / per_word) {
        case 1: if (eight) f(integral_constant<int, 1>(), integral_constant<int, 8>()); else f(integral_constant<int, 1>(), integral_constant<int, 4>()); break;
        case 2: if (eight) f(integral_constant<int, 2>(), integral_constant<int, 8>()); else f(integral_constant<int, 2>(), integral_constant<int, 4>()); break;
        case 4: if (eight) f(integral_constant<int, 4>(), integral_constant<int, 8>()); else f(integral_constant<int, 4>(), integral_constant<int, 4>()); break;
        case 8: f(integral_constant<int, 8>(), integral_constant<int, 4>()); break;
        default: f(integral_constant<int, 16>(), integral_constant<int, 4>()); break;
    }
}

// Score of block B by the b_o threads r = 0 .. b_o - 1 (thread r sums row r; `part` holds their row sums, those of one block
// `stride` apart at `bl`); valid in the thread with r = 0.  Every thread of the CTA must call it; `mine`: the thread has a row.
template <int DT, int NORM, int kBatch>
__device__ __forceinline__ typename Acc<DT>::type block_score(const uint32_t *W, int I, int HK, int bo, int bi, int NBi, long long B,
                                                              int r, bool mine, typename Acc<DT>::type *part, int bl, int stride)
{
    using acc_t = typename Acc<DT>::type;
    acc_t total = 0;
    if constexpr (NORM == BSP_NORM_VAR) {
        // variance about the block's own mean, n = b_o H K b_i entries: the mean from the row sums added in order of
        // r (every thread of the block adds them the same way), then the squared deviations in the same order, over n
        const double n_elems = (double)bo * HK * bi;
        part[threadIdx.x] = mine ? row_sum<DT, kNormSum, kBatch>(W, I, HK, bo, bi, NBi, B, r) : (acc_t)0;
        __syncthreads();
        double s = 0.0;
        if (mine)
            for (int q = 0; q < bo; ++q) s += (double)part[q * stride + bl];
        const double mean = s / n_elems;
        __syncthreads();
        part[threadIdx.x] = mine ? row_sum<DT, NORM, kBatch>(W, I, HK, bo, bi, NBi, B, r, mean) : (acc_t)0;
        __syncthreads();
        if (mine && r == 0) {
            double t = 0.0;
            for (int q = 0; q < bo; ++q) t += (double)part[q * stride + bl];
            total = (acc_t)(t / n_elems);
        }
    } else {
        part[threadIdx.x] = mine ? row_sum<DT, NORM, kBatch>(W, I, HK, bo, bi, NBi, B, r) : (acc_t)0;
        __syncthreads();
        if (mine && r == 0)
            for (int q = 0; q < bo; ++q) total += part[q * stride + bl];
    }
    return total;
}

// Scores of the blocks [lo, hi) by a CTA of kT threads, each handed to put(block, score); after_first() is called by every thread
// once the first round of blocks has been handed over (also where the range is empty).  One-tap layers take a thread per block,
// the others b_o threads per block, kT / b_o blocks a round, `step` rounds' worth of blocks apart.  `part`: kT row sums.
template <int DT, int NORM, int kBatch, int kT, typename P, typename A>
__device__ __forceinline__ void score_range(const uint32_t *W, int I, int HK, int bo, int bi, int NBi, long long lo, long long hi, int step,
                                            typename Acc<DT>::type *part, P put, A after_first)
{
    using acc_t = typename Acc<DT>::type;
    if constexpr (kBatch == 1 && NORM != BSP_NORM_VAR) {
        one_tap_form<DT>(bo, bi, [&](auto words, auto rows) {
            constexpr int kWords = decltype(words)::value, kRows = decltype(rows)::value;
            // (the next rows are on their way while these are summed: float64 arithmetic runs at 15 values a cycle and SM, and
            // waiting for either took 17 of the 33 us of a 4096 x 4096 layer)
            constexpr bool kAhead = kRows * kWords <= 32;    // (what the registers hold twice)
            uint32_t w[kRows][kWords], ahead[kAhead ? kRows : 1][kWords];
            const long long jump = (long long)step * kT;
            if (kAhead && lo + threadIdx.x < hi) one_tap_load<DT, kWords, kRows>(W, I, bo, NBi, lo + threadIdx.x, 0, w);
            for (long long B0 = lo; B0 < hi || B0 == lo; B0 += jump) {
                const long long B = B0 + threadIdx.x;
                acc_t total = 0;
                for (int r0 = 0; r0 < bo; r0 += kRows) {     // (b_o is a multiple of kRows)
                    if constexpr (kAhead) {
                        const bool more = r0 + kRows < bo;
                        const long long next = more ? B : B + jump;
                        if (next < hi) one_tap_load<DT, kWords, kRows>(W, I, bo, NBi, next, more ? r0 + kRows : 0, ahead);
                    } else if (B < hi) one_tap_load<DT, kWords, kRows>(W, I, bo, NBi, B, r0, w);
                    if (B < hi) total = one_tap_add<DT, NORM, kWords, kRows>(w, total);
                    if constexpr (kAhead) {
#pragma unroll
                        for (int u = 0; u < kRows; ++u)
#pragma unroll
                            for (int j = 0; j < kWords; ++j) w[u][j] = ahead[u][j];
                    }
                }
                if (B < hi) put(B, total);
                if (B0 == lo) after_first();
            }
        });
    } else {
        const int per = kT / bo, bl = threadIdx.x % per, r = threadIdx.x / per;
        for (long long B0 = lo; B0 < hi || B0 == lo; B0 += (long long)step * per) {
            const long long B = B0 + bl;
            const acc_t total = block_score<DT, NORM, kBatch>(W, I, HK, bo, bi, NBi, B, r, B < hi, part, bl, per);
            if (B < hi && r == 0) put(B, total);
            if (B0 == lo) after_first();
            __syncthreads();
        }
    }
}

// A bounded grid of long-lived CTAs, each taking every gridDim.x-th round of blocks.
template <int DT, int NORM, int kBatch>
__global__ void __launch_bounds__(kScoreThreads)
score_kernel(const uint32_t *W, int I, int HK, int bo, int bi, int NBo, int NBi, typename Acc<DT>::type *score)
{
    using acc_t = typename Acc<DT>::type;
    __shared__ acc_t part[kScoreThreads];
    const int per = kBatch == 1 && NORM != BSP_NORM_VAR ? kScoreThreads : kScoreThreads / bo;
    wait_for_previous<false>();
    score_range<DT, NORM, kBatch, kScoreThreads>(from_here(W), I, HK, bo, bi, NBi, (long long)blockIdx.x * per, (long long)NBo * NBi, (int)gridDim.x, part,
                                                 [&](long long B, acc_t total) { score[B] = total; }, []() {});
}

// Scores are non-negative, so the bit pattern of a float64 orders like the value, as does an int64.
// One CTA ranks one segment (the whole layer, or one row of Gamma): an 8-pass most-significant-digit
// radix select finds the key T of the n_zero-th smallest (key, index) pair and how many keys equal to T
// are still to be zeroed; a final pass in index order writes Gamma, zeroing the keys below T and the first
// `ties` keys equal to T.
__global__ void __launch_bounds__(kSelectThreads)
select_kernel(const unsigned long long *__restrict__ key, long long seg_len, long long n_zero,
              uint8_t *__restrict__ gamma)
{
    __shared__ unsigned int hist[256];
    __shared__ unsigned long long s_prefix;
    __shared__ long long s_k;
    __shared__ unsigned int warp_cnt[kSelectThreads / 32];
    __shared__ long long s_run;

    const unsigned long long *k = key + (size_t)blockIdx.x * seg_len;
    uint8_t *g = gamma + (size_t)blockIdx.x * seg_len;
    const int tid = threadIdx.x;

    if (n_zero <= 0 || n_zero >= seg_len) {
        const uint8_t v = (n_zero <= 0) ? 1 : 0;
        for (long long i = tid; i < seg_len; i += kSelectThreads) g[i] = v;
        return;
    }
    if (tid == 0) { s_prefix = 0ull; s_k = n_zero; }
    for (int pass = 7; pass >= 0; --pass) {
        if (tid < 256) hist[tid] = 0u;
        __syncthreads();
        const unsigned long long prefix = s_prefix;
        const int shift = 8 * pass;
        for (long long i = tid; i < seg_len; i += kSelectThreads) {
            const unsigned long long v = k[i];
            const bool in = (pass == 7) || ((v >> (shift + 8)) == prefix);
            if (in) atomicAdd(&hist[(unsigned)((v >> shift) & 0xFFull)], 1u);
        }
        __syncthreads();
        if (tid == 0) {
            long long need = s_k, cum = 0;
            int d = 0;
            for (; d < 255; ++d) {
                if (cum + (long long)hist[d] >= need) break;
                cum += hist[d];
            }
            s_k = need - cum;
            s_prefix = (prefix << 8) | (unsigned long long)d;
        }
        __syncthreads();
    }
    const unsigned long long T = s_prefix;
    const long long ties = s_k;        // keys equal to T to zero, lowest indices first
    if (tid == 0) s_run = 0;
    __syncthreads();
    const int lane = tid & 31, warp = tid >> 5;
    for (long long base = 0; base < seg_len; base += kSelectThreads) {
        const long long i = base + tid;
        unsigned long long v = ~0ull;
        if (i < seg_len) v = k[i];
        const bool eq = (i < seg_len) && (v == T);
        const unsigned ball = __ballot_sync(0xFFFFFFFFu, eq);
        if (lane == 0) warp_cnt[warp] = __popc(ball);
        __syncthreads();
        long long before = s_run;
        for (int w = 0; w < warp; ++w) before += warp_cnt[w];
        before += __popc(ball & ((1u << lane) - 1u));
        if (i < seg_len) g[i] = (v < T || (eq && before < ties)) ? 0 : 1;
        __syncthreads();
        if (tid == 0) {
            long long tot = 0;
            for (int w = 0; w < kSelectThreads / 32; ++w) tot += warp_cnt[w];
            s_run += tot;
        }
        __syncthreads();
    }
}

// Barriers of a cooperative launch (all CTAs co-resident): CTAs add to `sync[0]`, and those that wait poll it until every CTA has
// arrived `k` times.  (A generation word that the last arriver writes costs a trip to L2 more: 3900 cycles a barrier against
// 2600 on 148 CTAs.)  `sync[1]` counts the CTAs that are done: the last one zeroes both words for the next launch.  Thread 0 of each
// CTA takes part (the CTA barriers around it extend its release and acquire to the other threads); waits are bounded, and a count that
// cannot be this launch's (the caller did not zero the header) ends them too.
constexpr unsigned kGridSpinLimit = 1u << 22;
__device__ __forceinline__ void grid_arrive(unsigned *sync)
{
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(sync) : "memory");
}
__device__ __forceinline__ bool grid_wait(const unsigned *sync, unsigned k)
{
    __shared__ int s_wait_ok;
    if (threadIdx.x == 0) {
        const unsigned want = k * gridDim.x;
        unsigned c, spin = 0;
        do {
            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];\n" : "=r"(c) : "l"(sync) : "memory");
        } while (c < want && ++spin < kGridSpinLimit);
        asm volatile("fence.acq_rel.gpu;\n" ::: "memory");
        s_wait_ok = c >= want && c <= 32u * gridDim.x ? 1 : 0;
    }
    __syncthreads();
    return s_wait_ok != 0;
}
__device__ __forceinline__ void grid_leave(unsigned *sync)
{
    if (threadIdx.x == 0 && atomicAdd(sync + 1, 1u) == gridDim.x - 1u) { sync[0] = 0u; sync[1] = 0u; }
}

// True in every thread of the CTA that arrives last: what the other CTAs wrote before is then visible to it, and nobody has waited.
// Zeroes the count for the next launch; a count that cannot be this launch's is reported.
__device__ __forceinline__ bool last_to_arrive(unsigned *sync, int *status)
{
    __shared__ unsigned s_before;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned before;
        asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;\n" : "=r"(before) : "l"(sync) : "memory");
        if (before == gridDim.x - 1u) *sync = 0u;
        else if (before >= gridDim.x) atomicMax(status, (int)BSP_ERR_TIMEOUT);
        s_before = before;
    }
    __syncthreads();
    return s_before == gridDim.x - 1u;
}

// The digit d of a histogram of kBins bins with cum(d - 1) < need <= cum(d), by a CTA of kT threads: each sums kBins / kT
// neighbouring bins, a scan over the CTA finds the thread that holds it.  Writes the remaining count, the extended prefix and
// the number of keys in the chosen bin, and synchronises the CTA.
template <int kT, int kBins>
__device__ __forceinline__ void select_digit(const unsigned *hist, unsigned *warp_sums, unsigned long long prefix, long long *s_k,
                                             unsigned long long *s_prefix, unsigned *s_left, int width)
{
    constexpr int kPer = kBins / kT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long need = *s_k;
    unsigned h[kPer], mine = 0u;
#pragma unroll
    for (int q = 0; q < kPer; ++q) { h[q] = hist[tid * kPer + q]; mine += h[q]; }
    unsigned inc = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned n = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += n;
    }
    if (lane == 31) warp_sums[warp] = inc;
    __syncthreads();
    long long cum = (long long)inc - mine;
    for (int w = 0; w < warp; ++w) cum += warp_sums[w];
    if (cum < need && need <= cum + mine) {                // (need <= the sum of all bins: one thread)
        int q = 0;
        for (; q < kPer - 1; ++q) {
            if (cum + h[q] >= need) break;
            cum += h[q];
        }
        *s_k = need - cum;
        *s_prefix = (prefix << width) | (unsigned long long)(tid * kPer + q);
        *s_left = h[q];
    }
    __syncthreads();
}

// Select within one CTA of kT threads, on n keys in shared memory, all of them in the span [lo, hi].  The span is cut into up to
// 2048 (4096) equal bins, so that the bin of the threshold holds a few keys whatever the scores look like; it is the next span, until
// at most kFew keys are left for a warp to rank.  `T` is the threshold key, `ties` how many keys equal to it are still to be
// zeroed (lowest index first), `same` how many there are.  0 < need <= n; every thread must call it
// (its first barrier makes the keys visible to all).  Every round but the first starts on a span of fewer bits than the one before
// (bsp_span.cuh), and the rounds are counted, so that the loop ends whatever the keys are.
// (What bounds it is the trip of its instructions to an SM that has not run them before: with the keys in registers and every loop over
// them unrolled it took 4500 cycles for 4096 keys, digits of ten bits and 128 keys ranked one after the other 7800.)
constexpr int kRankMax = 4096;
constexpr int kFew = 32;
constexpr int kShort = 128;              // segments that are ranked without a select: 64 keys 1000 cycles, 2900 with
template <int kT>
struct SmallSelect {
    static constexpr int kWidth = kT >= 1024 ? 12 : 11, kBins = 1 << kWidth;
    __align__(16) unsigned hist[kBins];
    unsigned long long least[kT / 32], most[kT / 32], cand[kFew], T;
    unsigned warp_sums[kT / 32];
    long long need;
    unsigned bin, count, n;
};
__device__ __forceinline__ unsigned long long warp_min(unsigned long long v)
{
    const unsigned h = __reduce_min_sync(0xFFFFFFFFu, (unsigned)(v >> 32));
    const unsigned l = __reduce_min_sync(0xFFFFFFFFu, (unsigned)(v >> 32) == h ? (unsigned)v : 0xFFFFFFFFu);
    return ((unsigned long long)h << 32) | l;
}
// f(i, key) for the keys of this thread, eight loads in flight.
template <int kT, typename L, typename F>
__device__ __forceinline__ void for_keys(int n, L load, F f)
{
#pragma unroll 1
    for (int base = threadIdx.x; base < n; base += 8 * kT) {
        unsigned long long v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (base + u * kT < n) v[u] = load(base + u * kT);
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (base + u * kT < n) f(base + u * kT, v[u]);
    }
}
// The span of the keys of the CTA from every thread's smallest and largest; synchronises the CTA.
template <int kT>
__device__ __forceinline__ void block_span(unsigned long long least, unsigned long long most, SmallSelect<kT> &sh, unsigned long long &lo, unsigned long long &hi)
{
    const int lane = threadIdx.x & 31;
    least = warp_min(least);
    most = ~warp_min(~most);
    if (lane == 0) { sh.least[threadIdx.x >> 5] = least; sh.most[threadIdx.x >> 5] = most; }
    __syncthreads();
    lo = warp_min(sh.least[lane % (kT / 32)]);
    hi = ~warp_min(~sh.most[lane % (kT / 32)]);
}
// Copies keys to shared memory (written by other CTAs: read through L2) and notes this thread's smallest and largest.
template <int kT>
__device__ __forceinline__ void fetch_keys(const unsigned long long *key, int n, unsigned long long *to, unsigned long long &least, unsigned long long &most)
{
    for_keys<kT>(n, [&](int i) { return __ldcg(key + i); }, [&](int i, unsigned long long v) {
        to[i] = v;
        least = v < least ? v : least;
        most = v > most ? v : most;
    });
}
template <int kT>
__device__ __forceinline__ void select_small(const unsigned long long *keys, int n, unsigned long long lo, unsigned long long hi, long long need, SmallSelect<kT> &sh,
                                             unsigned long long &T, long long &ties, unsigned &same)
{
    constexpr int kBins = SmallSelect<kT>::kBins, kMine = kBins / kT, kWarps = kT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto load = [&](int i) { return keys[i]; };
    if (tid == 0) sh.n = 0u;
    unsigned left = (unsigned)n;
    T = hi; ties = need; same = left;                      // (a span of one key)
    for (int round = 0; round < span_rounds(SmallSelect<kT>::kWidth) && lo != hi; ++round) {
        if (left <= (unsigned)kFew) {
            __syncthreads();
            for_keys<kT>(n, load, [&](int, unsigned long long v) {
                if (v >= lo && v <= hi) sh.cand[atomicAdd(&sh.n, 1u)] = v;
            });
            __syncthreads();
            if (warp == 0) {
                const unsigned long long mine_key = lane < (int)left ? sh.cand[lane] : ~0ull;
                unsigned less = 0u, eq = 0u;
#pragma unroll 1
                for (unsigned j = 0; j < left; ++j) {
                    const unsigned long long o = sh.cand[j];
                    less += o < mine_key ? 1u : 0u;
                    eq += o == mine_key ? 1u : 0u;
                }
                // (lanes holding equal keys write the same values)
                if (lane < (int)left && (long long)less < need && need <= (long long)(less + eq)) { sh.T = mine_key; sh.need = need - less; sh.count = eq; }
            }
            __syncthreads();
            T = sh.T; ties = sh.need; same = sh.count;
            break;
        }
#pragma unroll
        for (int q = 0; q < kMine; q += 4) *(uint4 *)(sh.hist + tid * kMine + q) = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        const int shift = span_shift(lo, hi, SmallSelect<kT>::kWidth);
        for_keys<kT>(n, load, [&](int, unsigned long long v) {
            if (v >= lo && v <= hi) atomicAdd(&sh.hist[(unsigned)((v - lo) >> shift)], 1u);
        });
        __syncthreads();
        // the bin with cum(bin - 1) < need <= cum(bin): each thread sums its bins, a scan over the CTA finds the one that holds it
        unsigned h[kMine], mine = 0u;
#pragma unroll
        for (int q = 0; q < kMine; q += 4) {
            const uint4 x = *(const uint4 *)(sh.hist + tid * kMine + q);
            h[q] = x.x; h[q + 1] = x.y; h[q + 2] = x.z; h[q + 3] = x.w;
            mine += x.x + x.y + x.z + x.w;
        }
        unsigned inc = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned o = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += o;
        }
        if (lane == 31) sh.warp_sums[warp] = inc;
        __syncthreads();
        const unsigned before = __reduce_add_sync(0xFFFFFFFFu, lane < warp && lane < kWarps ? sh.warp_sums[lane] : 0u);
        const long long cum = (long long)before + inc - mine;
        if (cum < need && need <= cum + mine) {            // (need <= the sum of all bins: one thread)
            const unsigned want = (unsigned)(need - cum);
            unsigned sum = 0u;
            int bin = -1;
#pragma unroll
            for (int q = 0; q < kMine; ++q) {
                if (bin < 0 && sum + h[q] >= want) { bin = q; sh.need = want - sum; sh.count = h[q]; }
                sum += h[q];
            }
            sh.bin = (unsigned)(tid * kMine + bin);
        }
        __syncthreads();
        need = sh.need;
        left = sh.count;
        span_to_bin(lo, hi, sh.bin, shift);
        T = hi; ties = need; same = left;                  // (a bin of one key: the loop ends)
    }
}

// One large segment (the whole layer) in one cooperative launch: CTA c scores a contiguous slice of the blocks, whose keys stay in its
// shared memory, and the CTAs find the threshold together.  A key is the bit pattern of the score as a float64 (int8 scores are exact in it),
// which orders like the score.
//   1. Histogram of the leading 19 bits (sign, exponent and seven bits of the mantissa) of the keys in 2048 bins, from 14 octaves below the largest key
//      of the first CTA's first blocks to two above, into a global histogram; the CTAs meet, and each derives the bin of the
//      threshold.  (The bins need no look at all keys before; starting at the highest bit in which two keys differ took one more barrier.)
//   2. Only while more than kLocalMax keys are left, or where the bin is one of the ends: digits of eleven bits in the same way.
//   3. The keys that match the prefix are appended to one list with their blocks' numbers, the CTAs meet, and every CTA finishes
//      on the list in its own shared memory (select_small); keys equal to the threshold are zeroed lowest block first, by the same
//      select on their numbers.
//   4. Where more keys than the list holds are equal to the threshold: counts per slice and one more barrier.
// The scratch is zeroed by the CTAs themselves, behind a barrier that they pass while they score.
constexpr int kCoopThreads = 512;
constexpr int kFirstShift = 45, kFirstBelow = 14 * 128;      // leading bits of the first pass; its bins below the reference
constexpr int kCoopBins = 2048, kCoopWidth = 11;
static_assert(3 * kCoopBins <= kSelectHist, "a histogram in use, one that others may still read, one that is being zeroed");
constexpr int kLocalMax = kSelectList;   // candidates that the CTAs finish on their own, in (dynamic) shared memory
constexpr int kSliceMax = 4096;          // keys of a CTA's slice that are kept in shared memory
constexpr size_t kCoopSmem = (size_t)(kLocalMax + kSliceMax) * sizeof(unsigned long long) + (size_t)kLocalMax * sizeof(unsigned);

template <typename A>
__device__ __forceinline__ unsigned long long key_bits(A score) { return (unsigned long long)__double_as_longlong((double)score); }

template <int DT, int NORM, int kBatch>
__global__ void __launch_bounds__(kCoopThreads, 1)
mask_coop_kernel(const uint32_t *W, int I, int HK, int bo, int bi, int NBo, int NBi, typename Acc<DT>::type *score, int keep_scores,
                 long long n_zero, uint8_t *gamma, unsigned *ghist, unsigned *gcount, unsigned long long *cand, unsigned *cand_at, unsigned *geq, unsigned *sync, int *status)
{
    using acc_t = typename Acc<DT>::type;
    __shared__ unsigned hist[kCoopBins], warp_sums[kCoopThreads / 32];
    __shared__ acc_t part[kCoopThreads];
    __shared__ SmallSelect<kCoopThreads> sel;
    extern __shared__ unsigned long long s_dyn[];
    unsigned long long *s_mine = s_dyn;                  // [kLocalMax] this CTA's candidates
    unsigned long long *s_keys = s_dyn + kLocalMax;      // [kSliceMax]
    unsigned *s_at_mine = (unsigned *)(s_keys + kSliceMax);      // [kLocalMax] block numbers of the candidates
    __shared__ unsigned long long s_prefix, s_top;
    __shared__ long long s_k;
    __shared__ unsigned s_left, s_n, s_at;
    __shared__ unsigned warp_cnt[kCoopThreads / 32];
    __shared__ long long s_run;
    const int tid = threadIdx.x;
    const long long n = (long long)NBo * NBi, slice = (n + gridDim.x - 1) / gridDim.x;
    const long long lo = min(n, (long long)blockIdx.x * slice), hi = min(n, lo + slice);
    const int len = (int)(hi - lo);                      // (a slice of more than 2^31 keys would need more CTAs than the launch allows)
    const bool held = len <= kSliceMax;
    for (int q = tid; q < kCoopBins; q += kCoopThreads) hist[q] = 0u;
    if (tid == 0) { s_top = 0ull; s_n = 0u; }
    wait_for_previous();
    W = from_here(W);
    for (int i = (int)blockIdx.x * kCoopThreads + tid; i < kSelectHist + 1; i += (int)gridDim.x * kCoopThreads) ghist[i] = 0u;      // (with gcount[0])
    __syncthreads();
    unsigned long long largest = 0ull;
    score_range<DT, NORM, kBatch, kCoopThreads>(W, I, HK, bo, bi, NBi, lo, hi, 1, part,
        [&](long long B, acc_t total) {
            const unsigned long long key = key_bits(total);
            if (held) s_keys[B - lo] = key;
            if (keep_scores || !held) score[B] = total;
            largest = key > largest ? key : largest;
        },
        [&]() {
            if (blockIdx.x == 0) {
                if (largest) atomicMax(&s_top, largest);
                __syncthreads();
                if (tid == 0) *(unsigned long long *)(gcount + 2) = s_top;
            }
            grid_arrive(sync);
        });
    __syncthreads();
    auto key_at = [&](int i) -> unsigned long long { return held ? s_keys[i] : key_bits(score[lo + i]); };
    unsigned arrived = 1;
    auto give_up = [&]() { if (tid == 0) atomicMax(status, (int)BSP_ERR_TIMEOUT); };
    auto meet = [&]() -> bool { grid_arrive(sync); return grid_wait(sync, ++arrived); };
    if (!grid_wait(sync, 1)) { give_up(); return; }
    // ---- first pass ----
    const unsigned long long ref = __ldcg((const unsigned long long *)(gcount + 2)) >> kFirstShift;
    const unsigned long long first = ref > (unsigned long long)kFirstBelow ? ref - kFirstBelow : 0ull;
    for (int i = tid; i < len; i += kCoopThreads) {
        const unsigned long long b = key_at(i) >> kFirstShift;
        atomicAdd(&hist[b < first ? 0 : (int)min(b - first, (unsigned long long)(kCoopBins - 1))], 1u);
    }
    __syncthreads();
    for (int q = tid; q < kCoopBins; q += kCoopThreads)
        if (hist[q]) atomicAdd(&ghist[q], hist[q]);
    if (tid == 0) s_k = n_zero;
    if (!meet()) { give_up(); return; }
    for (int q = tid; q < kCoopBins; q += kCoopThreads) hist[q] = __ldcg(&ghist[q]);
    __syncthreads();
    select_digit<kCoopThreads, kCoopBins>(hist, warp_sums, 0ull, &s_k, &s_prefix, &s_left, 0);
    // bits above `top` are settled: they are the prefix
    int top = kFirstShift - 1;
    {
        const unsigned long long bin = s_prefix;
        const bool end = bin == (unsigned long long)(kCoopBins - 1) || (bin == 0ull && first > 0ull);
        if (end) top = 63;                               // (keys that the bins do not tell apart: from the start)
        __syncthreads();
        if (tid == 0) {
            if (end) { s_prefix = 0ull; s_k = n_zero; s_left = n > 0xFFFFFFFFll ? 0xFFFFFFFFu : (unsigned)n; }
            else s_prefix = first + bin;
        }
    }
    // ---- further digits ----
    int pi = 1;
    while (top >= 0) {
        for (int q = tid; q < kCoopBins; q += kCoopThreads) hist[q] = 0u;
        __syncthreads();
        if (s_left <= (unsigned)kLocalMax) break;          // few enough candidates: the rest is local
        const unsigned long long prefix = s_prefix;
        const int width = min(kCoopWidth, top + 1), shift = top + 1 - width;
        const unsigned dmask = (1u << width) - 1u;
        for (int i = tid; i < len; i += kCoopThreads) {
            const unsigned long long v = key_at(i);
            if (top >= 63 || ((v >> (top + 1)) == prefix)) atomicAdd(&hist[(unsigned)(v >> shift) & dmask], 1u);
        }
        __syncthreads();
        for (int q = tid; q < kCoopBins; q += kCoopThreads)
            if (hist[q]) atomicAdd(&ghist[pi % 3 * kCoopBins + q], hist[q]);
        if (!meet()) { give_up(); return; }
        for (int q = tid; q < kCoopBins; q += kCoopThreads) hist[q] = __ldcg(&ghist[pi % 3 * kCoopBins + q]);
        // (every CTA has read the histogram before this one: it is zeroed for the pass after the next)
        for (int q = (int)blockIdx.x * kCoopThreads + tid; q < kCoopBins; q += (int)gridDim.x * kCoopThreads) ghist[(pi + 2) % 3 * kCoopBins + q] = 0u;
        __syncthreads();
        select_digit<kCoopThreads, kCoopBins>(hist, warp_sums, prefix, &s_k, &s_prefix, &s_left, width);
        top -= width;
        ++pi;
    }
    if (top >= 0) {
        // bits top .. 0 are still open: gather the keys that match the prefix (one addition to the length of the list per CTA), then
        // finish locally
        const unsigned long long prefix = s_prefix;
        for (int base = 0; base < len; base += kCoopThreads) {
            const int i = base + tid;
            const unsigned long long v = i < len ? key_at(i) : 0ull;
            const bool in = i < len && (top >= 63 || (v >> (top + 1)) == prefix);
            const unsigned ball = __ballot_sync(0xFFFFFFFFu, in);
            unsigned at = 0u;
            if ((tid & 31) == 0 && ball) at = atomicAdd(&s_n, (unsigned)__popc(ball));
            at = __shfl_sync(0xFFFFFFFFu, at, 0) + (unsigned)__popc(ball & ((1u << (tid & 31)) - 1u));
            if (in && at < (unsigned)kLocalMax) { s_mine[at] = v; s_at_mine[at] = (unsigned)(lo + i); }
        }
        __syncthreads();
        const unsigned mine = min(s_n, (unsigned)kLocalMax);
        if (tid == 0 && mine) s_at = atomicAdd(gcount, mine);
        __syncthreads();
        for (unsigned i = tid; i < mine; i += kCoopThreads)
            if (s_at + i < (unsigned)kLocalMax) { cand[s_at + i] = s_mine[i]; cand_at[s_at + i] = s_at_mine[i]; }
        if (!meet()) { give_up(); return; }
        const int cnt = (int)min(__ldcg(gcount), (unsigned)kLocalMax);
        unsigned long long T;
        long long ties;
        unsigned same;
        unsigned long long least = ~0ull, most = 0ull, span_lo, span_hi;
        fetch_keys<kCoopThreads>(cand, cnt, s_mine, least, most);       // (every thread is past its own list: the barrier above)
        block_span<kCoopThreads>(least, most, sel, span_lo, span_hi);
        select_small<kCoopThreads>(s_mine, cnt, span_lo, span_hi, s_k, sel, T, ties, same);
        // of the keys equal to T the first `ties` blocks are zeroed: the select once more, on their numbers
        unsigned long long until = ~0ull;
        if ((long long)same != ties) {
            __syncthreads();
            if (tid == 0) s_n = 0u;
            __syncthreads();
            for (int i = tid; i < cnt; i += kCoopThreads)
                if (s_mine[i] == T) s_at_mine[atomicAdd(&s_n, 1u)] = __ldcg(cand_at + i);
            __syncthreads();
            for (int i = tid; i < (int)same; i += kCoopThreads) s_mine[i] = s_at_mine[i];
            unsigned one;
            long long none;
            select_small<kCoopThreads>(s_mine, (int)same, 0ull, (unsigned long long)(n - 1), ties, sel, until, none, one);
        }
        grid_leave(sync);
        for (int i = tid; i < len; i += kCoopThreads) {
            const unsigned long long v = key_at(i);
            gamma[lo + i] = v < T || (v == T && (unsigned long long)(lo + i) <= until) ? 0 : 1;
        }
        return;
    }
    // every bit is settled and more keys than the list holds are equal to the threshold
    __syncthreads();
    const unsigned long long T = s_prefix;
    const long long ties = s_k;        // keys equal to T to zero, lowest indices first
    if ((long long)s_left == ties) {
        // (every CTA derived the same counts) all keys equal to T are zeroed: no order among them
        grid_leave(sync);
        for (int i = tid; i < len; i += kCoopThreads) gamma[lo + i] = key_at(i) <= T ? 0 : 1;
        return;
    }
    // keys equal to T in this slice
    {
        unsigned c = 0;
        for (int i = tid; i < len; i += kCoopThreads) c += key_at(i) == T ? 1u : 0u;
        for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, d);
        if ((tid & 31) == 0) warp_cnt[tid >> 5] = c;
        __syncthreads();
        if (tid == 0) {
            unsigned tot = 0;
            for (int w = 0; w < kCoopThreads / 32; ++w) tot += warp_cnt[w];
            geq[blockIdx.x] = tot;
        }
    }
    if (!meet()) { give_up(); return; }
    grid_leave(sync);
    const int lane = tid & 31, warp = tid >> 5;
    {
        long long before = 0;
        for (unsigned c = tid; c < blockIdx.x; c += kCoopThreads) before += __ldcg(&geq[c]);
        for (int d = 16; d > 0; d >>= 1) before += __shfl_xor_sync(0xFFFFFFFFu, before, d);
        if (tid == 0) s_run = 0;
        __syncthreads();
        if (lane == 0 && before) atomicAdd((unsigned long long *)&s_run, (unsigned long long)before);
        __syncthreads();
    }
    for (int base = 0; base < len; base += kCoopThreads) {
        const int i = base + tid;
        unsigned long long v = ~0ull;
        if (i < len) v = key_at(i);
        const bool eq = (i < len) && (v == T);
        const unsigned ball = __ballot_sync(0xFFFFFFFFu, eq);
        if (lane == 0) warp_cnt[warp] = __popc(ball);
        __syncthreads();
        long long before = s_run;
        for (int w = 0; w < warp; ++w) before += warp_cnt[w];
        before += __popc(ball & ((1u << lane) - 1u));
        if (i < len) gamma[lo + i] = (v < T || (eq && before < ties)) ? 0 : 1;
        __syncthreads();
        if (tid == 0) {
            long long tot = 0;
            for (int w = 0; w < kCoopThreads / 32; ++w) tot += warp_cnt[w];
            s_run += tot;
        }
        __syncthreads();
    }
}

// Gamma of a segment by one CTA of kT threads, from keys in shared memory and every thread's smallest and largest.
template <int kT>
__device__ __forceinline__ void segment_gamma(const unsigned long long *keys, int n, unsigned long long least, unsigned long long most, long long n_zero, uint8_t *g,
                                              SmallSelect<kT> &sh)
{
    const int tid = threadIdx.x;
    if (n_zero <= 0 || n_zero >= n) {
        for (int i = tid; i < n; i += kT) g[i] = n_zero <= 0 ? 1 : 0;
        return;
    }
    if (n <= kShort) {                                     // ranked directly, a thread per key
        __syncthreads();
        if (tid < n) {
            const unsigned long long mine = keys[tid];
            int rank = 0;
#pragma unroll 4
            for (int j = 0; j < n; ++j) {
                const unsigned long long o = keys[j];
                rank += (o < mine || (o == mine && j < tid)) ? 1 : 0;
            }
            g[tid] = (long long)rank < n_zero ? 0 : 1;
        }
        return;
    }
    unsigned long long lo, hi, T;
    long long ties;
    unsigned same;
    block_span<kT>(least, most, sh, lo, hi);
    select_small<kT>(keys, n, lo, hi, n_zero, sh, T, ties, same);
    if ((long long)same == ties) {                         // every key equal to T is zeroed
        for_keys<kT>(n, [&](int i) { return keys[i]; }, [&](int i, unsigned long long v) { g[i] = v <= T ? 0 : 1; });
        return;
    }
    long long before = 0;                                  // keys equal to T in the stretches of kT before this one
    for (int base = 0; base < n; base += kT) {
        const int i = base + tid;
        const unsigned long long v = i < n ? keys[i] : ~0ull;
        const bool eq = i < n && v == T;
        const unsigned ball = __ballot_sync(0xFFFFFFFFu, eq);
        __syncthreads();
        if ((tid & 31) == 0) sh.warp_sums[tid >> 5] = (unsigned)__popc(ball);
        __syncthreads();
        long long rank = before + __popc(ball & ((1u << (tid & 31)) - 1u));
        for (int w = 0; w < kT / 32; ++w) {
            if (w < (tid >> 5)) rank += sh.warp_sums[w];
            before += sh.warp_sums[w];
        }
        if (i < n) g[i] = (v < T || (eq && rank < ties)) ? 0 : 1;
    }
}
// Segments whose scores another kernel wrote, one CTA each (rows of Gamma; a small layer without a workspace).
__global__ void __launch_bounds__(kScoreThreads)
segment_kernel(const unsigned long long *key, int n, long long n_zero, uint8_t *gamma)
{
    __shared__ SmallSelect<kScoreThreads> sh;
    extern __shared__ unsigned long long s_dyn[];          // [n] keys
    wait_for_previous<false>();
    key += (size_t)blockIdx.x * n;
    gamma += (size_t)blockIdx.x * n;
    unsigned long long least = ~0ull, most = 0ull;
    fetch_keys<kScoreThreads>(key, n, s_dyn, least, most);
    segment_gamma<kScoreThreads>(s_dyn, n, least, most, n_zero, gamma, sh);
}

// Per-row scope, rows of up to kRankMax blocks: a CTA scores a row of Gamma and selects in it, in one launch and without meeting
// any other CTA.
template <int DT, int NORM, int kBatch>
__global__ void __launch_bounds__(kRankThreads)
mask_row_kernel(const uint32_t *W, int I, int HK, int bo, int bi, int NBi, typename Acc<DT>::type *score, int keep_scores, long long n_zero, uint8_t *gamma)
{
    using acc_t = typename Acc<DT>::type;
    __shared__ acc_t part[kRankThreads];
    __shared__ SmallSelect<kRankThreads> sh;
    extern __shared__ unsigned long long s_dyn[];          // [NBi] keys
    const long long lo = (long long)blockIdx.x * NBi;
    unsigned long long least = ~0ull, most = 0ull;
    wait_for_previous();
    score_range<DT, NORM, kBatch, kRankThreads>(from_here(W), I, HK, bo, bi, NBi, lo, lo + NBi, 1, part,
        [&](long long B, acc_t total) {
            unsigned long long key;
            memcpy(&key, &total, 8);
            s_dyn[B - lo] = key;
            if (keep_scores) score[B] = total;
            least = key < least ? key : least;
            most = key > most ? key : most;
        }, []() {});
    segment_gamma<kRankThreads>(s_dyn, NBi, least, most, n_zero, gamma + lo, sh);
}

// One segment of up to kMidMax keys: every CTA finds the threshold for itself, on all keys, and writes 1024 entries of Gamma.
constexpr int kMidThreads = 1024;
constexpr int kMidMax = 24576;           // (keys of eight bytes in shared memory)
__global__ void __launch_bounds__(kMidThreads)
select_mid_kernel(const unsigned long long *key, int n, long long n_zero, uint8_t *gamma)
{
    __shared__ SmallSelect<kMidThreads> sh;
    extern __shared__ unsigned long long s_dyn[];          // [n] keys
    const int tid = threadIdx.x, i = blockIdx.x * kMidThreads + tid;
    wait_for_previous<false>();
    if (n_zero <= 0 || n_zero >= n) {
        if (i < n) gamma[i] = n_zero <= 0 ? 1 : 0;
        return;
    }
    unsigned long long least = ~0ull, most = 0ull, lo, hi, T;
    long long ties;
    unsigned same;
    fetch_keys<kMidThreads>(key, n, s_dyn, least, most);
    block_span<kMidThreads>(least, most, sh, lo, hi);
    select_small<kMidThreads>(s_dyn, n, lo, hi, n_zero, sh, T, ties, same);
    const unsigned long long mine = i < n ? s_dyn[i] : ~0ull;
    long long rank = 0;                                    // keys equal to T before this one
    const bool eq = i < n && mine == T;
    if ((long long)same != ties) {                         // (else every key equal to T is zeroed)
        unsigned before = 0u;
        for (int j = tid; j < (int)blockIdx.x * kMidThreads; j += kMidThreads) before += s_dyn[j] == T ? 1u : 0u;
        before = __reduce_add_sync(0xFFFFFFFFu, before);
        const unsigned ball = __ballot_sync(0xFFFFFFFFu, eq);
        if ((tid & 31) == 0) { sh.hist[tid >> 5] = before; sh.hist[32 + (tid >> 5)] = (unsigned)__popc(ball); }
        __syncthreads();
        rank = __popc(ball & ((1u << (tid & 31)) - 1u));
        for (int w = 0; w < kMidThreads / 32; ++w) rank += sh.hist[w] + (w < (tid >> 5) ? sh.hist[32 + w] : 0u);
    }
    if (i < n) gamma[i] = (mine < T || (eq && rank < ties)) ? 0 : 1;
}

// Layers of up to kRankMax blocks in one launch: every CTA scores its blocks, and the one that arrives last selects on all of them.
// (Nobody waits, so the launch need not be cooperative: those start on a grid of about 2 us and after the kernel before them has drained.)
template <int DT, int NORM, int kBatch>
__global__ void __launch_bounds__(kRankThreads)
mask_small_kernel(const uint32_t *W, int I, int HK, int bo, int bi, int NBo, int NBi, int BC,
                  typename Acc<DT>::type *score, long long n_zero, uint8_t *gamma, unsigned *sync, int *status)
{
    using acc_t = typename Acc<DT>::type;
    __shared__ acc_t part[kRankThreads];
    __shared__ SmallSelect<kRankThreads> sh;
    extern __shared__ unsigned long long s_dyn[];          // [NB] keys
    const int NB = NBo * NBi;
    wait_for_previous();
    W = from_here(W);
    // BC blocks per CTA: b_o threads score one block
    {
        const int bl = threadIdx.x % BC, r = threadIdx.x / BC;
        const long long B = (long long)blockIdx.x * BC + bl;
        const bool mine = r < bo && B < NB;
        const acc_t total = block_score<DT, NORM, kBatch>(W, I, HK, bo, bi, NBi, B, r, mine, part, bl, BC);
        if (mine && r == 0) score[B] = total;
    }
    if (!last_to_arrive(sync, status)) return;
    unsigned long long least = ~0ull, most = 0ull;
    fetch_keys<kRankThreads>((const unsigned long long *)score, NB, s_dyn, least, most);
    segment_gamma<kRankThreads>(s_dyn, NB, least, most, n_zero, gamma, sh);
}

// How a call is made up: the layer, and what its kernels share.
struct MaskCall {
    const bsp_wdesc &wd;
    const uint32_t *W;
    bool keep_scores;                    // the caller wants them
    long long n_zero;
    uint8_t *gamma;
    void *scores;
    void *ws;                            // NULL: none
    cudaStream_t st;
    int NBo, NBi;
    long long NB;
};

int mask_sm_count(int dev)
{
    static int n_sm[64] = {};
    if (n_sm[dev] == 0 && cudaDeviceGetAttribute(&n_sm[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return n_sm[dev];
}

// Whole layer of up to kRankMax blocks, with a workspace.
template <int DT, int NORM, int kBatch>
bsp_status run_mask_small(const MaskCall &c)
{
    // few blocks per CTA spread the layer over the SMs
    int BC = 8;
    while ((c.NB + BC - 1) / BC > 128 && BC * 2 * c.wd.bo <= kRankThreads) BC *= 2;
    BSP_CUDA_OK(launch_after(mask_small_kernel<DT, NORM, kBatch>, dim3((unsigned)((c.NB + BC - 1) / BC)), dim3(kRankThreads), (size_t)c.NB * 8, c.st, c.W, c.wd.I, c.wd.H * c.wd.K,
                             c.wd.bo, c.wd.bi, c.NBo, c.NBi, BC, (typename Acc<DT>::type *)c.scores, c.n_zero, c.gamma, (unsigned *)c.ws + kWsSyncWord, (int *)c.ws));
    return BSP_OK;
}

// Rows of up to kRankMax blocks.
template <int DT, int NORM, int kBatch>
bsp_status run_mask_rows(const MaskCall &c)
{
    BSP_CUDA_OK(launch_after(mask_row_kernel<DT, NORM, kBatch>, dim3((unsigned)c.NBo), dim3(kRankThreads), (size_t)c.NBi * 8, c.st, c.W, c.wd.I, c.wd.H * c.wd.K, c.wd.bo,
                             c.wd.bi, c.NBi, (typename Acc<DT>::type *)c.scores, c.keep_scores ? 1 : 0, c.n_zero, c.gamma));
    return BSP_OK;
}

// Whole layer of more than kMidMax blocks, with a workspace; BSP_ERR_CAPACITY: not all CTAs fit (a partitioned GPU).
template <int DT, int NORM, int kBatch>
bsp_status run_mask_coop(const MaskCall &c)
{
    static bool opted[64] = {};
    int dev = 0;
    BSP_CUDA_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return BSP_ERR_CUDA;
    if (!opted[dev]) {
        BSP_CUDA_OK(cudaFuncSetAttribute(mask_coop_kernel<DT, NORM, kBatch>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCoopSmem));
        opted[dev] = true;
    }
    const int n_sm = mask_sm_count(dev);
    if (n_sm <= 0) return BSP_ERR_CUDA;
    const int grid = n_sm < kSelectMaxCtas ? n_sm : kSelectMaxCtas;      // one CTA per SM
    unsigned *ghist = (unsigned *)((char *)c.ws + kWsHeader + align_up((size_t)c.NB * 8, 256)), *gcount = ghist + kSelectHist, *geq = gcount + 8;
    unsigned long long *cand = (unsigned long long *)(geq + kSelectMaxCtas);
    unsigned *cand_at = (unsigned *)(cand + kSelectList);
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(kCoopThreads); cfg.dynamicSmemBytes = kCoopSmem; cfg.stream = c.st;
    cfg.attrs = attr; cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, mask_coop_kernel<DT, NORM, kBatch>, c.W, (int)c.wd.I, (int)(c.wd.H * c.wd.K), (int)c.wd.bo, (int)c.wd.bi, c.NBo, c.NBi,
                                             (typename Acc<DT>::type *)c.scores, c.keep_scores ? 1 : 0, c.n_zero, c.gamma, ghist, gcount, cand, cand_at, geq,
                                             (unsigned *)c.ws + kWsSyncWord, (int *)c.ws);
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        (void)cudaGetLastError();
        return BSP_ERR_CAPACITY;
    }
    BSP_CUDA_OK(e);
    return BSP_OK;
}

// Scores in a launch of their own.
template <int DT, int NORM, int kBatch>
bsp_status run_scores(const MaskCall &c)
{
    // eight CTAs per SM's worth, each looping
    const int per_cta = kBatch == 1 && NORM != BSP_NORM_VAR ? kScoreThreads : kScoreThreads / c.wd.bo;
    const long long rounds = (c.NB + per_cta - 1) / per_cta;
    const unsigned grid = (unsigned)(rounds < 148 * 8 ? rounds : 148 * 8);
    BSP_CUDA_OK(launch_after(score_kernel<DT, NORM, kBatch>, dim3(grid), dim3(kScoreThreads), 0, c.st, c.W, c.wd.I, c.wd.H * c.wd.K, c.wd.bo, c.wd.bi, c.NBo, c.NBi,
                             (typename Acc<DT>::type *)c.scores));
    return BSP_OK;
}

template <int DT, int NORM, int kBatch>
bsp_status run_mask(const MaskCall &c, bsp_scope scope)
{
    const bool layer = scope == BSP_SCOPE_LAYER;
    // (A row per CTA where there is a wave of them at most, or rows are short; more and longer ones score faster on all threads of the GPU:
    // 4096 x 4096 bfloat16 with its compaction 52 us by rows, 45 in two launches; 64 x 4096 10.7 and 12.4.  So does the variance, whose two
    // passes over a block keep too much at hand for 512 threads: 512 x 512 3x3 18.2 us by rows, 14.4 in two launches.)
    if constexpr (NORM != BSP_NORM_VAR)
        if (!layer && (c.NBi <= 128 || (c.NBi <= kRankMax && c.NBo <= 128))) return run_mask_rows<DT, NORM, kBatch>(c);
    if (layer && c.ws != nullptr && c.NB <= kRankMax) return run_mask_small<DT, NORM, kBatch>(c);
    if (layer && c.ws != nullptr && c.NB > kMidMax && c.n_zero > 0 && c.n_zero < c.NB) {
        const bsp_status rc = run_mask_coop<DT, NORM, kBatch>(c);
        if (rc != BSP_ERR_CAPACITY) return rc;
    }
    const bsp_status rc = run_scores<DT, NORM, kBatch>(c);
    if (rc != BSP_OK) return rc;
    // (Programmatic dependents of the score kernel, without the gap between launches.  The score kernel lets nothing in early, as its
    // CTAs fill the SMs several times over.)
    const unsigned long long *keys = (const unsigned long long *)c.scores;
    const long long seg = layer ? c.NB : (long long)c.NBi;
    if (seg <= kRankMax)
        BSP_CUDA_OK(launch_after(segment_kernel, dim3((unsigned)(c.NB / seg)), dim3(kScoreThreads), (size_t)seg * 8, c.st, keys, (int)seg, c.n_zero, c.gamma));
    else if (layer && c.NB <= kMidMax) {
        static bool opted[64] = {};
        int dev = 0;
        BSP_CUDA_OK(cudaGetDevice(&dev));
        if (dev < 0 || dev >= 64) return BSP_ERR_CUDA;
        if (!opted[dev]) {
            BSP_CUDA_OK(cudaFuncSetAttribute(select_mid_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMidMax * 8));
            opted[dev] = true;
        }
        BSP_CUDA_OK(launch_after(select_mid_kernel, dim3((unsigned)((c.NB + kMidThreads - 1) / kMidThreads)), dim3(kMidThreads), (size_t)c.NB * 8, c.st, keys, (int)c.NB, c.n_zero, c.gamma));
    }
    else {
        select_kernel<<<layer ? 1u : (unsigned)c.NBo, kSelectThreads, 0, c.st>>>(keys, layer ? c.NB : (long long)c.NBi, c.n_zero, c.gamma);
        BSP_CUDA_OK(cudaGetLastError());
    }
    return BSP_OK;
}

template <int DT, int NORM>
bsp_status run_mask(const MaskCall &c, bsp_scope scope)
{
    return c.wd.H * c.wd.K == 1 ? run_mask<DT, NORM, 1>(c, scope) : run_mask<DT, NORM, 9>(c, scope);
}

}  // namespace

bsp_status launch_mask(const bsp_wdesc &wd, const void *W, bsp_norm norm, bsp_scope scope, int64_t n_zero,
                       uint8_t *gamma, void *scores, bool keep_scores, void *ws, cudaStream_t st)
{
    const int NBo = wd.O / wd.bo, NBi = wd.I / wd.bi;
    const MaskCall c = {wd, (const uint32_t *)W, keep_scores, (long long)n_zero, gamma, scores, ws, st, NBo, NBi, (long long)NBo * NBi};
    if (wd.wtype == BSP_I8) return norm == BSP_NORM_L2 ? run_mask<BSP_I8, BSP_NORM_L2>(c, scope) : run_mask<BSP_I8, BSP_NORM_L1>(c, scope);
    if (wd.wtype == BSP_BF16)
        return norm == BSP_NORM_L2 ? run_mask<BSP_BF16, BSP_NORM_L2>(c, scope) : norm == BSP_NORM_L1 ? run_mask<BSP_BF16, BSP_NORM_L1>(c, scope) : run_mask<BSP_BF16, BSP_NORM_VAR>(c, scope);
    return norm == BSP_NORM_L2 ? run_mask<BSP_F32, BSP_NORM_L2>(c, scope) : norm == BSP_NORM_L1 ? run_mask<BSP_F32, BSP_NORM_L1>(c, scope) : run_mask<BSP_F32, BSP_NORM_VAR>(c, scope);
}

}  // namespace bsp
