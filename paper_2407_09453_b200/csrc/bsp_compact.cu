// Compaction of Gamma (.) W: compressed block rows (row_ptr, col_idx, canonical payload) and the packed form read by
// the product kernel.  Section "Block Sparsity in a Matrix" (compress block row) and Section "Subvolumes, Data
// Compression, and Data Movements" of the paper.
#include <cuda.h>
#include "bsp_internal.cuh"

namespace bsp {

PackedLayout packed_layout(const bsp_wdesc &wd)
{
    PackedLayout L;
    const int esz = elem_bytes(wd.wtype);
    L.enabled = ((long long)wd.I * esz) % 16 == 0 && wd.O % 8 == 0;
    L.off_payload = 256;
    L.total_bytes = align_up(L.off_payload + (L.enabled ? (size_t)wd.O * wd.H * wd.K * wd.I * esz : 0) + 256, 256);
    return L;
}

bool packed_spans(const bsp_wdesc &wd, const void *packed)
{
    typedef CUresult (*RangeFn)(CUdeviceptr *, size_t *, CUdeviceptr);
    static const RangeFn range = []() -> RangeFn {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        return cudaGetDriverEntryPoint("cuMemGetAddressRange", &ptr, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess ? (RangeFn)ptr : nullptr;
    }();
    CUdeviceptr base = 0;
    size_t size = 0;
    if (range == nullptr || range(&base, &size, (CUdeviceptr)(uintptr_t)packed) != CUDA_SUCCESS) return false;
    const size_t at = (size_t)((uintptr_t)packed - (uintptr_t)base);
    return at <= size && packed_layout(wd).total_bytes <= size - at;
}

namespace {

constexpr int kThreads = 256;

// b_o and b_i are 4, 8 or 16: divisions by them are shifts by lg().
__device__ __forceinline__ int lg(int b) { return 31 - __clz(b); }

// Exclusive prefix sum of v over the CTA's threads; every thread of the CTA must call it.
__device__ __forceinline__ int block_exclusive_scan(int v, int *warp_sums, int &total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int n = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += n;
    }
    if (lane == 31) warp_sums[warp] = inc;
    __syncthreads();
    int before = 0, tot = 0;
    for (int w = 0; w < kThreads / 32; ++w) {
        const int s = warp_sums[w];
        if (w < warp) before += s;
        tot += s;
    }
    __syncthreads();
    total = tot;
    return before + inc - v;
}


// Copies the cnt stored blocks of row l (columns s_cols[]) into the canonical payload in pieces of type V (one or
// several elements; a block row of b_i elements is contiguous in W and in the payload).  Each thread loads four
// pieces before it stores them.
template <typename T, typename V>
__device__ __forceinline__ void fill_copy(int l, int part, int parts, const T *W, int I, int HK, int bo, int bi,
                                          int first, int cnt, const int *s_cols, T *__restrict__ payload,
                                          long long capacity_blocks)
{
    constexpr int per = (int)(sizeof(V) / sizeof(T));
    const int bi_v = bi / per;                          // pieces per block row, a power of two
    const int blk = bo * HK * bi;
    const unsigned blk_v = (unsigned)(bo * HK * bi_v);
    const unsigned total = (unsigned)cnt * blk_v;       // at most I * b_o * H * K: fits 32 bits
    const unsigned stride = (unsigned)parts * kThreads;
    for (unsigned e0 = (unsigned)part * kThreads + threadIdx.x; e0 < total; e0 += 4 * stride) {
        V v[4];
        V *dst[4];
        bool ok[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned e = e0 + u * stride;
            ok[u] = e < total;
            const int n = ok[u] ? (int)(e / blk_v) : 0;
            const int q = ok[u] ? (int)(e - (unsigned)n * blk_v) : 0;
            const int c = q & (bi_v - 1), rt = q >> lg(bi_v);
            const int r = rt / HK, t = rt - r * HK;
            ok[u] = ok[u] && (long long)(first + n) < capacity_blocks;
            dst[u] = (V *)(payload + (size_t)(first + n) * blk + (size_t)rt * bi) + c;
            if (ok[u]) v[u] = *((const V *)(W + ((size_t)(l * bo + r) * HK + t) * I + (size_t)s_cols[n] * bi) + c);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (ok[u]) *dst[u] = v[u];
    }
}

// Final launch, first part.  `parts` CTAs per row of Gamma: column indices in ascending order and the canonical payload
// payload[n][r][h][k][c] = W[l b_o + r][h][k][iota b_i + c].  `first` = stored blocks in the rows above; returns
// the number of stored blocks of row l.  kHeld: Gamma is in shared memory
// (`held`), and a row starts without a trip to L2 (about 0.1 us of a call: mask and compaction of 64x64 3x3, int8, 7.10 -> 6.98 us).
template <typename T, bool kHeld>
__device__ __forceinline__ int csr_fill_body(int l, int part, int parts, const T *W,
                                              const uint8_t *gamma, const uint8_t *held, int NBi, int I, int HK, int bo, int bi,
                                              int first, int32_t *__restrict__ col_idx,
                                              T *__restrict__ payload, long long capacity_blocks)
{
    __shared__ int warp_sums[kThreads / 32];
    __shared__ int s_run;
    extern __shared__ int s_cols[];      // NBi ints: columns of this row's stored blocks
    const uint8_t *g = gamma + (size_t)l * NBi;
    if (threadIdx.x == 0) s_run = 0;
    __syncthreads();
    for (int base = 0; base < NBi; base += kThreads) {
        const int i = base + threadIdx.x;
        const int v = (i < NBi && (kHeld ? (uint32_t)held[(size_t)l * NBi + i] : load_free(g + i))) ? 1 : 0;
        int tot;
        const int before = block_exclusive_scan(v, warp_sums, tot);
        if (v) {
            const int n = s_run + before;
            s_cols[n] = i;
            if (part == 0 && (long long)(first + n) < capacity_blocks) col_idx[first + n] = i;
        }
        __syncthreads();
        if (threadIdx.x == 0) s_run += tot;
        __syncthreads();
    }
    if (payload == nullptr) return s_run;
    const int cnt = s_run;
    // the CTAs of one row (`parts` of them) all build the column list, then share the copy, in the widest pieces
    // (up to 16 bytes) that the block width, the row pitch of W and the two base addresses allow
    const size_t row_bytes = (size_t)bi * sizeof(T), pitch = (size_t)I * sizeof(T);
    const uintptr_t bases = (uintptr_t)W | (uintptr_t)payload;
    size_t vb = 16;
    while (vb > sizeof(T) && (row_bytes % vb || pitch % vb || bases % vb)) vb >>= 1;
    if (vb == 16) fill_copy<T, uint4>(l, part, parts, W, I, HK, bo, bi, first, cnt, s_cols, payload, capacity_blocks);
    else if (vb == 8) fill_copy<T, uint2>(l, part, parts, W, I, HK, bo, bi, first, cnt, s_cols, payload, capacity_blocks);
    else if (vb == 4 && sizeof(T) < 4) fill_copy<T, uint32_t>(l, part, parts, W, I, HK, bo, bi, first, cnt, s_cols, payload, capacity_blocks);
    else fill_copy<T, T>(l, part, parts, W, I, HK, bo, bi, first, cnt, s_cols, payload, capacity_blocks);
    return cnt;
}

// Sum of v over the CTA's threads; every thread of the CTA must call it.
__device__ __forceinline__ int block_sum(int v, int *warp_sums)
{
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = v;
    __syncthreads();
    int tot = 0;
    for (int w = 0; w < kThreads / 32; ++w) tot += warp_sums[w];
    return tot;
}

// Non-zero bytes among the first n bytes of Gamma in shared memory (the array is 16-byte aligned), four per load:
// this thread's share; the caller adds the shares with block_sum().
__device__ __forceinline__ int ones_share(const uint8_t *g, int n)
{
    int c = 0;
    const int nw = n >> 2;
    for (int i = threadIdx.x; i < nw; i += kThreads) c += __popc(__vsetne4(((const uint32_t *)g)[i], 0u));
    if ((int)threadIdx.x < (n & 3)) c += g[(nw << 2) + threadIdx.x] ? 1 : 0;
    return c;
}

// The same count over the first n bytes of Gamma in global memory (layers whose Gamma does not fit shared memory): 16-byte
// loads, eight in flight per thread, when the addresses allow.
__device__ __forceinline__ int ones_share_global(const uint8_t *g, int n)
{
    int c = 0;
    if ((((uintptr_t)g) & 15u) == 0) {
        const uint4 *g4 = (const uint4 *)g;
        const int n4 = n >> 4;
        for (int i0 = threadIdx.x; i0 < n4; i0 += 8 * kThreads) {
            uint4 q[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = i0 + u * kThreads;
                q[u] = i < n4 ? load_free(g4 + i) : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u)
                c += __popc(__vsetne4(q[u].x, 0u)) + __popc(__vsetne4(q[u].y, 0u)) + __popc(__vsetne4(q[u].z, 0u)) + __popc(__vsetne4(q[u].w, 0u));
        }
        for (int i = (n4 << 4) + threadIdx.x; i < n; i += kThreads) c += load_free(g + i) ? 1 : 0;
    } else {
        for (int i = threadIdx.x; i < n; i += kThreads) c += load_free(g + i) ? 1 : 0;
    }
    return c;
}

// The packed form: Gamma (.) W in the layout of W, [O][H][K][I], the channels of zeroed blocks cleared.  The b_o H K rows
// (o, tap) of a row of Gamma share its entries, so a thread takes one 16-byte chunk of input channels of up to eight of
// these rows: Gamma is read once, then the rows that are needed are loaded together.  (One chunk at a time, each behind its
// own look at Gamma, took 16.9 us for 4096 x 4096 bf16, and 20.9 with the index part beside it, which is 15.5 like this.)
constexpr int kDenseRows = 8;
template <int esz>
__device__ __forceinline__ void dense_body(int idx, int n_ctas, const void *W, const uint8_t *gamma, int I, int HK, int bo, int bi,
                                           int NBo, int NBi, uint8_t *__restrict__ out)
{
    const bool aligned = (((uintptr_t)W) & 15u) == 0;
    constexpr int cpc = 16 / esz;                     // channels per chunk
    const int cpr = I / cpc;                          // chunks per row
    const int rows = bo * HK, groups = (rows + kDenseRows - 1) / kDenseRows;
    const long long total = (long long)NBo * groups * cpr, stride = (long long)n_ctas * kThreads;
    const bool small = total < (1ll << 31);
    for (long long e = (long long)idx * kThreads + threadIdx.x; e < total; e += stride) {
        // (a 64-bit division costs an order of magnitude more than a 32-bit one: taken only by layers that need it)
        const int lg_ = small ? (int)((unsigned)e / (unsigned)cpr) : (int)(e / cpr);
        const int c = (int)(e - (long long)lg_ * cpr);
        const int l = lg_ / groups, r0 = (lg_ - l * groups) * kDenseRows, n = min(kDenseRows, rows - r0);
        // which 4-byte words of the chunk are kept (a word's channels lie in one block: b_i is a multiple of 4)
        const uint8_t *g = gamma + (size_t)l * NBi + ((c * cpc) >> lg(bi));
        uint32_t keep[4];
        if (bi >= cpc) {
            keep[0] = keep[1] = keep[2] = keep[3] = load_free(g) ? 0xFFFFFFFFu : 0u;
        } else if (cpc / bi == 2) {
            keep[0] = keep[1] = load_free(g) ? 0xFFFFFFFFu : 0u;
            keep[2] = keep[3] = load_free(g + 1) ? 0xFFFFFFFFu : 0u;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) keep[q] = load_free(g + q) ? 0xFFFFFFFFu : 0u;
        }
        const bool any = (keep[0] | keep[1] | keep[2] | keep[3]) != 0u;
        const size_t pitch = (size_t)cpr * 16, at = ((size_t)l * rows + r0) * pitch + (size_t)c * 16;
        const uint8_t *src = (const uint8_t *)W + at;
        uint4 v[kDenseRows];
#pragma unroll
        for (int u = 0; u < kDenseRows; ++u) {
            v[u] = make_uint4(0u, 0u, 0u, 0u);
            if (u < n && any) {
                if (aligned) v[u] = load_free((const uint4 *)(src + u * pitch));
                else {                                // W only 4-byte aligned: word by word
                    const uint32_t *s4 = (const uint32_t *)(src + u * pitch);
                    v[u] = make_uint4(load_free(s4), load_free(s4 + 1), load_free(s4 + 2), load_free(s4 + 3));
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kDenseRows; ++u)
            if (u < n) *(uint4 *)(out + at + u * pitch) = make_uint4(v[u].x & keep[0], v[u].y & keep[1], v[u].z & keep[2], v[u].w & keep[3]);
    }
}

// Column indices and row pointers of kIndexRows rows of Gamma without a payload, one row per warp: the CTA counts the stored
// blocks of all rows before its first one together (one count for eight rows instead of one for each: with 512 rows of 512
// the counts read 67 MB and took 13 us), then every warp counts and lists its own row, 16 entries per lane and step.
constexpr int kIndexRows = kThreads / 32;
__device__ __forceinline__ void index_rows(int cta, const uint8_t *gamma, int NBo, int NBi, int32_t *__restrict__ row_ptr,
                                           int32_t *__restrict__ col_idx, long long capacity_blocks, int *s_sum, int *status)
{
    __shared__ int s_cnt[kIndexRows];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, l0 = cta * kIndexRows, l = l0 + warp;
    const uint8_t *g = gamma + (size_t)l * NBi;
    const bool wide = NBi % 16 == 0 && (((uintptr_t)gamma) & 15u) == 0;
    // bit q of the result: entry i + q of the row is kept (i = 16 entries of this lane)
    auto bits_of = [&](int i) -> unsigned {
        unsigned m = 0u;
        if (wide) {
            if (i < NBi) {
                const uint4 w = load_free((const uint4 *)(g + i));
                const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t one = __vsetne4(x[k], 0u);       // 1 in every non-zero byte
                    m |= ((one | (one >> 7) | (one >> 14) | (one >> 21)) & 15u) << (4 * k);
                }
            }
        } else {
            for (int q = 0; q < 16 && i + q < NBi; ++q) m |= load_free(g + i + q) ? 1u << q : 0u;
        }
        return m;
    };
    int cnt = 0;
    if (l < NBo)
        for (int i = lane * 16; i < NBi; i += 512) cnt += __popc(bits_of(i));
    for (int d = 16; d > 0; d >>= 1) cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, d);
    if (lane == 0) s_cnt[warp] = cnt;
    int first = block_sum(ones_share_global(gamma, l0 * NBi), s_sum);      // (its barriers publish s_cnt too)
    for (int w = 0; w < warp; ++w) first += s_cnt[w];
    if (l >= NBo) return;
    if (lane == 0) {
        row_ptr[l] = first;
        if (l == NBo - 1) {
            row_ptr[NBo] = first + cnt;
            if ((long long)(first + cnt) > capacity_blocks) atomicMax(status, (int)BSP_ERR_CAPACITY);
        }
    }
    int at = first;
    for (int base = 0; base < NBi; base += 512) {
        const int i = base + lane * 16;
        unsigned m = i < NBi ? bits_of(i) : 0u;
        int inc = __popc(m);
        const int mine = inc;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += o;
        }
        int n = at + inc - mine;
        for (; m; m &= m - 1, ++n)
            if ((long long)n < capacity_blocks) col_idx[n] = i + __ffs(m) - 1;
        at += __shfl_sync(0xFFFFFFFFu, inc, 31);
    }
}

struct CompactArgs {
    const void *W;
    const uint8_t *gamma;
    int O, I, HK, bo, bi, NBo, NBi;
    int32_t *row_ptr_out;
    int32_t *col_idx;
    void *payload;
    long long capacity_blocks;
    int fill_parts;                   // CTAs per row of Gamma in the first part of the grid
    int n_fill;                       // CTAs of the first part
    uint8_t *dense;                   // packed form (NULL: none)
    int dense_ctas;                   // CTAs of the second part of the grid
    PackedHeader *hdr;
    PackedHeader hdr_init;
    int *status;
};

// The whole compaction in ONE launch: CTAs [0, NBo * fill_parts) write col_idx and the canonical payload, one row of
// Gamma each, the rest write the packed form.  Every CTA of the first part counts for itself the stored blocks that
// precede its row (no scan launch, nobody waits): from a copy of Gamma in shared memory for layers of up to
// kSmallBlocks blocks, from global memory (through L2, while the other CTAs write the packed form) for larger ones.
// T is the storage type of a weight.
constexpr int kSmallBlocks = 4096;

template <typename T, bool kBig>
__global__ void __launch_bounds__(kThreads, 5) compact_kernel(const CompactArgs args)
{
    __shared__ __align__(16) uint8_t s_gamma[kBig ? 16 : kSmallBlocks];
    __shared__ int s_sum[kThreads / 32];
    wait_for_previous();
    CompactArgs a = args;
    a.W = from_here((const uint8_t *)args.W);
    a.gamma = from_here(args.gamma);
    const int n_fill = a.n_fill;
    if ((int)blockIdx.x >= n_fill) {
        if ((int)blockIdx.x == n_fill && threadIdx.x == 0 && a.hdr != nullptr) *a.hdr = a.hdr_init;
        if (a.dense != nullptr)
            dense_body<(int)sizeof(T)>((int)blockIdx.x - n_fill, a.dense_ctas, a.W, a.gamma, a.I, a.HK, a.bo, a.bi, a.NBo, a.NBi, a.dense);
        return;
    }
    if constexpr (kBig)
        if (a.payload == nullptr) {
            index_rows((int)blockIdx.x, a.gamma, a.NBo, a.NBi, a.row_ptr_out, a.col_idx, a.capacity_blocks, s_sum, a.status);
            return;
        }
    const int l = (int)blockIdx.x / a.fill_parts, part = (int)blockIdx.x % a.fill_parts;
    int first;
    if constexpr (kBig) {
        first = block_sum(ones_share_global(a.gamma, l * a.NBi), s_sum);      // (NB_o NB_i < 2^31: checked by the host)
    } else {
        const int NB = a.NBo * a.NBi;
        const bool word_ok = (((uintptr_t)a.gamma) & 3u) == 0;
        for (int i = threadIdx.x * 4; i < NB; i += kThreads * 4) {
            if (i + 4 <= NB && word_ok) *(uint32_t *)(s_gamma + i) = load_free((const uint32_t *)(a.gamma + i));
            else for (int q = i; q < min(NB, i + 4); ++q) s_gamma[q] = a.gamma[q];
        }
        __syncthreads();
        first = block_sum(ones_share(s_gamma, l * a.NBi), s_sum);
    }
    const int cnt = csr_fill_body<T, !kBig>(l, part, a.fill_parts, (const T *)a.W, a.gamma, s_gamma, a.NBi, a.I, a.HK, a.bo, a.bi, first,
                                     a.col_idx, (T *)a.payload, a.capacity_blocks);
    if (part == 0 && threadIdx.x == 0) {
        a.row_ptr_out[l] = first;
        if (l == a.NBo - 1) {
            a.row_ptr_out[a.NBo] = first + cnt;
            if ((long long)(first + cnt) > a.capacity_blocks) atomicMax(a.status, (int)BSP_ERR_CAPACITY);
        }
    }
}

__global__ void count_ones_kernel(const uint8_t *__restrict__ gamma, long long n, unsigned long long *out)
{
    unsigned long long c = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        c += gamma[i] ? 1 : 0;
    for (int d = 16; d > 0; d >>= 1) c += __shfl_down_sync(0xFFFFFFFFu, c, d);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

}  // namespace

bsp_status launch_count(const uint8_t *gamma, int64_t n, unsigned long long *out, cudaStream_t st)
{
    BSP_CUDA_OK(cudaMemsetAsync(out, 0, sizeof(unsigned long long), st));
    int64_t grid = (n + 255) / 256;
    if (grid > 296) grid = 296;
    if (grid < 1) grid = 1;
    count_ones_kernel<<<(unsigned)grid, 256, 0, st>>>(gamma, n, out);
    BSP_CUDA_OK(cudaGetLastError());
    return BSP_OK;
}

bsp_status launch_compact(const bsp_wdesc &wd, const void *W, const uint8_t *gamma, int32_t *row_ptr,
                          int32_t *col_idx, void *payload, void *packed, int64_t capacity_blocks, void *ws,
                          cudaStream_t st)
{
    const int NBo = wd.O / wd.bo, NBi = wd.I / wd.bi, HK = wd.H * wd.K;
    const PackedLayout L = packed_layout(wd);
    int *status = (int *)ws;
    uint8_t *pk = (uint8_t *)packed;
    const bool dense_on = pk != nullptr && L.enabled;
    const int esz = elem_bytes(wd.wtype);

    CompactArgs a = {};
    a.W = W; a.gamma = gamma; a.O = wd.O; a.I = wd.I; a.HK = HK; a.bo = wd.bo; a.bi = wd.bi; a.NBo = NBo; a.NBi = NBi;
    a.row_ptr_out = row_ptr; a.col_idx = col_idx; a.payload = payload; a.capacity_blocks = capacity_blocks;
    a.dense = dense_on ? pk + L.off_payload : nullptr;
    a.hdr = (PackedHeader *)pk; a.status = status;
    PackedHeader &h = a.hdr_init;
    h.magic = kPackedMagic; h.dtype = wd.wtype; h.O = wd.O; h.I = wd.I; h.H = wd.H; h.K = wd.K; h.bo = wd.bo; h.bi = wd.bi;
    h.forms = dense_on ? kFormDense : 0; h.off_payload = (int64_t)L.off_payload;
    // packed form: a chunk of up to eight rows per thread and pass, at most 16 CTAs per SM's worth of CTAs
    const long long units = dense_on ? (long long)NBo * ((wd.bo * HK + kDenseRows - 1) / kDenseRows) * (wd.I * esz / 16) : 0;
    long long dg = (units + kThreads - 1) / kThreads;
    if (dg > 2368) dg = 2368;
    a.dense_ctas = dense_on ? (int)(dg < 1 ? 1 : dg) : (pk ? 1 : 0);      // (a packed buffer without the form still gets its header)
    const size_t smem = (size_t)NBi * sizeof(int);

    if ((long long)NBo * NBi <= kSmallBlocks) {
        // enough CTAs per row that a thread moves about four pieces of the canonical payload
        a.fill_parts = 1;
        if (payload) {
            const long long row_pieces = (long long)NBi * wd.bo * HK * ((wd.bi * esz + 15) / 16);   // a row with every block stored
            const long long p = (row_pieces / 2 + 4LL * kThreads - 1) / (4LL * kThreads);
            a.fill_parts = (int)(p < 1 ? 1 : (p > 8 ? 8 : p));
        }
        a.n_fill = NBo * a.fill_parts;
        const unsigned grid = (unsigned)(a.n_fill + a.dense_ctas);
        if (wd.wtype == BSP_I8) BSP_CUDA_OK(launch_after(compact_kernel<uint8_t, false>, dim3(grid), dim3(kThreads), smem, st, a));
        else if (wd.wtype == BSP_BF16) BSP_CUDA_OK(launch_after(compact_kernel<uint16_t, false>, dim3(grid), dim3(kThreads), smem, st, a));
        else BSP_CUDA_OK(launch_after(compact_kernel<uint32_t, false>, dim3(grid), dim3(kThreads), smem, st, a));
        return BSP_OK;
    }
    if ((long long)NBo * NBi > 0x7FFFFFFF) return BSP_ERR_SHAPE;
    // enough CTAs per row to give every SM some of the payload copy
    a.fill_parts = payload ? (296 + NBo - 1) / NBo : 1;
    if (a.fill_parts > 16) a.fill_parts = 16;
    if (a.fill_parts < 1) a.fill_parts = 1;
    a.n_fill = payload ? NBo * a.fill_parts : (NBo + kIndexRows - 1) / kIndexRows;
    const unsigned grid = (unsigned)(a.n_fill + a.dense_ctas);
    if (wd.wtype == BSP_I8) BSP_CUDA_OK(launch_after(compact_kernel<uint8_t, true>, dim3(grid), dim3(kThreads), smem, st, a));
    else if (wd.wtype == BSP_BF16) BSP_CUDA_OK(launch_after(compact_kernel<uint16_t, true>, dim3(grid), dim3(kThreads), smem, st, a));
    else BSP_CUDA_OK(launch_after(compact_kernel<uint32_t, true>, dim3(grid), dim3(kThreads), smem, st, a));
    return BSP_OK;
}

}  // namespace bsp
