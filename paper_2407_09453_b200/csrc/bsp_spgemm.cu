// Block-sparse x block-sparse product C = (Gamma . A)(Omega . B)^t on the compressed block rows of both operands, and the
// relative column index.  Section "Block-Sparse Matrix-Matrix Multiplication" and Section "Block Sparsity in a Matrix"
// ("a relative row/col index") of the paper.
//
// C_{i,j} = sum over the block columns k that row i of A and row j of B both keep of A_{i,k} B_{j,k}^t, 8 x 8 blocks.
// A CTA owns one row i of A: the positions of its kept blocks are spread into a table over the block columns in shared
// memory (the table replaces one side of the paper's merge of two sorted lists), and every warp takes rows j of B in
// turn: 32 entries of B's column list are looked up at once, a ballot gives the common columns in ascending order, and
// for each of them the warp adds the 8 x 8 x 8 product, lane (r, c) holding C[r][2c], C[r][2c + 1] in fp32 (fp32 blocks:
// fused multiply-adds; bfloat16 blocks: one m16n8k16 tensor-core instruction per two common columns).  Work and
// traffic follow the kept blocks only: nothing is read or multiplied where either mask has a zero.  bfloat16 operands whose
// masks leave enough common columns take the dense form on tcgen05 below, fp32 operands tiles of 64 x 64.
#include <math.h>
#include <atomic>
#include <mutex>
#include "bsp_tc.cuh"

namespace bsp {
namespace {

constexpr int kSpThreads = 256;
constexpr int kSpEdge = 8;

// Row kRow (from p on) of an 8 x 8 fp32 block.
template <int kRow>
__device__ __forceinline__ void sp_row(const float *p, float (&v)[8])
{
    const float4 a = load_free<kRow * 32>((const float4 *)p), b = load_free<kRow * 32 + 16>((const float4 *)p);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
// The 8 x 8 block of C of one row of A and one row of B: acc0, acc1 are this lane's entries (r, 2c), (r, 2c + 1) with
// r = lane / 4, c = lane % 4.  `pos_of` gives the payload position of the A row's block in column k, or -1.  The pointers come
// through from_here().
template <typename T, typename F>
__device__ __forceinline__ void sp_pair(const T *a_payload, const int32_t *b_col_idx, const T *b_payload,
                                        int lo, int hi, int NBk, int lane, F pos_of, float &acc0, float &acc1, int *status)
{
    const int r = lane >> 2, c = (lane & 3) * 2;
    for (int base = lo; base < hi; base += 32) {
        const int nb = base + lane;
        int pa = -1;
        if (nb < hi) {
            const int k = load_free(b_col_idx + nb);
            if (k >= 0 && k < NBk) pa = pos_of(k);
            else atomicMax(status, (int)BSP_ERR_INDEX);
        }
        unsigned both = __ballot_sync(0xFFFFFFFFu, pa >= 0);
        if constexpr (sizeof(T) == 2) {
            // bfloat16 blocks: two common columns per tensor-core instruction (m16n8k16: the 8 x 8 block of C sits in
            // rows 0-7 of the 16 x 8 result, K = the eight channels of the first column followed by those of the
            // second).  Lane (r, c) holds exactly the words it needs: entries (r, 2c), (r, 2c + 1) of each block of A
            // and of B, so a warp reads each 128-byte block once, four bytes per lane.
            while (both) {
                const int s1 = __ffs(both) - 1;
                both &= both - 1;
                const int s2 = both ? __ffs(both) - 1 : -1;
                both &= both - 1;                         // (0 & -1 stays 0)
                const int na1 = __shfl_sync(0xFFFFFFFFu, pa, s1);
                const int na2 = __shfl_sync(0xFFFFFFFFu, pa, s2 < 0 ? s1 : s2);
                const uint32_t *Aw = (const uint32_t *)a_payload, *Bw = (const uint32_t *)b_payload;
                const uint32_t a0 = load_free(Aw + (size_t)na1 * 32 + lane), b0 = load_free(Bw + (size_t)(base + s1) * 32 + lane);
                uint32_t a2 = 0u, b1 = 0u;
                if (s2 >= 0) { a2 = load_free(Aw + (size_t)na2 * 32 + lane); b1 = load_free(Bw + (size_t)(base + s2) * 32 + lane); }
                float d2 = 0.f, d3 = 0.f;
                asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};\n"
                             : "+f"(acc0), "+f"(acc1), "+f"(d2), "+f"(d3) : "r"(a0), "r"(0u), "r"(a2), "r"(0u), "r"(b0), "r"(b1));
            }
        } else
        while (both) {                                    // common columns, ascending
            const int src = __ffs(both) - 1;
            both &= both - 1;
            const int na = __shfl_sync(0xFFFFFFFFu, pa, src);
            const T *Ab = a_payload + ((size_t)na * kSpEdge + r) * kSpEdge;
            const T *Bb = b_payload + ((size_t)(base + src) * kSpEdge + c) * kSpEdge;
            float av[8], b0[8], b1[8];
            sp_row<0>(Ab, av); sp_row<0>(Bb, b0); sp_row<1>(Bb, b1);
#pragma unroll
            for (int t = 0; t < kSpEdge; ++t) {
                acc0 = fmaf(av[t], b0[t], acc0);
                acc1 = fmaf(av[t], b1[t], acc1);
            }
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(kSpThreads)
spgemm_kernel(const int32_t *a_row_ptr, const int32_t *a_col_idx, const T *a_payload,
              const int32_t *b_row_ptr, const int32_t *b_col_idx, const T *b_payload,
              int NBb, int NBk, float *C, int *status)
{
    extern __shared__ int s_pos[];                 // [NBk]: payload position of row i's block in column k, or -1
    const int i = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = threadIdx.x; k < NBk; k += kSpThreads) s_pos[k] = -1;
    // (The next kernel is not let in before this one has ended: its CTAs, several per SM, would be placed where slots happen to be
    // free and stay uneven.  A stream of 1768 x 208 x 992 bfloat16 products at 50 % takes 10.0 us a call like this, 13.4 with the
    // next one let in at once, 12.2 without programmatic launches; 232 x 2264 x 632 fp32 at 25 % 62.0, 78.1 let in at the end of
    // each CTA, 64.3.)
    wait_for_previous<false>();
    a_payload = from_here(a_payload); a_col_idx = from_here(a_col_idx); a_row_ptr = from_here(a_row_ptr);
    b_payload = from_here(b_payload); b_col_idx = from_here(b_col_idx); b_row_ptr = from_here(b_row_ptr);
    __syncthreads();
    const int a_end = load_free(a_row_ptr + i + 1);
    for (int n = load_free(a_row_ptr + i) + threadIdx.x; n < a_end; n += kSpThreads) {
        const int k = load_free(a_col_idx + n);
        if (k >= 0 && k < NBk) s_pos[k] = n;
        else atomicMax(status, (int)BSP_ERR_INDEX);          // a column outside the matrix: skipped
    }
    __syncthreads();
    const int r = lane >> 2, c = (lane & 3) * 2;             // this lane's two entries of the 8 x 8 block of C
    const size_t ldc = (size_t)NBb * kSpEdge;
    for (int j = blockIdx.y * (kSpThreads / 32) + warp; j < NBb; j += gridDim.y * (kSpThreads / 32)) {
        float acc0 = 0.f, acc1 = 0.f;
        sp_pair<T>(a_payload, b_col_idx, b_payload, load_free(b_row_ptr + j), load_free(b_row_ptr + j + 1), NBk, lane, [&](int k) { return s_pos[k]; }, acc0, acc1, status);
        *(float2 *)(C + ((size_t)i * kSpEdge + r) * ldc + (size_t)j * kSpEdge + c) = make_float2(acc0, acc1);
    }
}

// ---- fp32 operands, tiles of 64 x 64 ------------------------------------------------------------------------------------
// The kernel above reads six 16-byte pieces through L1 for every 16 fused multiply-adds of a thread, which bounds it.  Here a CTA owns
// eight block rows of A x eight of B.  It walks the block columns in chunks of four: the kept blocks of both are loaded a chunk ahead into
// registers and written to shared memory transposed, so that a thread, which owns 4 x 4 sums, reads four rows of A and four of B at one
// column with one 16-byte load each.  A warp owns one block row of A: it passes by the columns that this row dropped, and a lane
// those that its row of B dropped; nothing is multiplied where either mask has a zero, and the terms of a sum are added in the same order
// (ascending columns, fused) as above, so that both give the same bits.
constexpr int kSfThreads = 256;
constexpr int kSfRows = 8;                        // block rows of A, and of B, per tile
constexpr int kSfChunk = 4;                       // block columns per chunk
constexpr int kSfPitch = 8 * 64 + 16;             // floats of one block column of a chunk: [channel][row of the tile] (+ 16: the stores of two columns take different banks)
constexpr int kSfMaxCols = 1024;                  // block columns (positions of 16 rows in 32 KB)
struct SfShared {
    float tile[2][2][kSfChunk * kSfPitch];        // [buffer][A, B]
};

__global__ void __launch_bounds__(kSfThreads, 2)
spgemm_f32_kernel(const int32_t *a_row_ptr, const int32_t *a_col_idx, const float *a_payload,
                  const int32_t *b_row_ptr, const int32_t *b_col_idx, const float *b_payload,
                  int NBa, int NBb, int NBk, float *C, int *status)
{
    __shared__ __align__(16) SfShared sh;
    extern __shared__ __align__(16) int16_t sf_pos[];          // [16][pitch]: position within its row's stored blocks, or -1
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int i0 = (int)blockIdx.y * kSfRows, j0 = (int)blockIdx.x * kSfRows;
    const int n_chunks = (NBk + kSfChunk - 1) / kSfChunk, pitch = n_chunks * kSfChunk;
    for (int k = tid; k < 2 * kSfRows * pitch / 4; k += kSfThreads) ((uint2 *)sf_pos)[k] = make_uint2(~0u, ~0u);
    wait_for_previous<false>();                                // (the next kernel starts when this one has ended, as above)
    a_payload = from_here(a_payload); a_col_idx = from_here(a_col_idx); a_row_ptr = from_here(a_row_ptr);
    b_payload = from_here(b_payload); b_col_idx = from_here(b_col_idx); b_row_ptr = from_here(b_row_ptr);
    __syncthreads();
    auto row_of = [&](int b, int &lo, int &hi) {               // a block row's first and last stored block (rows past the last one are empty)
        const bool is_a = b < kSfRows;
        const int g = is_a ? i0 + b : j0 + b - kSfRows;
        const int32_t *rp = is_a ? a_row_ptr : b_row_ptr;
        const bool in = g < (is_a ? NBa : NBb);
        lo = in ? load_free(rp + g) : 0;
        hi = in ? load_free(rp + g + 1) : 0;
    };
    for (int b = warp; b < 2 * kSfRows; b += kSfThreads / 32) {
        int lo, hi;
        row_of(b, lo, hi);
        const int32_t *ci = b < kSfRows ? a_col_idx : b_col_idx;
        for (int n = lo + lane; n < hi; n += 32) {
            const int k = load_free(ci + n);
            if (k >= 0 && k < NBk) sf_pos[b * pitch + k] = (int16_t)(n - lo);
            else atomicMax(status, (int)BSP_ERR_INDEX);        // a column outside the matrix: skipped
        }
    }
    __syncthreads();
    // loads: four threads per block of the chunk, two rows of it each
    const int lb = tid >> 4, lk = (tid >> 2) & 3, lr = (tid & 3) * 2;
    int first, last;
    row_of(lb, first, last);
    const float *src = (lb < kSfRows ? a_payload : b_payload) + (size_t)first * 64 + lr * 8;
    float4 v[4];
    auto load = [&](int c) {
        const int n = c < n_chunks ? sf_pos[lb * pitch + c * kSfChunk + lk] : -1;
        if (n >= 0) {
            const float4 *p = (const float4 *)(src + (size_t)n * 64);
            v[0] = load_free(p); v[1] = load_free(p + 1); v[2] = load_free(p + 2); v[3] = load_free(p + 3);
        }
    };
    const int at = lk * kSfPitch + (lb & 7) * 8 + lr;
    auto put = [&](int buf) {                                  // (what a dropped block leaves there is not read)
        float *t = sh.tile[buf][lb >> 3] + at;
        const float lo8[8] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w};
        const float hi8[8] = {v[2].x, v[2].y, v[2].z, v[2].w, v[3].x, v[3].y, v[3].z, v[3].w};
#pragma unroll
        for (int q = 0; q < 8; ++q) *(float2 *)(t + q * 64) = make_float2(lo8[q], hi8[q]);
    };
    v[0] = v[1] = v[2] = v[3] = make_float4(0.f, 0.f, 0.f, 0.f);
    load(0);
    float acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = 0.f;
    const int ay = warp * 8 + (lane >> 4) * 4, bx = (lane & 15) * 4;
    const int16_t *pos_a = sf_pos + warp * pitch, *pos_b = sf_pos + (kSfRows + ((lane & 15) >> 1)) * pitch;
    for (int c = 0; c < n_chunks; ++c) {
        const int buf = c & 1;
        put(buf);
        load(c + 1);
        const short4 na = *(const short4 *)(pos_a + c * kSfChunk), nb = *(const short4 *)(pos_b + c * kSfChunk);
        __syncthreads();                                       // (buffers are written two chunks apart: one barrier a chunk)
        const short ka[4] = {na.x, na.y, na.z, na.w}, kb[4] = {nb.x, nb.y, nb.z, nb.w};
#pragma unroll
        for (int k = 0; k < kSfChunk; ++k) {
            if (ka[k] < 0 || kb[k] < 0) continue;
            const float *pa = sh.tile[buf][0] + k * kSfPitch + ay, *pb = sh.tile[buf][1] + k * kSfPitch + bx;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float4 a = *(const float4 *)(pa + q * 64), b = *(const float4 *)(pb + q * 64);
                const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int t = 0; t < 4; ++t) acc[r][t] = fmaf(av[r], bv[t], acc[r][t]);
            }
        }
    }
    const size_t ldc = (size_t)NBb * kSpEdge;
    const int row = i0 * kSpEdge + ay, col = j0 * kSpEdge + bx;
    if (row < NBa * kSpEdge && col < NBb * kSpEdge) {
        const bool wide = ((uintptr_t)C & 15u) == 0;           // (rows of C are multiples of 32 bytes)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            float *dst = C + (size_t)(row + r) * ldc + col;
            if (wide) *(float4 *)dst = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
            else { *(float2 *)dst = make_float2(acc[r][0], acc[r][1]); *(float2 *)(dst + 2) = make_float2(acc[r][2], acc[r][3]); }
        }
    }
}

// ---- bfloat16 operands on 5th-generation tensor cores -----------------------------------------------------------------
// A CTA owns 128 rows of A (16 block rows) x BN rows of B (BN = 64, 128 or 256), or with split reductions a share of the
// columns of such a tile.  The payload positions of its block rows are spread into a table over the block columns in
// shared memory; then 16 producer warps walk the columns in chunks of eight blocks (64 values, the span of the 128-byte
// swizzle), in groups that take turns: the 8 rows of a kept block are 16 bytes each, one per lane, loaded ahead and written
// straight into the swizzled operand layout, dropped blocks as zeros; one warp issues the four MMAs of a chunk into one
// accumulator of BN columns.  Zeroed blocks are multiplied, but nothing is read for them.
// A dropped block must not turn a non-finite weight into NaN (0 * inf): a piece of C whose sums are not all finite is
// computed again by the sparse form.
constexpr int kStProducers = 16;
constexpr int kStFencers = 2;                     // (pairs)
__host__ __device__ constexpr int st_threads(bool pair) { return (kStProducers + 1 + (pair ? kStFencers : 0)) * 32; }
constexpr int kStMaxStages = 8;
constexpr int kStARows = kGtBM / kSpEdge;         // block rows of A per tile

// Groups of producer warps by tile width: a group's chain of wait, store, arrive and load is longer than the MMAs of
// a chunk, so groups overlap theirs.  2048 x 2048 x 4096 at 50 %, us: one group 52 / 82 / 130 (256 / 128 / 64 columns), two
// 50 / 72 / 113, four 105 with 64; 16-byte cp.async straight to shared memory instead of registers: 72 / 93 / 143.  (These with
// a proxy fence in the producers, all in short bursts with the same operands; a call in a stream with operands that change
// takes 51 with 256 columns.)
__host__ __device__ constexpr int st_groups(int BN) { return BN == 64 ? 4 : 2; }

struct StParams {
    const int32_t *a_row_ptr, *a_col_idx, *b_row_ptr, *b_col_idx;
    const uint8_t *a_payload, *b_payload;
    float *C;
    int *status;
    int NBa, NBb, NBk, n_chunks, stages, split;
};

// kPair (BN = 256): the tiles of 2 x 128 rows of A and the same 256 rows of B are taken by a cluster of two CTAs; each fills its own rows of A
// and half of those of B, and MMAs with M = 256 over the pair read both halves.  A CTA then writes and its MMAs read 32 KB a chunk
// instead of 48.  The proxy fence between a chunk's stores and its MMAs, about 700 cycles beside the producers' traffic, is taken by warps of
// its own, ahead of the MMA warp, which had stood still for it: 2048 x 2048 x 4096 at 50 % in a stream of calls 51.0 us alone, 51.6 as
// pairs with the fence in the MMA warp, 41.7 with two warps that fence, 43.9 with three, 47.3 with six (a fence holds up the producers'
// loads and stores), 42.4 with one that fences every second chunk; on single CTAs warps that fence made it 54.
__host__ __device__ constexpr int st_rows(int BN, bool pair) { return kStARows + BN / kSpEdge / (pair ? 2 : 1); }   // block rows that a CTA fills
template <int BN, bool kPair>
__global__ void __launch_bounds__(st_threads(kPair), 1) spgemm_tc_kernel(const __grid_constant__ StParams p)
{
    constexpr int kGroups = st_groups(BN), kDepth = BN == 128 ? 2 : 1;    // (chunks loaded ahead per group: what 120 registers hold)
    constexpr int kRows = st_rows(BN, kPair);                 // block rows of the tile: 16 of A, then those of B
    constexpr int kThreads = st_threads(kPair);
    constexpr int kW = kStProducers / kGroups;                // warps of a group: they share a chunk
    constexpr int kUnits = kRows * 2 / kW;                    // half block rows (four blocks of a chunk) per warp
    constexpr uint32_t kStage = kRows * 1024u;                // a block row of a chunk: 8 rows of 128 bytes
    extern __shared__ __align__(16) uint8_t st_smem_raw[];
    uint8_t *smem = st_smem_raw + ((1024u - (sm32(st_smem_raw) & 1023u)) & 1023u);
    __shared__ __align__(8) uint64_t s_full[kStMaxStages], s_ready[kStMaxStages], s_empty[kStMaxStages], s_acc;
    __shared__ uint32_t s_tmem;
    __shared__ volatile uint32_t s_fail;
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    const int S = p.stages, pitch = p.n_chunks * 8;
    const uint32_t ring = sm32(smem);
    int16_t *s_pos = (int16_t *)(smem + (size_t)S * kStage);  // [kRows][pitch]: position within its row's stored blocks, or -1
    uint32_t rank = 0;
    if constexpr (kPair) asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(rank));
    const int i0 = (kPair ? (int)(blockIdx.y * 2 + rank) : (int)blockIdx.y) * kStARows, j0 = (kPair ? (int)(blockIdx.x >> 1) : (int)blockIdx.x) * (BN / kSpEdge);
    const int jb0 = j0 + (int)rank * (kRows - kStARows);      // the first row of B that this CTA fills
    // this CTA's chunks: all of them, or its share of a split reduction (the CTAs of a tile are a cluster along z)
    const int share = (p.n_chunks + p.split - 1) / p.split;
    const int c_lo = (int)blockIdx.z * share, c_hi = min(p.n_chunks, c_lo + share);

    if (tid == 0) {
        s_fail = 0u;
        for (int s = 0; s < S; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&s_full[s])), "r"(kW) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&s_ready[s])), "r"(2) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&s_empty[s])), "r"(1) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&s_acc)), "r"(1) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == kStProducers) {
        if constexpr (kPair) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(sm32(&s_tmem)), "r"(BN) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(sm32(&s_tmem)), "r"(BN) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
        }
    }
    wait_for_previous<false>();
    if (warp == kStProducers) let_next_start();        // (behind its allocation)
    // a block row's first and last stored block (rows past the last one are empty)
    auto row_of = [&](int b, int &lo, int &hi) {
        const bool is_a = b < kStARows;
        const int g = is_a ? i0 + b : jb0 + b - kStARows;
        const int32_t *rp = is_a ? p.a_row_ptr : p.b_row_ptr;
        const bool in = g < (is_a ? p.NBa : p.NBb);
        lo = in ? rp[g] : 0;
        hi = in ? rp[g + 1] : 0;
    };
    for (int k = tid; k < kRows * pitch / 8; k += kThreads) ((uint4 *)s_pos)[k] = make_uint4(~0u, ~0u, ~0u, ~0u);
    __syncthreads();
    for (int b = warp; b < kRows; b += kThreads / 32) {
        int lo, hi;
        row_of(b, lo, hi);
        const int32_t *ci = b < kStARows ? p.a_col_idx : p.b_col_idx;
        for (int n = lo + lane; n < hi; n += 128) {
            int k[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) k[u] = n + 32 * u < hi ? ci[n + 32 * u] : 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (n + 32 * u >= hi) continue;
                if (k[u] >= 0 && k[u] < p.NBk) s_pos[b * pitch + k[u]] = (int16_t)(n + 32 * u - lo);
                else atomicMax(p.status, (int)BSP_ERR_INDEX);          // a column outside the matrix: skipped
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    gt_sync_all<kPair>();                   // (a pair: both CTAs' barriers are initialised before either signals the other)
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, s_tmem, 0);
    const uint32_t full0 = sm32(&s_full[0]), empty0 = sm32(&s_empty[0]);

    if (warp < kStProducers) {
        // ================= producers =================
        // Group g takes every kGroups-th chunk.  Unit u of a warp: a half (four blocks) of block row b0 + (kW / 2) u;
        // lane = row q of block j of the chunk.
        const int grp = warp / kW, wg = warp % kW;
        const int q = lane & 7, j = (wg & 1) * 4 + (lane >> 3), b0 = wg >> 1;
        const uint8_t *src[kUnits];
        const int16_t *pos = s_pos + b0 * pitch + j;
#pragma unroll
        for (int u = 0; u < kUnits; ++u) {
            int lo, hi;
            row_of(b0 + (kW / 2) * u, lo, hi);
            src[u] = (u < 2 * kStARows / kW ? p.a_payload : p.b_payload) + (size_t)lo * 128 + q * 16;
        }
        const uint32_t off = (uint32_t)(b0 * 1024 + q * 128 + ((j ^ q) << 4));
        uint4 v[kDepth][kUnits];
        auto load = [&](int c, uint4 (&w)[kUnits]) {
            if (c >= c_hi) return;
#pragma unroll
            for (int u = 0; u < kUnits; ++u) {
                const int n = pos[(kW / 2) * u * pitch + c * 8];
                w[u] = make_uint4(0u, 0u, 0u, 0u);
                if (n >= 0) w[u] = *(const uint4 *)(src[u] + (size_t)n * 128);
            }
        };
        uint32_t slot = (uint32_t)grp, epar = 1;               // (a fresh barrier counts as released)
        bool ok = true;
        auto put = [&](const uint4 (&w)[kUnits]) {
            if (!gt_wait(empty0 + slot * 8u, epar)) ok = false;
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) return;
            const uint32_t dst = ring + slot * kStage + off;
#pragma unroll
            for (int u = 0; u < kUnits; ++u)
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(dst + u * (uint32_t)(kW * 512)), "r"(w[u].x), "r"(w[u].y), "r"(w[u].z), "r"(w[u].w) : "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(full0 + slot * 8u) : "memory");
            slot += kGroups;
            if (slot >= (uint32_t)S) { slot -= (uint32_t)S; epar ^= 1u; }
        };
#pragma unroll
        for (int d = 0; d < kDepth; ++d) load(c_lo + grp + d * kGroups, v[d]);
        for (int c = c_lo + grp; c < c_hi && ok; c += kDepth * kGroups)
#pragma unroll
            for (int d = 0; d < kDepth; ++d)
                if (c + d * kGroups < c_hi && ok) {
                    put(v[d]);
                    load(c + (d + kDepth) * kGroups, v[d]);
                }
        if (!gt_wait(sm32(&s_acc), 0u)) ok = false;
        if (!__all_sync(0xFFFFFFFFu, ok) && lane == 0) atomicExch((uint32_t *)&s_fail, 1u);
    } else if (kPair && warp > kStProducers) {
        // ================= fences of a pair =================
        // Two warps take turns with the chunks: wait until one is full, fence, pass it on to the MMA warp of the pair's leader.  (They meet
        // every second slot of a ring of an even number of stages, so that no other chunk passes a barrier between two of their looks.)
        const uint32_t first = (uint32_t)(warp - kStProducers - 1);
        uint32_t ready0, slot = first, par = 0;
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;\n" : "=r"(ready0) : "r"(sm32(&s_ready[0])));
        bool ok = true;
        for (int c = c_lo + (int)first; c < c_hi; c += kStFencers) {
            if (!__all_sync(0xFFFFFFFFu, gt_poll(full0 + slot * 8u, par))) { ok = false; break; }
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];\n" ::"r"(ready0 + slot * 8u) : "memory");
            slot += kStFencers;
            if (slot >= (uint32_t)S) { slot -= (uint32_t)S; par ^= 1u; }
        }
        if (!ok && lane == 0) atomicExch((uint32_t *)&s_fail, 1u);
    } else if (rank == 0) {
        // ================= MMA issuer (of a pair, the leader's issues for both CTAs) =================
        const uint32_t ready0 = kPair ? sm32(&s_ready[0]) : full0;
        constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | (((kPair ? 256u : 128u) >> 4) << 24);
        uint32_t slot = 0, par = 0, a16 = ring >> 4;
        bool ok = true, full_now = false;
        for (int c = c_lo; c < c_hi; ++c) {
            if (!full_now && !gt_poll_stage(ready0 + slot * 8u, par)) { ok = false; break; }
            const bool wrap = slot + 1u == (uint32_t)S;
            // (the stage's stores come before this thread through its barrier, and before the MMAs by this one fence: a fence in
            // every producer also waited for the loads it had in flight; 2048 x 2048 x 4096 at 50 % 48.9 -> 46.0 us in a burst)
            if constexpr (!kPair) {
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            }
            full_now = gt_issue_stage<BSP_BF16, kPair>(tmem, kGtDesc | (uint64_t)(a16 & 0x3FFFu), kGtDesc | (uint64_t)((a16 + (kGtABytes >> 4)) & 0x3FFFu),
                                                       idesc, empty0 + slot * 8u, c != c_lo ? 1u : 0u, 4u, ready0 + (wrap ? 0u : slot + 1u) * 8u, wrap ? par ^ 1u : par) != 0u;
            if (wrap) { slot = 0; par ^= 1u; a16 = ring >> 4; } else { ++slot; a16 += kStage >> 4; }
        }
        if (ok) gt_commit_elected<kPair>(sm32(&s_acc));
        else if (lane == 0) atomicExch((uint32_t *)&s_fail, 1u);
    }
    __syncthreads();
    const bool ok = (s_fail & 1u) == 0u;

    // ================= epilogue =================
    // The tile is cut into pieces of 32 x 32 sums (piece = 32-column part * 4 + quarter of the tensor-memory lanes), which go
    // through 4 KB of the idle ring each, so that rows of C are written 128 bytes at a time.
    constexpr int kPieces = BN / 8;
    const bool wide = ((uintptr_t)p.C & 15u) == 0;         // (rows of C are multiples of 32 bytes)
    const size_t ldc = (size_t)p.NBb * kSpEdge;
    auto to_smem = [&](int piece) {
        uint32_t w[32];
        gt_load32(tmem + ((uint32_t)((piece & 3) * 32) << 16) + (uint32_t)(piece >> 2) * 32u, w);
        const uint32_t buf = ring + (uint32_t)piece * 4096u + lane * 128u;
#pragma unroll
        for (int e = 0; e < 8; ++e)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(buf + (uint32_t)((e ^ (lane & 7)) << 4)), "r"(w[4 * e]), "r"(w[4 * e + 1]), "r"(w[4 * e + 2]), "r"(w[4 * e + 3]) : "memory");
    };
    // sums the shares of a piece in the order of the CTAs (`peers` of them) and writes it
    auto to_global = [&](int piece, int peers) {
        const int row0 = i0 * kSpEdge + (piece & 3) * 32, col = j0 * kSpEdge + (piece >> 2) * 32 + (lane & 7) * 4;
        const uint32_t buf = ring + (uint32_t)piece * 4096u;
        bool odd = false;                                      // a sum that is not finite
#pragma unroll
        for (int it = 0; it < 8; ++it) {
            const int r = it * 4 + (lane >> 3);
            const uint32_t at = buf + r * 128u + (uint32_t)(((lane & 7) ^ (r & 7)) << 4);
            float4 x;
            if (peers == 1) {
                asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "r"(at) : "memory");
            } else {
                x = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int k = 0; k < peers; ++k) {
                    uint32_t far;
                    float4 y;
                    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(far) : "r"(at), "r"(k));
                    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];\n" : "=f"(y.x), "=f"(y.y), "=f"(y.z), "=f"(y.w) : "r"(far) : "memory");
                    x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w;
                }
            }
            odd |= !(isfinite(x.x) && isfinite(x.y) && isfinite(x.z) && isfinite(x.w));
            if (row0 + r < p.NBa * kSpEdge && col < p.NBb * kSpEdge) {
                float *dst = p.C + (size_t)(row0 + r) * ldc + col;
                if (wide) *(float4 *)dst = x;
                else { *(float2 *)dst = make_float2(x.x, x.y); *(float2 *)(dst + 2) = make_float2(x.z, x.w); }
            }
        }
        if (!__any_sync(0xFFFFFFFFu, odd)) return;
        for (int t = 0; t < 16; ++t) {
            const int bi = (piece & 3) * 4 + (t & 3), i = i0 + bi, jj = j0 + (piece >> 2) * 4 + (t >> 2);
            if (i >= p.NBa || jj >= p.NBb) continue;
            float acc0 = 0.f, acc1 = 0.f;
            const int first = p.a_row_ptr[i];
            const int16_t *row = s_pos + bi * pitch;
            sp_pair<__nv_bfloat16>(from_here((const __nv_bfloat16 *)p.a_payload), from_here(p.b_col_idx), from_here((const __nv_bfloat16 *)p.b_payload), p.b_row_ptr[jj], p.b_row_ptr[jj + 1],
                                   p.NBk, lane, [&](int k) { const int n = row[k]; return n < 0 ? -1 : first + n; }, acc0, acc1, p.status);
            *(float2 *)(p.C + ((size_t)i * kSpEdge + (lane >> 2)) * ldc + (size_t)jj * kSpEdge + (lane & 3) * 2) = make_float2(acc0, acc1);
        }
    };
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (p.split == 1) {
        if (ok && warp < kStProducers)
            for (int piece = warp; piece < kPieces; piece += kStProducers) { to_smem(piece); __syncwarp(); to_global(piece, 1); }
    } else {
        if (ok && warp < kStProducers)
            for (int piece = warp; piece < kPieces; piece += kStProducers) to_smem(piece);
        gt_sync_all<true>();
        if (ok && warp < kStProducers)
            for (int piece = (int)blockIdx.z + p.split * warp; piece < kPieces; piece += p.split * kStProducers) to_global(piece, p.split);
        gt_sync_all<true>();                                   // (no CTA leaves while another still reads its sums)
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    gt_sync_all<kPair>();                   // (a pair: neither CTA leaves while the other may still signal its barriers)
    if (!ok && tid == 0) atomicMax(p.status, (int)BSP_ERR_TIMEOUT);
    if (warp == kStProducers) {
        if constexpr (kPair) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(BN) : "memory");
        else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(BN) : "memory");
    }
}

// Stages that fit beside the position table of a tile (zero: too many block columns).
int spgemm_tc_stages(int BN, int n_chunks, bool pair = false)
{
    const long long rows = st_rows(BN, pair);
    const long long room = (long long)kGtMaxSmem - 1024 - rows * n_chunks * 16;
    const long long n = room / (rows * 1024);
    const int stages = n < 0 ? 0 : (n > kStMaxStages ? kStMaxStages : (int)n);
    return pair ? stages / kStFencers * kStFencers : stages;
}

// Tile width and split of the tensor-core form, or BN = 0 where the sparse form is expected to be faster.  Estimates in
// microseconds, fitted on a B200.  Tensor-core form: a tile costs a start, a share per chunk for the table and the fill of
// the operands (0.30 / 0.42 / 0.57 a chunk at 64 / 128 / 256 columns, bound by shared memory: stores of the fill, reads
// of the MMAs; 0.49 on pairs of 2 x 128 rows and 256 columns), whatever the masks hold.  Sparse form: 28.7 per million pairs of blocks with a common column plus 3.6 per
// million look-ups, or the chain of one warp where there are few rows.  Measured in bursts, sparse / tensor core: 2048 x 2048 x 4096
// at 50 % 304 / 46, at 75 % 90 / 43, 512 x 512 x 4096 at 50 % 27 / 14; with the fence in the
// producers 25 / 44 at 90 %, and 11 / 14 for the smaller one at 75 %.
// The densities come from the host counts; a wrong count costs time only.
struct StPlan { int BN, split, pair; };
// What the choice needs to know of a GPU.  slots[k] = CTAs of clusters of 2^k that it holds at once (clusters of eight do not reach every
// SM: 512 x 512 x 4096 on 16 of them took two waves, 28.5 us, against 15.3 on 32 clusters of four); pair_slots = those of pairs.
struct StDevice { int slots[4], pair_slots; };
StPlan spgemm_plan(int NBa, int NBb, int NBk, long long nnz_a, long long nnz_b, int gy, const StDevice &gpu)
{
    const int(&slots)[4] = gpu.slots;
    auto density = [](long long nnz, double nb) { return nnz <= 0 ? 0.0 : (nnz >= nb ? 1.0 : nnz / nb); };
    const double da = density(nnz_a, (double)NBa * NBk), db = density(nnz_b, (double)NBb * NBk);
    const double common = NBk * da * db, lookups = NBk * db;
    const double rows = (NBb + gy * (kSpThreads / 32) - 1) / (gy * (kSpThreads / 32));
    const double pairs = (double)NBa * NBb;
    const double bulk = pairs * (28.7e-6 * common + 3.6e-6 * lookups), chain = rows * (0.14 * common + 0.3 * (int)(lookups / 32 + 1));
    double best = 0.95 * (2.9 + (bulk > chain ? bulk : chain));
    StPlan plan = {0, 1, 0};
    const int n_chunks = (NBk + 7) / 8;
    // (the row tiles of A are the grid's y extent, which ends at 65535; the sparse form has a row of A per CTA along x)
    if ((NBa + kStARows - 1) / kStARows > 65535) return plan;
    for (int w = 0; w < 3; ++w) {
        const int BN = 64 << w;
        const int stages = spgemm_tc_stages(BN, n_chunks);
        if (stages < (BN == 256 ? 3 : st_groups(BN))) continue;        // (the ring also holds the tile's sums)
        const double start = w == 0 ? 5.7 : (w == 1 ? 6.4 : 9.0), chunk = w == 0 ? 0.30 : (w == 1 ? 0.42 : 0.57);
        const long long tiles = (long long)((NBa + kStARows - 1) / kStARows) * ((NBb * kSpEdge + BN - 1) / BN);
        for (int k = 0; k < 4 && slots[k] > 0; ++k) {
            const int split = 1 << k;
            const int share = (n_chunks + split - 1) / split;
            if ((split - 1) * share >= n_chunks) break;                // (every CTA of a split has at least one chunk)
            const long long waves = (tiles * split + slots[k] - 1) / slots[k];
            const double t = waves * (start + 0.03 * n_chunks + chunk * share) + (split > 1 ? 2.5 : 0.0);
            if (t < best) { best = t; plan = {BN, split, 0}; }
        }
    }
    if (spgemm_tc_stages(256, n_chunks, true) >= 4 && gpu.pair_slots > 0) {
        const long long tiles = 2ll * ((NBa + 2 * kStARows - 1) / (2 * kStARows)) * ((NBb * kSpEdge + 255) / 256);
        const double t = (double)((tiles + gpu.pair_slots - 1) / gpu.pair_slots) * (9.4 + 0.03 * n_chunks + 0.49 * n_chunks);
        if (t < best) { best = t; plan = {256, 1, 1}; }
    }
    return plan;
}

// Whether fp32 operands take the kernel on tiles.  Estimates in microseconds, fitted on a B200.  By rows of A: 174 per million pairs of blocks
// with a common column, 3.6 per million look-ups.  On tiles: every chunk of four columns costs a start and the columns that the rows
// of A kept, twice as much where two CTAs share an SM.  us, rows / tiles: 1024 x 1024 x 2048 at 25 % 408 / 135, at 50 % 183 / 99, at 75 %
// 49 / 62; 232 x 2048 x 632 at 25 % 76 / 26; 2048 x 2048 x 1024 at 50 % 387 / 174, at 90 % 25 / 75; 512 x 512 x 1024 at 25 % 55 / 42, at 50 % 28 / 32.
bool spgemm_f32_tiles(int NBa, int NBb, int NBk, long long nnz_a, long long nnz_b, int n_sm)
{
    auto density = [](long long nnz, double nb) { return nnz <= 0 ? 0.0 : (nnz >= nb ? 1.0 : nnz / nb); };
    const double da = density(nnz_a, (double)NBa * NBk), db = density(nnz_b, (double)NBb * NBk), pairs = (double)NBa * NBb;
    const double by_rows = 2.9 + pairs * NBk * db * (174e-6 * da + 3.6e-6);
    const double ctas = (double)((NBa + kSfRows - 1) / kSfRows) * ((NBb + kSfRows - 1) / kSfRows), chunks = (NBk + kSfChunk - 1) / kSfChunk;
    const double on_tiles = 4.0 + chunks * (ctas <= n_sm ? 0.35 + 1.12 * da : ceil(ctas / (2.0 * n_sm)) * (0.45 + 2.1 * da));
    return on_tiles * 1.1 < by_rows;
}

// Per device, once: the kernels' shared-memory limit and what spgemm_plan needs.  Calls come from any thread: who finds the
// flag set finds the rest, too.
bsp_status spgemm_tc_device(const StDevice **gpu)
{
    static StDevice known[kGtMaxDevices] = {};
    static std::atomic<bool> done[kGtMaxDevices] = {};
    static std::mutex once;
    int dev = 0;
    BSP_CUDA_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kGtMaxDevices) return BSP_ERR_CUDA;
    if (!done[dev].load(std::memory_order_acquire)) {
        const std::lock_guard<std::mutex> lock(once);
        BSP_CUDA_OK(cudaFuncSetAttribute(spgemm_tc_kernel<64, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGtMaxSmem));
        BSP_CUDA_OK(cudaFuncSetAttribute(spgemm_tc_kernel<128, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGtMaxSmem));
        BSP_CUDA_OK(cudaFuncSetAttribute(spgemm_tc_kernel<256, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGtMaxSmem));
        BSP_CUDA_OK(cudaFuncSetAttribute(spgemm_tc_kernel<256, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGtMaxSmem));
        for (int k = 0; k < 5; ++k) {                                  // (the last: pairs)
            const bool pair = k == 4;
            cudaLaunchAttribute attr[1];
            cudaLaunchConfig_t cfg = {};
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = pair ? 2 : 1; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = pair ? 1 : 1u << k;
            cfg.attrs = attr; cfg.numAttrs = 1;
            cfg.gridDim = pair ? dim3(2) : dim3(1, 1, 8); cfg.blockDim = dim3(st_threads(pair)); cfg.dynamicSmemBytes = kGtMaxSmem;
            int n = 0;
            BSP_CUDA_OK(cudaOccupancyMaxActiveClusters(&n, pair ? spgemm_tc_kernel<256, true> : spgemm_tc_kernel<64, false>, &cfg));
            (pair ? known[dev].pair_slots : known[dev].slots[k]) = pair ? 2 * n : n << k;
        }
        done[dev].store(true, std::memory_order_release);
    }
    *gpu = &known[dev];
    return BSP_OK;
}

// The same for the fp32 tiles: the kernel's limit, then the number of SMs.  (Two first calls do the same thing twice.)
bsp_status spgemm_f32_device(int *n_sm)
{
    static std::atomic<int> known[kGtMaxDevices] = {};
    int dev = 0;
    BSP_CUDA_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kGtMaxDevices) return BSP_ERR_CUDA;
    *n_sm = known[dev].load(std::memory_order_acquire);
    if (*n_sm == 0) {
        BSP_CUDA_OK(cudaFuncSetAttribute(spgemm_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kSfRows * kSfMaxCols * (int)sizeof(int16_t)));
        BSP_CUDA_OK(cudaDeviceGetAttribute(n_sm, cudaDevAttrMultiProcessorCount, dev));
        known[dev].store(*n_sm, std::memory_order_release);
    }
    return BSP_OK;
}

template <int BN, bool kPair = false>
bsp_status launch_spgemm_tc(StParams p, cudaStream_t st)
{
    constexpr int kRows = st_rows(BN, kPair);
    p.stages = spgemm_tc_stages(BN, p.n_chunks, kPair);
    unsigned nx = (unsigned)((p.NBb * kSpEdge + BN - 1) / BN), ny = (unsigned)((p.NBa + kStARows - 1) / kStARows);
    if (kPair) { nx *= 2; ny = (ny + 1) / 2; }
    const size_t smem = 1024 + (size_t)kRows * p.n_chunks * 16 + (size_t)p.stages * kRows * 1024;
    BSP_CUDA_OK(launch_after_clusters(spgemm_tc_kernel<BN, kPair>, dim3(nx, ny, (unsigned)p.split), dim3(st_threads(kPair)), smem, st, kPair ? 2 : 1, p.split, p));
    return BSP_OK;
}

// One thread per row of Gamma: the first kept block keeps its column, the others store the distance to their predecessor.
__global__ void index_to_relative_kernel(int NBo, const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col_idx,
                                         int32_t *__restrict__ rel)
{
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= NBo) return;
    int prev = 0;
    for (int n = row_ptr[l]; n < row_ptr[l + 1]; ++n) {
        const int cur = col_idx[n];
        rel[n] = cur - prev;
        prev = cur;
    }
}

__global__ void index_from_relative_kernel(int NBo, const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ rel,
                                           int32_t *__restrict__ col_idx)
{
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= NBo) return;
    int at = 0;
    for (int n = row_ptr[l]; n < row_ptr[l + 1]; ++n) {
        at += rel[n];
        col_idx[n] = at;
    }
}

}  // namespace
}  // namespace bsp

using namespace bsp;

extern "C" {

bsp_status bsp_spgemm(const bsp_wdesc *wa, const bsp_bcsr *a, const bsp_wdesc *wb, const bsp_bcsr *b, float *C, void *ws,
                      void *stream)
{
    bsp_status rc = check_wdesc(wa);
    if (rc != BSP_OK) return rc;
    rc = check_wdesc(wb);
    if (rc != BSP_OK) return rc;
    if (!a || !b || !C || !ws || !a->row_ptr || !a->col_idx || !a->payload || !b->row_ptr || !b->col_idx || !b->payload)
        return BSP_ERR_NULL;
    if (wa->H != 1 || wa->K != 1 || wb->H != 1 || wb->K != 1 || wa->I != wb->I) return BSP_ERR_SHAPE;
    if (wa->bo != kSpEdge || wa->bi != kSpEdge || wb->bo != kSpEdge || wb->bi != kSpEdge) return BSP_ERR_BLOCK;
    if (wa->wtype != wb->wtype || (wa->wtype != BSP_F32 && wa->wtype != BSP_BF16)) return BSP_ERR_DTYPE;
    if (((uintptr_t)C & 7u) != 0 || ((uintptr_t)a->payload & 15u) != 0 || ((uintptr_t)b->payload & 15u) != 0) return BSP_ERR_SHAPE;
    const int NBa = wa->O / kSpEdge, NBb = wb->O / kSpEdge, NBk = wa->I / kSpEdge;
    const size_t smem = (size_t)NBk * sizeof(int);
    if (smem > 48 * 1024) return BSP_ERR_SHAPE;
    // rows of B are dealt over the warps of gridDim.y CTAs per row of A: enough CTAs to fill the GPU a few times over
    int gy = (NBb + kSpThreads / 32 - 1) / (kSpThreads / 32);
    const int want = (148 * 8 + NBa - 1) / NBa;
    if (gy > want) gy = want;
    if (gy < 1) gy = 1;
    const dim3 grid((unsigned)NBa, (unsigned)gy);
    cudaStream_t st = (cudaStream_t)stream;
    if (wa->wtype == BSP_F32) {
        int n_sm = 0;
        rc = spgemm_f32_device(&n_sm);
        if (rc != BSP_OK) return rc;
        const dim3 tiles((unsigned)((NBb + kSfRows - 1) / kSfRows), (unsigned)((NBa + kSfRows - 1) / kSfRows));
        if (NBk <= kSfMaxCols && tiles.y <= 65535u && spgemm_f32_tiles(NBa, NBb, NBk, a->nnz, b->nnz, n_sm)) {
            const size_t pos = (size_t)2 * kSfRows * ((NBk + kSfChunk - 1) / kSfChunk * kSfChunk) * sizeof(int16_t);
            BSP_CUDA_OK(launch_after(spgemm_f32_kernel, tiles, dim3(kSfThreads), pos, st, a->row_ptr, a->col_idx, (const float *)a->payload, b->row_ptr, b->col_idx,
                                     (const float *)b->payload, NBa, NBb, NBk, C, (int *)ws));
            return BSP_OK;
        }
        BSP_CUDA_OK(launch_after(spgemm_kernel<float>, grid, dim3(kSpThreads), smem, st, a->row_ptr, a->col_idx, (const float *)a->payload, b->row_ptr, b->col_idx,
                                                             (const float *)b->payload, NBb, NBk, C, (int *)ws));
    } else {
        const StDevice *gpu = nullptr;
        rc = spgemm_tc_device(&gpu);
        if (rc != BSP_OK) return rc;
        const StPlan plan = spgemm_plan(NBa, NBb, NBk, a->nnz, b->nnz, gy, *gpu);
        const StParams q = {a->row_ptr, a->col_idx, b->row_ptr, b->col_idx, (const uint8_t *)a->payload, (const uint8_t *)b->payload,
                            C, (int *)ws, NBa, NBb, NBk, (NBk + 7) / 8, 0, plan.split};
        if (plan.pair) return launch_spgemm_tc<256, true>(q, st);
        if (plan.BN == 64) return launch_spgemm_tc<64>(q, st);
        if (plan.BN == 128) return launch_spgemm_tc<128>(q, st);
        if (plan.BN == 256) return launch_spgemm_tc<256>(q, st);
        BSP_CUDA_OK(launch_after(spgemm_kernel<__nv_bfloat16>, grid, dim3(kSpThreads), smem, st, a->row_ptr, a->col_idx, (const __nv_bfloat16 *)a->payload, b->row_ptr,
                                                                     b->col_idx, (const __nv_bfloat16 *)b->payload, NBb, NBk, C, (int *)ws));
    }
    return BSP_OK;
}

bsp_status bsp_index_to_relative(int NBo, const int32_t *row_ptr, const int32_t *col_idx, int32_t *rel, void *stream)
{
    if (!row_ptr || !col_idx || !rel) return BSP_ERR_NULL;
    if (NBo <= 0) return BSP_ERR_SHAPE;
    index_to_relative_kernel<<<(NBo + 127) / 128, 128, 0, (cudaStream_t)stream>>>(NBo, row_ptr, col_idx, rel);
    BSP_CUDA_OK(cudaGetLastError());
    return BSP_OK;
}

bsp_status bsp_index_from_relative(int NBo, const int32_t *row_ptr, const int32_t *rel, int32_t *col_idx, void *stream)
{
    if (!row_ptr || !col_idx || !rel) return BSP_ERR_NULL;
    if (NBo <= 0) return BSP_ERR_SHAPE;
    index_from_relative_kernel<<<(NBo + 127) / 128, 128, 0, (cudaStream_t)stream>>>(NBo, row_ptr, rel, col_idx);
    BSP_CUDA_OK(cudaGetLastError());
    return BSP_OK;
}

}  // extern "C"
