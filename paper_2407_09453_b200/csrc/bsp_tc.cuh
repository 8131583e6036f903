// Pieces shared by the tensor-core kernels (tcgen05.mma with accumulators in tensor memory, operands staged by tiled
// TMA loads under the 128-byte swizzle): constants, bounded barrier waits, shared-memory matrix descriptors, the issue of
// one K-stage, tensor-memory loads, the tensor-map encoder and the choice of position tiles.  Every translation unit
// that includes this file gets its own copies (anonymous namespace).
#pragma once
#include <cuda.h>
#include <stddef.h>
#include "bsp_internal.cuh"

namespace bsp {
namespace {

constexpr int kGtThreads = 320;                    // producer warp, MMA warp, two groups of four epilogue warps
constexpr int kGtBM = 128;                         // positions per tile (M of the MMA)
constexpr int kGtABytes = kGtBM * 128;             // activation bytes of a stage
constexpr int kGtStageRows = 32;                   // rows of Y per epilogue warp
constexpr int kGtStagingBytes = kGtStageRows * 128;   // one staging buffer of an epilogue warp
constexpr int kGtMaxStages = 8;
constexpr int kGtMaxSmem = 226 * 1024;
constexpr int kGtTmemCols = 512;
constexpr int kGtMaxDevices = 64;
constexpr uint32_t kGtSpin = 1u << 24;             // polls of a barrier before a wait gives up

__device__ __forceinline__ uint32_t sm32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool gt_poll(uint32_t bar, uint32_t parity)
{
    for (uint32_t spin = 0; spin < kGtSpin; ++spin) {
        uint32_t done;
        asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.b32 %0, 1, 0, p;\n}\n"
                     : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}
// One look at the barrier, without waiting: non-zero once the phase has completed.  The result of a poll reaches the
// branch that depends on it after about 90 cycles, so the producer and the MMA warp look at the barrier of the next
// stage while they issue the current one and fall back to gt_poll only when that look came too early.
__device__ __forceinline__ uint32_t gt_test(uint32_t bar, uint32_t parity)
{
    uint32_t done;
    asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.b32 %0, 1, 0, p;\n}\n"
                 : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done;
}
// The wait of the MMA warp for a stage that its look did not find: all lanes, then the fence that orders the MMAs behind it.
__device__ __forceinline__ bool gt_poll_stage(uint32_t bar, uint32_t parity)
{
    const bool ok = __all_sync(0xFFFFFFFFu, gt_poll(bar, parity));
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    return ok;
}
// The same wait for the threads of the epilogue warps: try_wait suspends the thread for a while.
__device__ __forceinline__ bool gt_wait(uint32_t bar, uint32_t parity)
{
    for (uint32_t spin = 0; spin < (kGtSpin >> 6); ++spin) {
        uint32_t done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.b32 %0, 1, 0, p;\n}\n"
                     : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}

// Shared-memory matrix descriptor of a K-major operand under the 128-byte swizzle (start address in 16-byte units in
// the low 14 bits): rows of 128 bytes, 8-row groups 1024 bytes apart; a K-step of 32 bytes inside the swizzle span is
// an advance of the start address by 2.
constexpr uint64_t kGtDesc = (1ull << 16) | ((uint64_t)(1024u >> 4) << 32) | (1ull << 46) | (2ull << 61);
// The same for rows of 64 bytes under the 64-byte swizzle (layers with at most 64 bytes of input channels): 8-row
// groups 512 bytes apart, two K-steps of 32 bytes.
constexpr uint64_t kGtDesc64 = (1ull << 16) | ((uint64_t)(512u >> 4) << 32) | (1ull << 46) | (4ull << 61);

// Rows of 32 bytes under the 32-byte swizzle (one K-step): 8-row groups 256 bytes apart.
constexpr uint64_t kGtDesc32 = (1ull << 16) | ((uint64_t)(256u >> 4) << 32) | (1ull << 46) | (6ull << 61);

// A descriptor with another distance between the groups of eight rows, in 16-byte units.
__device__ __forceinline__ uint64_t gt_desc_groups(uint64_t desc, uint32_t units) { return (desc & ~((uint64_t)0x3FFFu << 32)) | ((uint64_t)units << 32); }

// The place of row r of a kHalo tile's MMA in the tile's box of positions (as TMA stores read it), or -1 for a row between them.
__device__ __forceinline__ int gt_halo_row(int r, int eights, int Wt, int Ht, int Nt, int halo_w, int halo_rows)
{
    const int pitch = eights ? 8 : halo_w, per_image = halo_rows * pitch, n = r / per_image, y = (r - n * per_image) / pitch, x = r - n * per_image - y * pitch;
    return n < Nt && y < Ht && x < Wt ? (n * Ht + y) * Wt + x : -1;
}

// The MMAs of one stage (four, or two when the stage holds 64 bytes of K: `nk`), the commit that releases the stage, and a look at
// the barrier of the next stage, issued by one elected lane of a converged warp.  All lanes execute this statement with the same
// operands; the MMA of the first K-step overwrites the accumulator when `acc` is 0.  Returns non-zero once the next stage has arrived.
// The look stands between the second and the third MMA, and its result is taken at the end: the tensor pipe takes one or two
// instructions ahead, so that what stands before the first MMA of a stage it waits for.  (A stage of four MMAs with M = 64 and 64
// channels, 128 cycles of arithmetic: 172 cycles with the look before them, 156 with its result taken between them, 132 like this;
// 32 channels 161, 150 and 132; M = 128 with 64 channels 199, 192 and 192; 128 and more channels take their arithmetic either way.)
#define GT_ISSUE_STAGE(KIND, CG, COMMIT_TAIL)                                                                       \
    asm volatile("{\n .reg .pred e, e3, p, t, f, v;\n .reg .b64 a1, a2, a3, b1, b2, b3;\n"                           \
                 " elect.sync _|e, 0xFFFFFFFF;\n setp.ne.b32 p, %6, 0;\n setp.eq.b32 t, %6, %6;\n"                    \
                 " setp.gt.u32 e3, %8, 2;\n and.pred e3, e3, e;\n"                                                    \
                 " add.u64 a1, %2, 2;\n add.u64 a2, %2, 4;\n add.u64 a3, %2, 6;\n"                                    \
                 " add.u64 b1, %3, 2;\n add.u64 b2, %3, 4;\n add.u64 b3, %3, 6;\n"                                    \
                 " @e tcgen05.mma.cta_group::" CG ".kind::" KIND " [%1], %2, %3, %4, p;\n"                                 \
                 " @e tcgen05.mma.cta_group::" CG ".kind::" KIND " [%1], a1, b1, %4, t;\n"                                 \
                 " mbarrier.test_wait.parity.shared::cta.b64 f, [%9], %10;\n"                                              \
                 " @e3 tcgen05.mma.cta_group::" CG ".kind::" KIND " [%1], a2, b2, %4, t;\n"                                \
                 " @e3 tcgen05.mma.cta_group::" CG ".kind::" KIND " [%1], a3, b3, %4, t;\n"                                \
                 " @e tcgen05.commit.cta_group::" CG ".mbarrier::arrive::one.shared::cluster" COMMIT_TAIL ";\n"            \
                 " vote.sync.all.pred v, f, 0xFFFFFFFF;\n tcgen05.fence::after_thread_sync;\n selp.b32 %0, 1, 0, v;\n}\n"    \
                 : "=r"(next) : "r"(d), "l"(da), "l"(db), "r"(idesc), "r"(bar_empty), "r"(acc), "h"((unsigned short)3), "r"(nk), "r"(bar_next), "r"(par_next) : "memory")

// The MMAs of one tap without a commit (its activations stay in place for the taps to come): four K-steps inside the span of
// the 128-byte swizzle, or one or two (`two`) in planes of 32-byte rows, `pa` and `pb` 16-byte units apart.
#define GT_ISSUE_TAP(KIND)                                                                                           \
    asm volatile("{\n .reg .pred e, p, t;\n .reg .b64 a1, a2, a3, b1, b2, b3;\n"                                     \
                 " elect.sync _|e, 0xFFFFFFFF;\n setp.ne.b32 p, %4, 0;\n setp.eq.b32 t, %4, %4;\n"                    \
                 " add.u64 a1, %1, 2;\n add.u64 a2, %1, 4;\n add.u64 a3, %1, 6;\n"                                    \
                 " add.u64 b1, %2, 2;\n add.u64 b2, %2, 4;\n add.u64 b3, %2, 6;\n"                                    \
                 " @e tcgen05.mma.cta_group::1.kind::" KIND " [%0], %1, %2, %3, p;\n"                                   \
                 " @e tcgen05.mma.cta_group::1.kind::" KIND " [%0], a1, b1, %3, t;\n"                                   \
                 " @e tcgen05.mma.cta_group::1.kind::" KIND " [%0], a2, b2, %3, t;\n"                                   \
                 " @e tcgen05.mma.cta_group::1.kind::" KIND " [%0], a3, b3, %3, t;\n}\n"                                \
                 ::"r"(d), "l"(da), "l"(db), "r"(idesc), "r"(acc) : "memory")
#define GT_ISSUE_PLANES(KIND)                                                                                        \
    asm volatile("{\n .reg .pred e, e1, p, t;\n .reg .b64 a1, b1;\n"                                                 \
                 " elect.sync _|e, 0xFFFFFFFF;\n setp.ne.b32 p, %4, 0;\n setp.eq.b32 t, %4, %4;\n"                    \
                 " setp.ne.b32 e1, %7, 0;\n and.pred e1, e1, e;\n add.u64 a1, %1, %5;\n add.u64 b1, %2, %6;\n"        \
                 " @e tcgen05.mma.cta_group::1.kind::" KIND " [%0], %1, %2, %3, p;\n"                                   \
                 " @e1 tcgen05.mma.cta_group::1.kind::" KIND " [%0], a1, b1, %3, t;\n}\n"                               \
                 ::"r"(d), "l"(da), "l"(db), "r"(idesc), "r"(acc), "l"(pa), "l"(pb), "r"(two) : "memory")
template <int kWT>
__device__ __forceinline__ void gt_issue_tap(uint32_t d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc)
{
    if constexpr (kWT == BSP_BF16) GT_ISSUE_TAP("f16");
    else if constexpr (kWT == BSP_I8) GT_ISSUE_TAP("i8");
    else GT_ISSUE_TAP("tf32");
}
template <int kWT>
__device__ __forceinline__ void gt_issue_planes(uint32_t d, uint64_t da, uint64_t db, uint64_t pa, uint64_t pb, uint32_t two, uint32_t idesc, uint32_t acc)
{
    if constexpr (kWT == BSP_BF16) GT_ISSUE_PLANES("f16");
    else if constexpr (kWT == BSP_I8) GT_ISSUE_PLANES("i8");
    else GT_ISSUE_PLANES("tf32");
}

// kPair: the MMAs span a pair of CTAs (cta_group::2, M = 256: each CTA its own 128 positions and half of the weight
// tile); the commits then arrive on the barrier at the same shared-memory offset in both CTAs.
// The operand type is a template argument: a choice at run time costs a branch around every stage.
template <int kWT, bool kPair>
__device__ __forceinline__ uint32_t gt_issue_stage(uint32_t d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t bar_empty,
                                                   uint32_t acc, uint32_t nk, uint32_t bar_next, uint32_t par_next)
{
    uint32_t next;
    if constexpr (kPair) {
        if constexpr (kWT == BSP_BF16) GT_ISSUE_STAGE("f16", "2", ".multicast::cluster.b64 [%5], %7");
        else if constexpr (kWT == BSP_I8) GT_ISSUE_STAGE("i8", "2", ".multicast::cluster.b64 [%5], %7");
        else GT_ISSUE_STAGE("tf32", "2", ".multicast::cluster.b64 [%5], %7");
    } else {
        if constexpr (kWT == BSP_BF16) GT_ISSUE_STAGE("f16", "1", ".b64 [%5]");
        else if constexpr (kWT == BSP_I8) GT_ISSUE_STAGE("i8", "1", ".b64 [%5]");
        else GT_ISSUE_STAGE("tf32", "1", ".b64 [%5]");
    }
    return next;
}
// All MMAs issued so far by the elected lane complete -> one arrival on `bar` (in both CTAs of a pair).
template <bool kPair>
__device__ __forceinline__ void gt_commit_elected(uint32_t bar)
{
    if constexpr (kPair)
        asm volatile("{\n .reg .pred e;\n elect.sync _|e, 0xFFFFFFFF;\n"
                     " @e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n}\n"
                     ::"r"(bar), "h"((unsigned short)3) : "memory");
    else
        asm volatile("{\n .reg .pred e;\n elect.sync _|e, 0xFFFFFFFF;\n"
                     " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(bar) : "memory");
}

// Synchronises the CTA (the two CTAs of a pair).
template <bool kPair>
__device__ __forceinline__ void gt_sync_all()
{
    if constexpr (kPair) {
        asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    } else {
        __syncthreads();
    }
}

// True if `packed` is a buffer that bsp_compact filled for this descriptor, with the masked dense form in it.
// Where the host knows that memory is mapped as far as the descriptor's weights reach (packed_spans), the kernels
// look at the header twice.  First before wait_for_previous(), on the side of the kernel that still runs: if that look succeeds, loads
// need not wait for the look after the wait, a trip to L2 (0.1 to 0.5 us a call: fully connected 2048->1000, 64 positions, 5.79 -> 5.47 us,
// 3x3 128->128 at 28x28 4.85 -> 4.74, 1x1 256->1024 at 14x14, batch 64, 11.56 -> 11.06).  That one decides whether anything is stored:
// the header seen before may have been an old one of memory that held a larger buffer, or one that the kernel before was about to replace.
__device__ __forceinline__ bool gt_header_ok(const uint8_t *packed, int wtype, int O, int I, int H, int K, int bo, int bi)
{
    static_assert(offsetof(PackedHeader, H) == 16 && offsetof(PackedHeader, forms) == 32, "the header is read in pieces of 16 bytes");
    int m, t, o, i, h, k, r, c, f;
    asm volatile("ld.relaxed.gpu.global.v4.b32 {%0, %1, %2, %3}, [%4];\n" : "=r"(m), "=r"(t), "=r"(o), "=r"(i) : "l"(packed) : "memory");
    asm volatile("ld.relaxed.gpu.global.v4.b32 {%0, %1, %2, %3}, [%4];\n" : "=r"(h), "=r"(k), "=r"(r), "=r"(c) : "l"(packed + 16) : "memory");
    asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];\n" : "=r"(f) : "l"(packed + 32) : "memory");
    return (uint32_t)m == kPackedMagic && t == wtype && o == O && i == I && h == H && k == K && r == bo && c == bi && (f & kFormDense) != 0;
}

// n / d and n % d for 0 <= n < 2^31 by the multiplier m = floor(2^32 / d) (0xFFFFFFFF for d = 1): the product's high
// word is the quotient or one less, one correction settles it.
__device__ __forceinline__ void gt_divmod(int n, int d, uint32_t m, int &q, int &r)
{
    q = (int)__umulhi((uint32_t)n, m);
    r = n - q * d;
    if (r >= d) { ++q; r -= d; }
}

// Requantisation of the 8-bit path (Section "Compiler and its Code generation", Eq. (quant)): v / 2^s rounded to the
// nearest integer, halves away from zero, as a 32-bit value that is not yet saturated (|v| + 2^(s-1) < 2^32, so the
// magnitude is formed without overflow; -2^31 with s = 0 comes back as itself) ...
__device__ __forceinline__ int gt_round_shift(int v, uint32_t s)
{
    const uint32_t mag = v < 0 ? 0u - (uint32_t)v : (uint32_t)v;          // |v|, at most 2^31
    const uint32_t r = (mag + ((1u << s) >> 1)) >> s;
    return (int)(v < 0 ? 0u - r : r);
}
// The same for 1 <= s <= 30 and |v| <= 2^30, with half = 2^(s - 1): one is taken from negative values, then halves go up.
// (Integer operations run at half rate, and ten of them per value bound the 8-bit layers with few channels.)
__device__ __forceinline__ int gt_round_shift_small(int v, uint32_t half, uint32_t s) { return (v + (int)half + (v >> 31)) >> s; }
// ... and four such values saturated to int8 and packed, the first in the lowest byte (cvt.pack saturates two 32-bit
// values to bytes, its first source above its second, and shifts the third operand up by 16 bits).
__device__ __forceinline__ uint32_t gt_pack_s8x4(int v0, int v1, int v2, int v3)
{
    uint32_t hi, out;
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;\n" : "=r"(hi) : "r"(v3), "r"(v2), "r"(0u));
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;\n" : "=r"(out) : "r"(v1), "r"(v0), "r"(hi));
    return out;
}

// Barrier `id` (1..15) over the 128 threads of a group of four warps, and the same with the AND of a flag.
__device__ __forceinline__ void gt_group_sync(int id) { asm volatile("bar.sync %0, 128;\n" ::"r"(id) : "memory"); }
__device__ __forceinline__ bool gt_group_all(int id, bool flag)
{
    uint32_t r;
    asm volatile("{\n .reg .pred p, q;\n setp.ne.b32 p, %1, 0;\n bar.red.and.pred q, %2, 128, p;\n selp.b32 %0, 1, 0, q;\n}\n"
                 : "=r"(r) : "r"((uint32_t)flag), "r"(id) : "memory");
    return r != 0u;
}

// 32 consecutive accumulator columns of this thread's tensor-memory lane: the load, and the wait after which the values of
// the loads issued so far may be used (it names the registers, so that no use of them moves before it).
__device__ __forceinline__ void gt_load32_issue(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                   "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
                   "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ void gt_load32_wait(uint32_t (&v)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;\n"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                   "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]),
                   "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]),
                   "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31])
                 :: "memory");
}
__device__ __forceinline__ void gt_load32(uint32_t taddr, uint32_t (&v)[32])
{
    gt_load32_issue(taddr, v);
    gt_load32_wait(v);
}

// One round of an epilogue: 128 bytes of this lane's row of the output (32 channels of 4 bytes, 64 of bfloat16, 128 of
// int8) from the accumulator columns at `taddr`, after the bias.  kEy: bytes of an output element.  `bias` (raw bits), `half`
// and `shift` are the channels' own entries in shared memory, read four channels at a time by all lanes at once.  `n`:
// channels left; zeros past them (in steps of 32).  kRelu: max(., 0) if `relu`.
//
// 4-byte and bfloat16 output: into registers.
template <bool kInt, int kEy, bool kRelu>
__device__ __forceinline__ void gt_epilogue_round(uint32_t taddr, const uint32_t *bias, int n, int relu, uint32_t (&out)[32])
{
    if constexpr (kEy == 4) {
        gt_load32(taddr, out);
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
            const uint4 b = *(const uint4 *)(bias + e);
            if constexpr (kInt) { out[e] += b.x; out[e + 1] += b.y; out[e + 2] += b.z; out[e + 3] += b.w; }
            else {
                out[e] = __float_as_uint(__uint_as_float(out[e]) + __uint_as_float(b.x));
                out[e + 1] = __float_as_uint(__uint_as_float(out[e + 1]) + __uint_as_float(b.y));
                out[e + 2] = __float_as_uint(__uint_as_float(out[e + 2]) + __uint_as_float(b.z));
                out[e + 3] = __float_as_uint(__uint_as_float(out[e + 3]) + __uint_as_float(b.w));
            }
        }
    } else {                                             // rounded to nearest even after the bias
        uint32_t v[2][32];
        gt_load32_issue(taddr, v[0]);
        if (n > 32) gt_load32_issue(taddr + 32u, v[1]);
        else {
#pragma unroll
            for (int e = 0; e < 32; ++e) v[1][e] = 0u;
        }
        gt_load32_wait(v[0]);
        gt_load32_wait(v[1]);
#pragma unroll
        for (int sub = 0; sub < 2; ++sub)
#pragma unroll
            for (int e = 0; e < 32; e += 4) {
                const uint4 b = *(const uint4 *)(bias + sub * 32 + e);
                __nv_bfloat162 h0 = __floats2bfloat162_rn(__uint_as_float(v[sub][e]) + __uint_as_float(b.x), __uint_as_float(v[sub][e + 1]) + __uint_as_float(b.y));
                __nv_bfloat162 h1 = __floats2bfloat162_rn(__uint_as_float(v[sub][e + 2]) + __uint_as_float(b.z), __uint_as_float(v[sub][e + 3]) + __uint_as_float(b.w));
                if (kRelu && relu) { h0 = __hmax2(h0, __float2bfloat162_rn(0.f)); h1 = __hmax2(h1, __float2bfloat162_rn(0.f)); }
                out[sub * 16 + e / 2] = *(const uint32_t *)&h0;
                out[sub * 16 + e / 2 + 1] = *(const uint32_t *)&h1;
            }
    }
}
// ... and from there to the row at `srow` of a tile in shared memory under the 128-byte swizzle (`sw`: the row modulo 8;
// `live`: the lane has a row; `pieces`: 16-byte pieces of the row, 8, or 4 of rows of 64 bytes under the 64-byte swizzle, where `sw` is
// half the row modulo 4).
__device__ __forceinline__ void gt_store_round(uint32_t srow, uint32_t sw, bool live, const uint32_t (&out)[32], uint32_t pieces = 8u)
{
    if (live) {
#pragma unroll
        for (uint32_t j = 0; j < 8u; ++j)
            if (j < 4u || pieces > 4u) asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n"
                         ::"r"(srow + ((j ^ sw) << 4)), "r"(out[4 * j]), "r"(out[4 * j + 1]), "r"(out[4 * j + 2]), "r"(out[4 * j + 3]) : "memory");
    }
}
// int8 output: requantised after the bias and written piece by piece, 32 channels at a time in a loop that stays a loop.
// (Unrolled, a round is a thousand instructions that eight warps fetch in eight places: 4800 cycles a round in the pair
// 64->64->256 at 56x56, which took 89 us and 47 us like this.)  `small`: 1 <= shift <= 30 for all channels and every sum at
// most 2^30 (gt_round_shift_small holds, `half` has its 2^(s - 1)).  Shifts are words where shared memory has room for them, else bytes,
// each of which costs an integer operation more.
__device__ __forceinline__ uint4 gt_shifts(const uint32_t *shift) { return *(const uint4 *)shift; }
__device__ __forceinline__ uint4 gt_shifts(const uint8_t *shift)
{
    const uint32_t s = *(const uint32_t *)shift;
    return make_uint4(__byte_perm(s, 0u, 0x4440), __byte_perm(s, 0u, 0x4441), __byte_perm(s, 0u, 0x4442), s >> 24);
}
template <bool kRelu, typename S>
__device__ __forceinline__ void gt_epilogue_int8(uint32_t taddr, const uint32_t *bias, const uint32_t *half, const S *shift, bool small, int n, int relu,
                                                 uint32_t srow, uint32_t sw, bool live)
{
#pragma unroll 1
    for (int sub = 0; sub < 4; ++sub, n -= 32, taddr += 32u, bias += 32, half += 32, shift += 32) {
        uint32_t out[8];
        if (n <= 0) {
#pragma unroll
            for (int e = 0; e < 8; ++e) out[e] = 0u;
        } else {
            uint32_t v[32];
            gt_load32(taddr, v);
            if (small) {
#pragma unroll
                for (int e = 0; e < 32; e += 4) {
                    const uint4 b = *(const uint4 *)(bias + e), h = *(const uint4 *)(half + e);
                    const uint4 s = gt_shifts(shift + e);
                    out[e / 4] = gt_pack_s8x4(gt_round_shift_small((int)(v[e] + b.x), h.x, s.x), gt_round_shift_small((int)(v[e + 1] + b.y), h.y, s.y),
                                              gt_round_shift_small((int)(v[e + 2] + b.z), h.z, s.z), gt_round_shift_small((int)(v[e + 3] + b.w), h.w, s.w));
                }
            } else {
#pragma unroll
                for (int e = 0; e < 32; e += 4) {
                    const uint4 b = *(const uint4 *)(bias + e);
                    const uint4 s = gt_shifts(shift + e);
                    out[e / 4] = gt_pack_s8x4(gt_round_shift((int)(v[e] + b.x), s.x), gt_round_shift((int)(v[e + 1] + b.y), s.y),
                                              gt_round_shift((int)(v[e + 2] + b.z), s.z), gt_round_shift((int)(v[e + 3] + b.w), s.w));
                }
            }
            if (kRelu && relu) {
#pragma unroll
                for (int e = 0; e < 8; ++e) out[e] = __vmaxs4(out[e], 0u);
            }
        }
        if (live) {
#pragma unroll
            for (uint32_t j = 0; j < 2u; ++j)
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n"
                             ::"r"(srow + ((((uint32_t)sub * 2u + j) ^ sw) << 4)), "r"(out[4 * j]), "r"(out[4 * j + 1]), "r"(out[4 * j + 2]), "r"(out[4 * j + 3]) : "memory");
        }
    }
}

typedef CUresult (*GtEncodeFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                               const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                               CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

GtEncodeFn gt_encode()
{
    static GtEncodeFn fn = nullptr;
    if (!fn) {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (GtEncodeFn)ptr;
    }
    return fn;
}


// Position tile of a layer: Wt x Ht output positions of Nt images, at most 128, chosen for the fewest tiles (ties: the
// smaller box).  Several images share a tile only when a tile holds whole images.  A box of the tensor map spans
// Wt * s_w x Ht * s_h input positions and may not exceed 256 in any extent.
struct GtTile { int Wt, Ht, Nt; long long tiles; };
// (gt_pick_halo) `eights`: the rows of the MMA go by groups of eight positions of a row of the image.
struct GtHaloTile : GtTile { int eights; };

// A 1x1 layer without padding or stride is a matrix product over all N L J positions: taken as that many 1x1 images,
// so that a tile is 128 consecutive positions whatever the image size.
bsp_xdesc gt_flatten(const bsp_wdesc &wd, const bsp_xdesc &xd)
{
    const long long P = (long long)xd.N * xd.L * xd.J;
    if (wd.H == 1 && wd.K == 1 && xd.pad_h == 0 && xd.pad_w == 0 && xd.stride_h == 1 && xd.stride_w == 1 && P <= 0x7FFFFFFF)
        return bsp_xdesc{(int)P, 1, 1, 1, 1, 0, 0};
    return xd;
}

uint32_t gt_magic(int d) { return d <= 1 ? 0xFFFFFFFFu : (uint32_t)((1ull << 32) / (uint64_t)d); }

// For every width the tallest box that fits has the fewest tiles, and of the heights with that many tiles the lowest has
// the smallest area; the same holds for the widths with the same number of tiles across, so only the distinct tile
// counts in x are looked at, each with one height (about 2 sqrt(N_w) of them instead of every width and height).
GtTile gt_pick_tile(int N, int M, int Nw, int sh, int sw, int rows = kGtBM)
{
    GtTile best = {0, 0, 0, -1};
    if (sh > 256 || sw > 256) return best;
    for (int w = 1; w <= Nw && w <= rows && w * sw <= 256;) {
        int hmax = rows / w;
        if (hmax > M) hmax = M;
        if (hmax * sh > 256) hmax = 256 / sh;
        const int ty = (M + hmax - 1) / hmax, h = (M + ty - 1) / ty, tx = (Nw + w - 1) / w;
        int b = 1;
        if (w == Nw && h == M) { b = rows / (w * h); if (b > N) b = N; if (b > 256) b = 256; if (b < 1) b = 1; }
        const long long cnt = (long long)((N + b - 1) / b) * ty * tx;
        const long long area = (long long)b * h * w, best_area = (long long)best.Wt * best.Ht * best.Nt;
        if (best.tiles < 0 || cnt < best.tiles || (cnt == best.tiles && area < best_area)) best = {w, h, b, cnt};
        if (tx == 1) break;
        w = (Nw + tx - 2) / (tx - 1);                 // the narrowest box with one tile less across
    }
    return best;
}

// Position tile of a layer that takes several waves: parts of several images, so that the 128 rows of a tile are filled where no
// box of one image fills them (56 x 56: 112 of 128 rows, but 8 x 8 positions of two images all of them; 7 x 7: 98, but a row
// of 18 images 126): int8 3x3 256->256 at 56x56, batch 32, 48.9 -> 45.0 us in a short burst (52 to 53 in a stream of calls, under
// the power cap), TF32 3x3 464->432 at 17x17, batch 52, 141 -> 101 us.
// (The search takes 1 to 3 us of the host, hidden behind the waves of such a layer; a layer of one wave has no use for it.)  Looks at the distinct tile counts in x and y only, each with its smallest box.
GtTile gt_pick_packed(GtTile best, int N, int M, int Nw, int sh, int sw)
{
    const long long least = ((long long)N * M * Nw + kGtBM - 1) / kGtBM;
    if (N == 1 || best.tiles == least) return best;
    for (int w = 1; w <= Nw && w <= kGtBM && w * sw <= 256;) {
        const int tx = (Nw + w - 1) / w;
        for (int h = 1; h <= M && w * h <= kGtBM && h * sh <= 256;) {
            const int ty = (M + h - 1) / h;
            int b = kGtBM / (w * h);
            if (b > N) b = N;
            const long long cnt = (long long)((N + b - 1) / b) * ty * tx;
            // (of equal counts the box of fewer images, whose borders share more)
            if (cnt < best.tiles || (cnt == best.tiles && b < best.Nt)) best = {w, h, b, cnt};
            if (ty == 1) break;
            h = (M + ty - 2) / (ty - 1);
        }
        if (tx == 1) break;
        w = (Nw + tx - 2) / (tx - 1);
    }
    return best;
}

// Position tile of a stride-1 layer whose activations are staged once per tile, with the H - 1 rows and K - 1 columns that its
// taps reach beyond it.  The rows of the MMA are the 128 consecutive positions of that box from the tap's own offset on, so
// output (n, y, x) sits in row (n (Ht + H - 1) + y) (Wt + K - 1) + x and the rows between are not used; or, in tiles of eight columns
// (`eights`), 16 groups of eight positions a row of the box apart (the stride between groups of the matrix descriptor), so that
// output (n, y, x) sits in row (n (Ht + H - 1) + y) 8 + x and all rows of a tile of 8 x 16 are used: 8-bit 3x3 64->64 at 224x224,
// batch 32, 85.0 -> 75.3 us.  (Taken where they are fewer; with as many tiles they were up to 2 % slower.)
// Rows of the MMA that no output uses may lie past the last box of the ring, in tiles of eight columns by up to 32 KB (1x19 on six images of one
// row of seven columns; taps, tiles and row widths walked through on the host): what stands behind the ring covers that, the staging
// buffers of the product, layer two's weights and the tensor between the layers of the pair.
GtHaloTile gt_pick_halo(int N, int M, int Nw, int H, int K)
{
    GtHaloTile best = {{0, 0, 0, -1}, 0};
    long long best_area = 0;
    auto offer = [&](int w, int h, int b, int eights) {
        const int pitch = w + K - 1;
        const long long cnt = (long long)((N + b - 1) / b) * ((M + h - 1) / h) * ((Nw + w - 1) / w), area = (long long)b * (h + H - 1) * pitch;
        if (pitch <= 256 && h + H - 1 <= 256 && (best.tiles < 0 || cnt < best.tiles || (cnt == best.tiles && !eights && area < best_area))) {
            best = {{w, h, b, cnt}, eights};
            best_area = area;
        }
    };
    for (int w = 1; w <= Nw && w <= kGtBM;) {
        const int pitch = w + K - 1, tx = (Nw + w - 1) / w;
        int h = (kGtBM - w) / pitch + 1;
        if (h > M) h = M;
        const int ty = (M + h - 1) / h;
        h = (M + ty - 1) / ty;
        int b = 1;
        if (w == Nw && h == M) { b = (kGtBM - ((h - 1) * pitch + w)) / ((h + H - 1) * pitch) + 1; if (b > N) b = N; }
        offer(w, h, b, 0);
        if (tx == 1) break;
        w = (Nw + tx - 2) / (tx - 1);
    }
    const int w = Nw < 8 ? Nw : 8;
    int h = M < kGtBM / 8 ? M : kGtBM / 8;
    const int ty = (M + h - 1) / h;
    h = (M + ty - 1) / ty;
    int b = 1;
    if (h == M) { b = (kGtBM / 8 - M) / (M + H - 1) + 1; if (b > N) b = N; }
    if (w == 8 || b > 1) offer(w, h, w == Nw ? b : 1, 1);
    return best;
}

}  // namespace
}  // namespace bsp
