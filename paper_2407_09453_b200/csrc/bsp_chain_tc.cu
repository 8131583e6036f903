// Two consecutive block-sparse layers in one kernel: T = act(W1 * X + b1) stored as bfloat16, Y = W2 * T + b2 with a 1x1
// second layer; or the 8-bit chain, where T is the requantised int8 output of layer one (Section "Compiler and its Code
// generation": power-of-two scales) and Y is int32 or requantised int8.  Section "Depth-wise Tiling" of the paper: the output is cut into tiles, every tile is carried through
// the whole chain, and the tensor between the layers never goes to external memory.  A 1x1 second layer needs no
// overlap between tiles (its projection of one output position is one position of T), so the tiles are those of the
// first layer.
//
// Per tile of up to 128 output positions a persistent CTA runs
//   1. the first layer as an implicit GEMM over taps x 128-byte channel chunks (activation box + weight tile per
//      K-stage, both by tiled TMA loads) into accumulator one, all O1 <= 256 channels in tensor memory;
//   2. its epilogue: tensor memory -> registers -> + b1 -> max(., 0) if asked -> bfloat16 (int8: rounding shift, then
//      max(., 0)) -> shared memory, written in the K-major 128-byte-swizzled layout that an MMA reads as its A operand
//      (128 bytes of channels, that is 64 bfloat16 or 128 int8, per 16 KB chunk);
//   3. the second layer: for every tile of 128 output channels, MMAs of that tensor against weight chunks that arrive
//      through the same ring of stages, into one of two 128-column accumulators;
//   4. its epilogue: + b2 -> convert -> global memory, overlapping the MMAs of the next 128 channels.
// Where layer one has stride 1 and taps, its input channels fit one stage and shared memory allows (kHalo), its weights stay
// in shared memory and a tile's activations arrive once with the border that the taps reach, as in the product kernel; the
// weights of layer two then have a ring of their own, or stay too.
// Warps: 0 producer, 1 MMA issuer (both converged, one elected lane issues), 2.. epilogue in two or three groups of four, which
// take turns with the rounds of both epilogues: 128 bytes of T's or Y's channels each.  Every wait is bounded.
#include <type_traits>
#include "bsp_tc.cuh"

namespace bsp {
namespace {

// Epilogue groups of four warps: three where the tap-by-tap loads are gone and the epilogues bound the tile, else two (their
// staging buffers cost ring stages).
__host__ __device__ constexpr int ct_groups(bool halo) { return halo ? 3 : 2; }
constexpr int kCtBN2 = 128;                        // channels of layer two per accumulator buffer
constexpr int kCtChunk = kGtBM * 128;              // bytes of one chunk (128 bytes of channels) of the tensor between the layers

struct CtParams {
    CUtensorMap tmx;          // X as bytes: (I1 * esz, J, L, N), box of one operand row x the tile's positions (kHalo: with their border)
    CUtensorMap tmw1;         // Gamma1 (.) W1 as bytes: (I1 * esz, H K, O1), box of one operand row x 1 tap x O1p channels
    CUtensorMap tmw2;         // Gamma2 (.) W2 as bytes: (O1 * esz, 1, O2), box 128 bytes x 1 x 128 channels
    CUtensorMap tmy;          // Y as bytes: (O2 * ey, N_w, M, N), box 128 bytes x Wt x Ht x Nt positions (a tile)
    const void *bias1, *bias2;        // float32, or int32 for the 8-bit chain
    const int32_t *shift1, *shift2;   // 8-bit chain: rounding shifts of T (required) and of an int8 Y
    const uint8_t *packed1, *packed2;
    int *status;
    int O1, I1, H, K, bo1, bi1, O2, bo2, bi2, relu, wtype;
    int early_type;           // as in the product kernel, for both packed buffers
    int O1p;                  // O1 rounded up to a whole chunk of T (64 or 128 channels): columns of accumulator one
    int tcc;                  // channels per chunk of T: 64 (bfloat16) or 128 (int8)
    int n_ks1, cpt1, n_c2, n_t2;      // K-stages of layer one, its channel chunks per tap; chunks of T; channel tiles of layer two (of a CTA)
    int parts;                        // CTAs that share a position tile: each computes T and n_t2 channel tiles of layer two
    int stages, stage_bytes, n_tiles;
    int ahead;                // the first epilogue runs one tile ahead of the second
    int db, dbt;              // O1p <= 128: accumulator one is double-buffered, and without kHalo the tensor between the layers too
    int N, M, Nw, Wt, Ht, Nt, tiles_x, tiles_y;
    int sh, sw, ph, pw, a_bytes;
    uint32_t m_tx, m_ty;
    uint32_t off_ring, off_w2, off_t, off_staging, off_tail;         // bytes into shared memory
    uint32_t staging_bytes;           // a group's staging buffer: 128 bytes of every position of the tile
    // kHalo: bytes of K per position, planes and their pitch, pitch and rows of an image's box; slots of layer two's weights
    int kbytes, planes, plane_bytes, halo_w, halo_rows, w2_slots, w2_stay;
    int small1, small2;       // 8-bit: sums of products of either layer at most 2^29
};

// Barriers and constants, after everything else in shared memory (all of it dynamic: the base is 1024-byte aligned).
constexpr int kCtTaps = 30, kCtW2Slots = 8;
template <int kGroups>
struct CtTail {
    uint64_t full[kGtMaxStages], empty[kGtMaxStages], acc1_full[2], acc1_empty[2], t_full[2], t_empty[2], acc2_full[2], acc2_empty[2];
    uint64_t w1_full[kCtTaps], w2_full[kCtW2Slots], w2_empty[kCtW2Slots];
    uint64_t before_last;             // layer two of the last tile but one is done (used once)
    uint32_t tmem, fail, refused;
    uint32_t y_read[2];               // warps that have read accumulator two, counted over all tiles (kGroups > 2 kRpt)
    // per epilogue group: bias, 2^(shift - 1) and shift of its round's channels
    __align__(16) uint32_t bias[kGroups][128], half[kGroups][128];
    __align__(16) uint8_t shift[kGroups][128];
};
constexpr int kCtSmem = 227 * 1024;

__device__ __forceinline__ void ct_tile_origin(const CtParams &p, int mt, int &n0, int &y0, int &x0)
{
    int r, tx, ty, ni;
    gt_divmod(mt, p.tiles_x, p.m_tx, r, tx);
    gt_divmod(r, p.tiles_y, p.m_ty, ni, ty);
    x0 = tx * p.Wt; y0 = ty * p.Ht; n0 = ni * p.Nt;
}

// Waits (bounded) until a count in shared memory that only grows has reached n.
__device__ __forceinline__ bool ct_wait_count(const volatile uint32_t *count, uint32_t n)
{
    for (uint32_t spin = 0; spin < (kGtSpin >> 2); ++spin) {
        if (*count >= n) return true;
        __nanosleep(32);
    }
    return false;
}

// kI8: the 8-bit chain; kEy: bytes of an element of Y (compiled apart, so that no form carries another's epilogue code).  kEights: kHalo on tiles of
// eight columns, as in the product kernel.
template <bool kI8, int kEy, bool kHalo, bool kEights>
__global__ void __launch_bounds__(64 + 128 * ct_groups(kHalo), 1) chain_tc_kernel(const __grid_constant__ CtParams p)
{
    constexpr int kWt = kI8 ? BSP_I8 : BSP_BF16;
    extern __shared__ __align__(1024) uint8_t smem[];
    constexpr int kGroups = ct_groups(kHalo);
    CtTail<kGroups> &tail = *(CtTail<kGroups> *)(smem + p.off_tail);
    volatile uint32_t &s_fail = tail.fail;

    // (warp number, tensor-memory base and go-ahead through a shuffle: uniform to the compiler, as in the product kernel)
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    const int S = p.stages;
    const uint32_t base = sm32(smem), ring = base + p.off_ring;
    const uint32_t tbuf = base + p.off_t;                                // the tensor between the layers: n_c2 chunks
    const uint32_t tbytes = (uint32_t)(p.n_c2 * kCtChunk);
    const uint32_t staging = base + p.off_staging;
    const int t_first = (int)blockIdx.x / p.parts, t_step = (int)gridDim.x / p.parts, t_count = p.n_tiles;
    const int o2 = ((int)blockIdx.x - t_first * p.parts) * p.n_t2 * kCtBN2;      // this CTA's first channel of layer two
    constexpr int cpr = 128 / kEy, kRpt = kCtBN2 / cpr;                  // channels of a round of Y, rounds per 128-channel tile

    if (tid == 0) {
        tail.y_read[0] = tail.y_read[1] = 0u;
        for (int s = 0; s < S; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&tail.full[s])), "r"(1) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&tail.empty[s])), "r"(1) : "memory");
        }
        for (int b = 0; b < 2; ++b) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&tail.acc1_full[b])), "r"(1) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&tail.acc1_empty[b])), "r"(4 * p.n_c2) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&tail.t_full[b])), "r"(4 * p.n_c2) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&tail.t_empty[b])), "r"(1) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&tail.acc2_full[b])), "r"(1) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&tail.acc2_empty[b])), "r"(4 * kRpt) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&tail.before_last)), "r"(1) : "memory");
        if constexpr (kHalo) {
            for (int t = 0; t < p.n_ks1; ++t) asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&tail.w1_full[t])), "r"(1) : "memory");
            for (int t = 0; t < p.w2_slots; ++t) {
                asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&tail.w2_full[t])), "r"(1) : "memory");
                asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&tail.w2_empty[t])), "r"(1) : "memory");
            }
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(&p.tmx) : "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(&p.tmw1) : "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(&p.tmw2) : "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(&p.tmy) : "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(sm32(&tail.tmem)), "r"(kGtTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    auto header_ok = [&](int type) {
        const bool one = gt_header_ok(p.packed1, type, p.O1, p.I1, p.H, p.K, p.bo1, p.bi1), two = gt_header_ok(p.packed2, type, p.O2, p.O1, 1, 1, p.bo2, p.bi2);
        return one && two;
    };
    const bool early = tid == 0 && header_ok(p.early_type);
    wait_for_previous<false>();
    if (warp == 0) let_next_start();                  // (behind its allocation)
    if (tid == 0) {
        const bool ok = early || header_ok(p.wtype);
        const bool placed = (base & 1023u) == 0u;
        s_fail = ok && placed ? 0u : 2u;
        if (!ok) atomicMax(p.status, (int)BSP_ERR_INDEX);
        else if (!placed) atomicMax(p.status, (int)BSP_ERR_CUDA);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, tail.tmem, 0);
    const bool run = __shfl_sync(0xFFFFFFFFu, s_fail, 0) == 0u;
    const uint32_t full0 = sm32(&tail.full[0]), empty0 = sm32(&tail.empty[0]);

    if (warp == 0) {
        // ================= producer =================
        if (run) {
            const uint32_t stage_bytes = (uint32_t)p.stage_bytes;
            const uint32_t tx1 = (uint32_t)(p.a_bytes + (kHalo ? 0 : p.O1p * 128)), tx2 = (uint32_t)(kCtBN2 * 128);
            const int cpt128 = p.cpt1 * 128, Kw = p.K;
            uint32_t slot = 0, epar = 1, issued = 0, dst = ring;      // (a fresh barrier counts as released)
            uint32_t slot2 = 0, epar2 = 1, issued2 = 0;
            bool ok = true, free_now = true;
            // layer one of a tile: per 128-byte chunk of channels of a tap, the activation box shifted by the tap and the tap's
            // weights; kHalo: one box (of each plane), and with the first tile the weights of all taps
            auto load_layer_one = [&](int tile) {
                int n0, y0, x0;
                ct_tile_origin(p, tile, n0, y0, x0);
                const int xi0 = x0 * p.sw - p.pw;
                if constexpr (kHalo) {
                    if (!free_now && !__all_sync(0xFFFFFFFFu, gt_poll(empty0 + slot * 8u, epar))) { ok = false; return; }
                    const bool wrap = slot + 1u == (uint32_t)S;
                    const uint32_t next_free = gt_test(empty0 + (wrap ? 0u : slot + 1u) * 8u, wrap ? epar ^ 1u : epar);
                    asm volatile("{\n .reg .pred e, e1;\n elect.sync _|e, 0xFFFFFFFF;\n setp.ne.b32 e1, %8, 0;\n and.pred e1, e1, e;\n"
                                 " @e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n"
                                 " @e cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%2], [%3, {%4, %5, %6, %7}], [%0];\n"
                                 " @e1 cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%9], [%3, {%10, %5, %6, %7}], [%0];\n}\n"
                                 ::"r"(full0 + slot * 8u), "r"(tx1), "r"(dst), "l"(&p.tmx), "r"(0), "r"(xi0), "r"(y0 * p.sh - p.ph), "r"(n0),
                                   "r"(p.planes - 1), "r"(dst + (uint32_t)p.plane_bytes), "r"(32) : "memory");
                    ++issued;
                    free_now = __all_sync(0xFFFFFFFFu, next_free != 0u);
                    if (wrap) { slot = 0; epar ^= 1u; dst = ring; } else { ++slot; dst += stage_bytes; }
                    if (tile == t_first)
                        for (int t = 0; t < p.n_ks1; ++t) {
                            const uint32_t w = base + (uint32_t)(t * p.O1p * p.kbytes);
                            asm volatile("{\n .reg .pred e, e1;\n elect.sync _|e, 0xFFFFFFFF;\n setp.ne.b32 e1, %7, 0;\n and.pred e1, e1, e;\n"
                                         " @e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n"
                                         " @e cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%2], [%3, {%4, %5, %6}], [%0];\n"
                                         " @e1 cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%8], [%3, {%9, %5, %6}], [%0];\n}\n"
                                         ::"r"(sm32(&tail.w1_full[t])), "r"((uint32_t)(p.O1p * p.kbytes)), "r"(w), "l"(&p.tmw1), "r"(0), "r"(t), "r"(0),
                                           "r"(p.planes - 1), "r"(w + (uint32_t)(p.O1p * 32)), "r"(32) : "memory");
                        }
                } else {
                    int c128 = 0, kx = xi0, hy = y0 * p.sh - p.ph, tap = 0, kk = 0;
                    for (int ks = 0; ks < p.n_ks1; ++ks) {
                        if (!free_now && !__all_sync(0xFFFFFFFFu, gt_poll(empty0 + slot * 8u, epar))) { ok = false; return; }
                        const bool wrap = slot + 1u == (uint32_t)S;
                        const uint32_t next_free = gt_test(empty0 + (wrap ? 0u : slot + 1u) * 8u, wrap ? epar ^ 1u : epar);
                        asm volatile("{\n .reg .pred e;\n elect.sync _|e, 0xFFFFFFFF;\n"
                                     " @e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n"
                                     " @e cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%2], [%3, {%4, %5, %6, %7}], [%0];\n"
                                     " @e cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%8], [%9, {%4, %10, %11}], [%0];\n}\n"
                                     ::"r"(full0 + slot * 8u), "r"(tx1), "r"(dst), "l"(&p.tmx), "r"(c128), "r"(kx), "r"(hy), "r"(n0),
                                       "r"(dst + (uint32_t)kGtABytes), "l"(&p.tmw1), "r"(tap), "r"(0) : "memory");
                        ++issued;
                        free_now = __all_sync(0xFFFFFFFFu, next_free != 0u);
                        if (wrap) { slot = 0; epar ^= 1u; dst = ring; } else { ++slot; dst += stage_bytes; }
                        c128 += 128;
                        if (c128 == cpt128) {
                            c128 = 0; ++tap; ++kx;
                            if (++kk == Kw) { kk = 0; kx = xi0; ++hy; }
                        }
                    }
                }
            };
            // layer two: for every tile of 128 output channels, the weight chunk of each 128 bytes of T's channels
            auto load_layer_two = [&](int tile) {
                if (kHalo && p.w2_stay && tile != t_first) return;
                for (int t2 = 0; t2 < p.n_t2; ++t2)
                    for (int c2 = 0; c2 < p.n_c2; ++c2) {
                        uint32_t bar, to;
                        if constexpr (kHalo) {
                            if (!__all_sync(0xFFFFFFFFu, gt_poll(sm32(&tail.w2_empty[slot2]), epar2))) { ok = false; return; }
                            bar = sm32(&tail.w2_full[slot2]);
                            to = base + p.off_w2 + slot2 * tx2;
                            ++issued2;
                            if (++slot2 == (uint32_t)p.w2_slots) { slot2 = 0; epar2 ^= 1u; }
                        } else {
                            if (!free_now && !__all_sync(0xFFFFFFFFu, gt_poll(empty0 + slot * 8u, epar))) { ok = false; return; }
                            const bool wrap = slot + 1u == (uint32_t)S;
                            const uint32_t next_free = gt_test(empty0 + (wrap ? 0u : slot + 1u) * 8u, wrap ? epar ^ 1u : epar);
                            bar = full0 + slot * 8u;
                            to = dst;
                            ++issued;
                            free_now = __all_sync(0xFFFFFFFFu, next_free != 0u);
                            if (wrap) { slot = 0; epar ^= 1u; dst = ring; } else { ++slot; dst += stage_bytes; }
                        }
                        asm volatile("{\n .reg .pred e;\n elect.sync _|e, 0xFFFFFFFF;\n"
                                     " @e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n"
                                     " @e cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%2], [%3, {%4, %5, %6}], [%0];\n}\n"
                                     ::"r"(bar), "r"(tx2), "r"(to), "l"(&p.tmw2), "r"(c2 * 128), "r"(0), "r"(o2 + t2 * kCtBN2) : "memory");
                    }
            };
            // the loads follow the order in which the MMA warp consumes them: with double buffers, layer one of the next
            // tile goes before layer two of this one
            if (p.db && t_first < t_count) load_layer_one(t_first);
            for (int tile = t_first; tile < t_count && ok; tile += t_step) {
                if (s_fail) { ok = false; break; }
                if (p.db) { if (tile + t_step < t_count) load_layer_one(tile + t_step); }
                else load_layer_one(tile);
                if (ok) load_layer_two(tile);
            }
            if (!ok && lane == 0) {
                // winding down after a wait that ran out: the loads already issued still write into this CTA's shared
                // memory, so the barriers of the stages in flight are awaited (bounded) before the CTA may leave
                atomicExch((uint32_t *)&tail.fail, 1u);
                for (uint32_t back = 0; back < (uint32_t)S && back < issued; ++back) {
                    const uint32_t it = issued - 1u - back;
                    gt_poll(full0 + (it % (uint32_t)S) * 8u, (it / (uint32_t)S) & 1u);
                }
                if constexpr (kHalo) {
                    if (issued > 0)
                        for (int t = 0; t < p.n_ks1; ++t) gt_poll(sm32(&tail.w1_full[t]), 0u);
                    for (uint32_t back = 0; back < (uint32_t)p.w2_slots && back < issued2; ++back) {
                        const uint32_t it = issued2 - 1u - back;
                        gt_poll(sm32(&tail.w2_full[it % (uint32_t)p.w2_slots]), (it / (uint32_t)p.w2_slots) & 1u);
                    }
                }
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer =================
        if (run) {
            // instruction descriptors: A and B bf16 (signed int8), K-major both, M = 128; N = O1p for layer one, 128 for layer two
            const uint32_t dfmt = kI8 ? 2u : 1u;      // D int32 for int8 operands, fp32 otherwise
            const uint32_t idesc1 = (dfmt << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.O1p >> 3) << 17) | ((128u >> 4) << 24);
            const uint32_t idesc2 = (dfmt << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kCtBN2 >> 3) << 17) | ((128u >> 4) << 24);
            const uint32_t stage16 = (uint32_t)p.stage_bytes >> 4;
            uint32_t slot = 0, par = 0, a16 = ring >> 4, tile_i = 0, u2 = 0, slot2 = 0, par2 = 0;
            bool ok = true, full_now = false, full2_now = false;
            // the taps of a kHalo tile (see the product kernel)
            auto taps = [&](auto wide_c, auto first_c, uint32_t d) -> bool {
                constexpr bool kWide = decltype(wide_c)::value, kFirst = decltype(first_c)::value;
                constexpr uint64_t shape = kWide ? kGtDesc : kGtDesc32;
                const uint32_t row16 = kWide ? 8u : 2u, w_tap16 = (uint32_t)(p.O1p * p.kbytes) >> 4, row_step = (uint32_t)(p.halo_w - p.K) * row16;
                const uint64_t plane_a = (uint64_t)(p.plane_bytes >> 4), plane_b = (uint64_t)(p.O1p * 32 >> 4);
                const uint32_t two = (uint32_t)p.planes - 1u;
                uint64_t da = (kEights ? gt_desc_groups(shape, (uint32_t)p.halo_w * row16) : shape) | (uint64_t)a16, db = shape | (uint64_t)(base >> 4);
                uint32_t acc = 0u;
                int t = 0;
#pragma unroll 1
                for (int h = 0; h < p.H; ++h, da += row_step)
#pragma unroll 1
                    for (int k = 0; k < p.K; ++k, ++t, da += row16, db += w_tap16) {
                        if constexpr (kFirst) {
                            if (!__all_sync(0xFFFFFFFFu, gt_poll(sm32(&tail.w1_full[t]), 0u))) return false;
                            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                        }
                        if constexpr (kWide) gt_issue_tap<kWt>(d, da, db, idesc1, acc);
                        else gt_issue_planes<kWt>(d, da, db, plane_a, plane_b, two, idesc1, acc);
                        acc = 1u;
                    }
                return true;
            };
            // layer one of the CTA's i-th tile into accumulator one (buffer b, used for the u-th time)
            auto layer_one = [&](uint32_t i) {
                const uint32_t b = p.db ? (i & 1u) : 0u, u = p.db ? (i >> 1) : i;
                // the buffer is free once the first epilogue of its previous tile has read it
                if (!gt_poll(sm32(&tail.acc1_empty[b]), (u & 1u) ^ 1u) || s_fail != 0u) ok = false;
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) return;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint32_t d = tmem + b * 128u;
                if constexpr (kHalo) {
                    if (!__all_sync(0xFFFFFFFFu, gt_poll(full0 + slot * 8u, par))) { ok = false; return; }
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    if (p.kbytes == 128) { if (i == 0u) ok = taps(std::true_type(), std::true_type(), d); else taps(std::true_type(), std::false_type(), d); }
                    else { if (i == 0u) ok = taps(std::false_type(), std::true_type(), d); else taps(std::false_type(), std::false_type(), d); }
                    if (!ok) return;
                    gt_commit_elected<false>(empty0 + slot * 8u);
                    if (++slot == (uint32_t)S) { slot = 0; par ^= 1u; a16 = ring >> 4; } else a16 += stage16;
                } else {
                    for (int ks = 0; ks < p.n_ks1; ++ks) {
                        if (!full_now && !gt_poll_stage(full0 + slot * 8u, par)) { ok = false; return; }
                        const bool wrap = slot + 1u == (uint32_t)S;
                        const uint64_t da = kGtDesc | (uint64_t)(a16 & 0x3FFFu), db = kGtDesc | (uint64_t)((a16 + (kGtABytes >> 4)) & 0x3FFFu);
                        full_now = gt_issue_stage<kWt, false>(d, da, db, idesc1, empty0 + slot * 8u, ks != 0 ? 1u : 0u, 4u,
                                                              full0 + (wrap ? 0u : slot + 1u) * 8u, wrap ? par ^ 1u : par) != 0u;
                        if (wrap) { slot = 0; par ^= 1u; a16 = ring >> 4; } else { ++slot; a16 += stage16; }
                    }
                }
                gt_commit_elected<false>(sm32(&tail.acc1_full[b]));
            };
            // layer two of the i-th tile: the tensor between the layers is in shared memory once the first epilogue has written it
            auto layer_two = [&](uint32_t i) {
                const uint32_t b = p.dbt ? (i & 1u) : 0u, u = p.dbt ? (i >> 1) : i;
                if (!gt_poll(sm32(&tail.t_full[b]), u & 1u)) ok = false;
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) return;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                if (kHalo && p.w2_stay) { slot2 = 0; par2 = 0; }
                for (int t2 = 0; t2 < p.n_t2 && ok; ++t2, ++u2) {
                    const uint32_t buf = u2 & 1u, use = u2 >> 1;
                    if (!gt_poll(sm32(&tail.acc2_empty[buf]), (use & 1u) ^ 1u)) ok = false;
                    ok = __all_sync(0xFFFFFFFFu, ok);
                    if (!ok) return;
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    const uint32_t d = tmem + 256u + buf * (uint32_t)kCtBN2;
                    for (int c2 = 0; c2 < p.n_c2; ++c2) {
                        const uint64_t da = kGtDesc | (uint64_t)(((tbuf + b * tbytes + (uint32_t)(c2 * kCtChunk)) >> 4) & 0x3FFFu);
                        if constexpr (kHalo) {
                            if (!full2_now && !gt_poll_stage(sm32(&tail.w2_full[slot2]), par2)) { ok = false; return; }
                            const bool wrap = slot2 + 1u == (uint32_t)p.w2_slots;
                            const uint64_t db = kGtDesc | (uint64_t)((base + p.off_w2 + slot2 * (uint32_t)(kCtBN2 * 128)) >> 4);
                            // (weights that stay are never handed back: the arrivals on their barriers go unread)
                            // (and weights that stay have arrived for good once the first tile is done)
                            full2_now = gt_issue_stage<kWt, false>(d, da, db, idesc2, sm32(&tail.w2_empty[slot2]), c2 != 0 ? 1u : 0u, 4u,
                                                                   sm32(&tail.w2_full[wrap ? 0u : slot2 + 1u]), wrap && !p.w2_stay ? par2 ^ 1u : par2) != 0u;
                            if (wrap) { slot2 = 0; par2 ^= 1u; } else ++slot2;
                        } else {
                            if (!full_now && !gt_poll_stage(full0 + slot * 8u, par)) { ok = false; return; }
                            const bool wrap = slot + 1u == (uint32_t)S;
                            full_now = gt_issue_stage<kWt, false>(d, da, kGtDesc | (uint64_t)(a16 & 0x3FFFu), idesc2, empty0 + slot * 8u, c2 != 0 ? 1u : 0u, 4u,
                                                                  full0 + (wrap ? 0u : slot + 1u) * 8u, wrap ? par ^ 1u : par) != 0u;
                            if (wrap) { slot = 0; par ^= 1u; a16 = ring >> 4; } else { ++slot; a16 += stage16; }
                        }
                    }
                    gt_commit_elected<false>(sm32(&tail.acc2_full[buf]));
                }
                // all MMAs that read the tensor have been issued: their completion frees its buffer
                gt_commit_elected<false>(sm32(&tail.t_empty[b]));
            };
            if (p.db && t_first < t_count) layer_one(0u);
            for (int tile = t_first; tile < t_count && ok; tile += t_step, ++tile_i) {
                if (p.db) { if (tile + t_step < t_count) layer_one(tile_i + 1u); }
                else layer_one(tile_i);
                if (ok) layer_two(tile_i);
                if (ok && tile + t_step < t_count && tile + 2 * t_step >= t_count) gt_commit_elected<false>(sm32(&tail.before_last));
            }
            if (!ok && lane == 0) atomicExch((uint32_t *)&tail.fail, 1u);
        }
    } else {
        // ================= epilogues (warps 2-9, kHalo 2-13) =================
        // The work goes in steps: the n_c2 chunks of T of tile s + ahead, then the 128-byte rounds of Y of tile s; the groups take
        // turns with these rounds, across steps too.  With ahead = 1 the MMA warp finds the next T ready when it is
        // done with this tile (else layer two of a tile waited for both of the previous tile's epilogues).
        if (run) {
            const int q = warp & 3;                              // quarter of the tensor-memory lanes this warp reaches
            const int grp = (warp - 2) >> 2;
            // the group's staging buffer: 128 rows of 128 bytes
            const uint32_t sg = staging + (uint32_t)grp * p.staging_bytes;
            const bool issuer = q == 0 && lane == 0;             // one thread of the group issues its stores
            const int r = q * 32 + lane;                         // this lane's row of a tile
            int row = r;                                         // its row of the staging buffer (kHalo: the place in the box, or none)
            if constexpr (kHalo) row = gt_halo_row(r, kEights, p.Wt, p.Ht, p.Nt, p.halo_w, p.halo_rows);
            // constants of a round's channels, fetched one round ahead (thread c holds channel c)
            uint32_t *bias = tail.bias[grp], *half = tail.half[grp];
            uint8_t *shift = tail.shift[grp];
            const int ct = ((warp - 2) & 3) * 32 + lane;
            bool mine = true;                                    // (the look that decides, by one thread, on its way while the tile is made)
            if (tid == 64) mine = header_ok(p.wtype);
            const uint32_t *bias1 = from_here((const uint32_t *)p.bias1), *bias2 = from_here((const uint32_t *)p.bias2);
            const int32_t *shift1 = from_here(p.shift1), *shift2 = from_here(p.shift2);
            uint32_t next_bias = 0u, next_shift = 1u;
            bool small = false;
            const int n_rounds = p.n_c2 + p.n_t2 * kRpt;
            // A barrier's parity tells a phase from the next one only, so a group may look at a phase when it knows that the one
            // before it has completed.  What tells it, for each barrier (all rest on the commits of the MMA warp completing in the
            // order of its loop):
            //   acc2_full   of tile s: the group had its last look no further back than T of tile s + 1, if T runs ahead, or
            //               than the use of the other accumulator before the phase in question, and either comes after the
            //               buffer's previous use.  In the last tile, which has no such T, before_last stands in for it.
            //               With one round per tile of layer two and three groups this does not hold, and the reads of the
            //               previous use are counted (below).  (Checked over all orders in which the barriers can complete, for
            //               up to six tiles and five tiles of layer two, in every form.)
            //   acc1_full   of tile i: its previous phase is that of tile i - 2 (two accumulators) or i - 1 (one).  The group had a
            //               round in step i - 1 - ahead, as a step has at least as many rounds as there are groups (hence two
            //               groups for steps of two): T of tile i - 1, or Y of tile i - 1 - ahead, which came after it.
            //   t_empty     of the tile before in the same buffer: acc1_full of tile i, which the group has waited for just
            //               before, comes after layer two of tile i - 2 (i - 1 with one accumulator).
            const int groups = n_rounds < kGroups ? 2 : kGroups;
            auto fetch = [&](int rnd) {
                const bool one = rnd < p.n_c2;
                const int ch = (one ? rnd * p.tcc : o2 + (rnd - p.n_c2) * cpr) + ct, O = one ? p.O1 : p.O2;
                const uint32_t *b = one ? bias1 : bias2;
                const int32_t *s = one ? shift1 : shift2;
                const bool in = ct < (one ? p.tcc : cpr) && ch < O;
                next_bias = in && b != nullptr ? load_free(b + ch) : 0u;
                if constexpr (kI8) next_shift = in && s != nullptr ? (uint32_t)load_free(s + ch) & 31u : 1u;
            };
            bool mine_small = false, fresh = true;
            auto place = [&](int rnd) {                          // (between two barriers of the group)
                fresh = true;
                if constexpr (kI8)
                    mine_small = (rnd < p.n_c2 ? p.small1 : p.small2) != 0 && next_shift != 0u && next_shift != 31u && (int)next_bias <= (1 << 29) && (int)next_bias >= -(1 << 29);
                bias[ct] = next_bias;
                if constexpr (kI8) { half[ct] = (1u << next_shift) >> 1; shift[ct] = (uint8_t)next_shift; }
            };
            const int n_local = t_first < t_count ? (t_count - t_first + t_step - 1) / t_step : 0;       // tiles of this CTA
            int step = grp < groups ? -p.ahead : n_local, rnd = grp;
            bool ok = true;
            while (rnd >= n_rounds) { rnd -= n_rounds; ++step; }
            if (step < n_local) { fetch(rnd); place(rnd); }
            if (tid == 64) {
                tail.refused = mine ? 0u : 1u;
                if (!mine) atomicMax(p.status, (int)BSP_ERR_INDEX);
            }
            asm volatile("bar.sync 4, %0;\n" ::"n"(128 * kGroups) : "memory");      // (all groups)
            const bool store = tail.refused == 0u;
            while (step < n_local) {
                int next = rnd + groups, next_step = step;
                while (next >= n_rounds) { next -= n_rounds; ++next_step; }
                const bool change = next != rnd;
                if (change) fetch(next);
                const bool one = rnd < p.n_c2;
                const int idx = one ? step + p.ahead : step;     // which of the CTA's tiles
                const uint32_t tile_i = (uint32_t)idx;
                if (idx < 0 || idx >= n_local) {                 // (before the first Y, after the last T)
                    if (s_fail) ok = false;
                    if (idx >= n_local && n_local > 1 && ok && !gt_wait(sm32(&tail.before_last), 0u)) ok = false;
                    if (change) { gt_group_sync(1 + grp); place(next); gt_group_sync(1 + grp); }
                    rnd = next; step = next_step;
                    continue;
                }
                // what the round waits for: accumulator one and a free T (the MMAs of the second layer that read it have
                // completed), or accumulator two (int8: and a staging buffer that its last store has read)
                const int t2 = one ? 0 : (rnd - p.n_c2) / kRpt, c0 = one ? 0 : (rnd - p.n_c2) % kRpt * cpr, n0 = o2 + t2 * kCtBN2;
                const uint32_t b1 = p.db ? (tile_i & 1u) : 0u, u1 = p.db ? (tile_i >> 1) : tile_i;
                const uint32_t bt = p.dbt ? (tile_i & 1u) : 0u, ut = p.dbt ? (tile_i >> 1) : tile_i;
                const uint32_t u2 = tile_i * (uint32_t)p.n_t2 + (uint32_t)t2, buf = u2 & 1u, use = u2 >> 1;
                // A wait that ran out is latched below; the group goes on (its warps meet at barriers) and waits no more.
                if (s_fail) ok = false;
                if (one) {
                    if (ok && (!gt_wait(sm32(&tail.acc1_full[b1]), u1 & 1u) || !gt_wait(sm32(&tail.t_empty[bt]), (ut & 1u) ^ 1u))) ok = false;
                } else {
                    // (With one round per tile of layer two, a group of three may come to this phase while the barrier is still
                    // two before it, which the parity cannot tell from done.  So first the previous use of the buffer is seen
                    // to have been read, by a count: layer two waits for that anyway.  The parity of the other buffer's barrier
                    // would not do, as that one may have moved on by two phases already.)
                    if (kGroups > 2 * kRpt && ok && !ct_wait_count(&tail.y_read[buf], use * (uint32_t)(4 * kRpt))) ok = false;
                    if (ok && !gt_wait(sm32(&tail.acc2_full[buf]), use & 1u)) ok = false;
                    if (kEy == 1) {
                        if (issuer) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
                        if (!fresh) gt_group_sync(1 + grp);
                    }
                }
                if (kI8 && fresh) small = gt_group_all(1 + grp, mine_small);
                fresh = false;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint32_t lanes = tmem + ((uint32_t)(q * 32) << 16);
                const uint32_t sw = (uint32_t)(one ? lane : row) & 7u;
                // (an accumulator is handed back as soon as it has been read)
                auto hand_back = [&](uint64_t *bar) {
                    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                    __syncwarp();
                    if (kGroups > 2 * kRpt && !one && lane == 0) atomicAdd(&tail.y_read[buf], 1u);
                    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(sm32(bar)) : "memory");
                };
                if (one) {
                    // ---- first epilogue: accumulator one -> + b1 -> activation -> T in shared memory, K-major rows of 128 bytes ----
                    const uint32_t tcol = lanes + b1 * 128u + (uint32_t)(rnd * p.tcc), trow = tbuf + bt * tbytes + (uint32_t)(rnd * kCtChunk + r * 128);
                    if constexpr (kI8) {
                        gt_epilogue_int8<true>(tcol, bias, half, shift, small, p.O1 - rnd * p.tcc, p.relu, trow, sw, true);
                        hand_back(&tail.acc1_empty[b1]);
                    } else {
                        uint32_t out[32];
                        gt_epilogue_round<false, 2, true>(tcol, bias, p.O1 - rnd * p.tcc, p.relu, out);
                        hand_back(&tail.acc1_empty[b1]);
                        gt_store_round(trow, sw, true, out);
                    }
                    // the MMAs read T through the asynchronous proxy
                    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                    __syncwarp();
                    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(sm32(&tail.t_full[bt])) : "memory");
                    if (change) { gt_group_sync(1 + grp); place(next); gt_group_sync(1 + grp); }
                } else {
                    // ---- second epilogue: + b2 -> convert -> staging -> the tile's box of Y by one TMA store; what lies past the
                    // last channel, column, row or image of Y is clipped ----
                    const uint32_t tcol = lanes + 256u + buf * (uint32_t)kCtBN2 + (uint32_t)c0, srow = sg + (uint32_t)row * 128u;
                    if constexpr (kEy == 1) {
                        gt_epilogue_int8<false>(tcol, bias, half, shift, small, p.O2 - n0 - c0, 0, srow, sw, row >= 0);
                        hand_back(&tail.acc2_empty[buf]);
                    } else {
                        uint32_t out[32];
                        gt_epilogue_round<kI8, kEy, false>(tcol, bias, p.O2 - n0 - c0, 0, out);
                        hand_back(&tail.acc2_empty[buf]);
                        // (loads and arithmetic run while the last store reads the staging buffer)
                        if (issuer) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
                        gt_group_sync(1 + grp);
                        if (change) place(next);
                        gt_store_round(srow, sw, row >= 0, out);
                    }
                    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                    gt_group_sync(1 + grp);
                    if (kEy == 1 && change) place(next);
                    if (issuer && n0 + c0 < p.O2 && store) {
                        int in0, y0, x0;
                        ct_tile_origin(p, t_first + idx * t_step, in0, y0, x0);
                        asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];\n"
                                     ::"l"(&p.tmy), "r"(sg), "r"((n0 + c0) * kEy), "r"(x0), "r"(y0), "r"(in0) : "memory");
                        asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
                    }
                }
                rnd = next; step = next_step;
            }
            if (issuer) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");      // (the stores have read this CTA's memory)
            if (!ok && lane == 0) atomicExch((uint32_t *)&tail.fail, 1u);
        }
    }

    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (s_fail == 1u && tid == 0) atomicMax(p.status, (int)BSP_ERR_TIMEOUT);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kGtTmemCols) : "memory");
}

}  // namespace

// True if the fused kernel can run this pair: two bfloat16 or two int8 layers, a 1x1 second layer on the first one's
// output channels, at most 256 of them (accumulator one holds them all), rows of X, of both weights and of Y that are
// multiples of 16 bytes.
bool chain_tc_eligible(const bsp_wdesc &wd1, const bsp_wdesc &wd2, const bsp_xdesc &xd0, bsp_dtype ytype)
{
    if (wd1.wtype != wd2.wtype || (wd1.wtype != BSP_BF16 && wd1.wtype != BSP_I8)) return false;
    if (wd2.H != 1 || wd2.K != 1 || wd2.I != wd1.O) return false;
    if (wd1.O > 256 || wd1.O % 8 != 0 || wd1.I % 8 != 0 || wd2.O % 8 != 0) return false;
    const int esz = elem_bytes(wd1.wtype);
    if (wd1.wtype == BSP_I8) { if (ytype != BSP_I32 && ytype != BSP_I8) return false; }
    else if (ytype != BSP_F32 && ytype != BSP_BF16) return false;
    const int ey = ytype == BSP_BF16 ? 2 : (ytype == BSP_I8 ? 1 : 4);
    if ((wd1.I * esz) % 16 != 0 || (wd1.O * esz) % 16 != 0 || (wd2.O * ey) % 16 != 0) return false;
    if (!packed_layout(wd1).enabled || !packed_layout(wd2).enabled) return false;
    const bsp_xdesc xd = gt_flatten(wd1, xd0);
    const int M = (xd.L + 2 * xd.pad_h - wd1.H) / xd.stride_h + 1, Nw = (xd.J + 2 * xd.pad_w - wd1.K) / xd.stride_w + 1;
    if (M <= 0 || Nw <= 0) return false;
    if ((long long)xd.N * M * Nw > 0x7FFFFFFF - 4096 || (long long)xd.N * xd.L * xd.J > 0x7FFFFFFF) return false;
    return xd.stride_h <= 256 && xd.stride_w <= 256;       // (a box of one position then fits: gt_pick_tile)
}

bsp_status launch_chain_tc(const bsp_wdesc &wd1, const void *packed1, const bsp_wdesc &wd2, const void *packed2,
                           const bsp_xdesc &xd0, const void *X, const void *bias1, const int32_t *shift1, int relu,
                           const void *bias2, const int32_t *shift2, void *Y, bsp_dtype ytype, void *ws, cudaStream_t st)
{
    const bsp_xdesc xd = gt_flatten(wd1, xd0);
    const PackedLayout L1 = packed_layout(wd1), L2 = packed_layout(wd2);
    if (!L1.enabled || !L2.enabled) return BSP_ERR_SHAPE;
    const int ey = ytype == BSP_BF16 ? 2 : (ytype == BSP_I8 ? 1 : 4);
    const int esz = elem_bytes(wd1.wtype);
    if (wd1.wtype == BSP_I8 && (shift1 == nullptr || (ytype == BSP_I8 && shift2 == nullptr))) return BSP_ERR_NULL;
    CtParams p = {};
    p.bias1 = bias1; p.bias2 = bias2; p.shift1 = shift1; p.shift2 = shift2; p.wtype = wd1.wtype; p.packed1 = (const uint8_t *)packed1; p.packed2 = (const uint8_t *)packed2;
    p.status = (int *)ws;
    p.O1 = wd1.O; p.I1 = wd1.I; p.H = wd1.H; p.K = wd1.K; p.bo1 = wd1.bo; p.bi1 = wd1.bi;
    p.O2 = wd2.O; p.bo2 = wd2.bo; p.bi2 = wd2.bi; p.relu = relu ? 1 : 0;
    p.tcc = 128 / esz;
    p.O1p = (wd1.O + p.tcc - 1) / p.tcc * p.tcc;
    p.early_type = packed_spans(wd1, packed1) && packed_spans(wd2, packed2) ? (int)wd1.wtype : -1;
    p.N = xd.N; p.sh = xd.stride_h; p.sw = xd.stride_w; p.ph = xd.pad_h; p.pw = xd.pad_w;
    p.M = (xd.L + 2 * xd.pad_h - wd1.H) / xd.stride_h + 1;
    p.Nw = (xd.J + 2 * xd.pad_w - wd1.K) / xd.stride_w + 1;
    GtTile T = gt_pick_tile(xd.N, p.M, p.Nw, p.sh, p.sw);
    if (T.tiles <= 0 || T.tiles > 0x7FFFFFFF - 4096) return BSP_ERR_SHAPE;
    const int HK = wd1.H * wd1.K, row1 = wd1.I * esz;
    p.cpt1 = (row1 + 127) / 128;
    p.n_ks1 = HK * p.cpt1;
    p.n_c2 = p.O1p / p.tcc;
    p.n_t2 = (wd2.O + kCtBN2 - 1) / kCtBN2;
    p.parts = 1;
    static int n_sm[kGtMaxDevices] = {};
    int dev = 0;
    BSP_CUDA_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kGtMaxDevices) return BSP_ERR_CUDA;
    if (n_sm[dev] == 0) BSP_CUDA_OK(cudaDeviceGetAttribute(&n_sm[dev], cudaDevAttrMultiProcessorCount, dev));
    const GtHaloTile Th = gt_pick_halo(xd.N, p.M, p.Nw, wd1.H, wd1.K);
    // Where the position tiles fill less than half of the SMs, several CTAs take one: each computes T for itself and its share of
    // layer two's channels.  (Two 128-channel tiles of Y take about 1.2 us one after the other: 7x1 128->64->928 at 11x11 13.0 -> 6.6 us,
    // 3x3 64->80->768 at 22x22 12.3 -> 7.4, 1x1 96->128->592 at 34x34, batch 8, 14.9 -> 11.6.)
    const long long most = Th.tiles > T.tiles ? Th.tiles : T.tiles;
    // As many as fit, but where layer one's rows are not whole 32-byte sectors of L2.  Such rows cost twice the time of a CTA, and
    // 1.4 times that on more than half of the SMs, whatever their number: those layers take the CTAs with the lowest estimate, a
    // tile of Y being 1.2 us (4-byte output 1.8).  3x3 216->88, 1x1 88->336 at 40x40, batch 5, 20.8 us a call on 63 CTAs and 25.0 on
    // 126; 8 bits 3x3 208->64, 1x1 64->336 14.8 and 20.1.  (Over 1056 pairs with such rows 6 % faster than as many as fit; over
    // 2376 with rows of whole sectors half of the SMs were 7 % slower.)
    const bool stays = HK > 1 && HK <= kCtTaps && p.cpt1 == 1 && p.sh == 1 && p.sw == 1 && p.O1p <= 128 && Th.tiles > 0 && Th.tiles * 4 <= T.tiles * 5;
    if (most * 2 <= n_sm[dev] && p.n_t2 > 1) {
        const int planes = row1 <= 32 || row1 > 64 ? 1 : 2;
        const double rows = row1 % 32 == 0 ? 0.0 : stays ? HK * planes * p.O1p : p.n_ks1 * (kGtBM + p.O1p);
        const long long tiles = stays ? Th.tiles : T.tiles;
        const int n_all = p.n_t2;
        double best = -1.0;
        for (int parts = 1; parts <= n_sm[dev] / most && parts <= n_all; ++parts) {
            const int n = (n_all + parts - 1) / parts, used = (wd2.O + kCtBN2 * n - 1) / (kCtBN2 * n);
            const double t = rows * 3.0 / 1900.0 * (used * tiles * 2 <= n_sm[dev] ? 1.0 : 1.4) + (ey == 4 ? 1.8 : 1.2) * n;
            if (best < 0 || t < best) { best = t; p.n_t2 = n; p.parts = used; }
        }
    }
    p.db = p.O1p <= 128 ? 1 : 0;
    p.dbt = p.db;
    p.kbytes = 128; p.planes = 1;
    p.small1 = (long long)row1 * HK * 128 * 128 <= (1 << 29) ? 1 : 0;
    p.small2 = (long long)wd1.O * 128 * 128 <= (1 << 29) ? 1 : 0;
    const int fixed = ct_groups(false) * 4 * kGtStagingBytes + (int)sizeof(CtTail<2>);
    // kHalo: where two boxes of activations, the weights of layer one and at least two chunks of layer two's fit, and the
    // tiles with their border are not many more.  3x3 64->64 then 64->256 at 56x56, batch 64, in a short burst: 44.5 us loaded
    // tap by tap, 33.8 like this (36 in a stream of calls).
    bool halo = false, eights = false;
    int w2_slots = 0;
    if (stays) {
        const int kb = row1 <= 32 ? 32 : (row1 <= 64 ? 64 : 128), planes = kb == 128 ? 1 : kb / 32;
        const int plane = (Th.Nt * (Th.Ht + wd1.H - 1) * (Th.Wt + wd1.K - 1) * (kb / planes) + 1023) / 1024 * 1024;
        p.staging_bytes = (uint32_t)(Th.Wt * Th.Ht * Th.Nt * 128 + 1023) / 1024 * 1024;
        const int fixed_h = ct_groups(true) * (int)p.staging_bytes + (int)sizeof(CtTail<3>);
        const int room = kCtSmem - fixed_h - p.n_c2 * kCtChunk - HK * p.O1p * kb - 2 * planes * plane;
        const int room2 = room - p.n_c2 * kCtChunk;          // with two buffers for T
        int want = p.n_t2 * p.n_c2;
        if (want > kCtW2Slots) want = kCtW2Slots;
        const int one_t = room / (kCtBN2 * 128), two_t = room2 / (kCtBN2 * 128);
        // (a second buffer for T before the weights of layer two stay, where the tile does not fit both accumulators)
        const bool second = two_t >= want || (p.n_t2 > 2 && two_t >= 2);
        w2_slots = second ? two_t : one_t;
        if (w2_slots > want) w2_slots = want;
        if (w2_slots >= 2 || w2_slots == p.n_t2 * p.n_c2) {
            halo = true;
            T = Th;
            p.kbytes = kb; p.planes = planes; p.plane_bytes = plane; eights = Th.eights != 0;
            p.dbt = second ? 1 : 0;
            p.w2_slots = w2_slots; p.w2_stay = w2_slots == p.n_t2 * p.n_c2 ? 1 : 0;
            p.halo_w = T.Wt + wd1.K - 1; p.halo_rows = T.Ht + wd1.H - 1;
        }
    }
    if (!halo && T.tiles > n_sm[dev]) T = gt_pick_packed(T, xd.N, p.M, p.Nw, p.sh, p.sw);
    p.Wt = T.Wt; p.Ht = T.Ht; p.Nt = T.Nt;
    p.tiles_x = (p.Nw + T.Wt - 1) / T.Wt; p.tiles_y = (p.M + T.Ht - 1) / T.Ht;
    p.m_tx = gt_magic(p.tiles_x); p.m_ty = gt_magic(p.tiles_y);
    p.n_tiles = (int)T.tiles;
    size_t at = 0;                          // shared memory: (weights of layer one) ring (weights of layer two) T staging tail
    if (halo) {
        p.a_bytes = T.Nt * p.halo_rows * p.halo_w * p.kbytes;
        p.stage_bytes = p.planes * p.plane_bytes;
        at = (size_t)HK * p.O1p * p.kbytes;
        int stages = (kCtSmem - ct_groups(true) * (int)p.staging_bytes - (int)sizeof(CtTail<3>) - (p.dbt ? 2 : 1) * p.n_c2 * kCtChunk - (int)at - w2_slots * kCtBN2 * 128) / p.stage_bytes;
        p.stages = stages > 4 ? 4 : stages;
    } else {
        p.staging_bytes = 4 * kGtStagingBytes;
        p.a_bytes = T.Wt * T.Ht * T.Nt * 128;
        p.stage_bytes = kGtABytes + p.O1p * 128;
        int stages = (kCtSmem - fixed - (p.dbt ? 2 : 1) * p.n_c2 * kCtChunk) / p.stage_bytes;
        p.stages = stages > kGtMaxStages ? kGtMaxStages : stages;
    }
    if (p.stages < 2) return BSP_ERR_SHAPE;
    // (T of the next tile before Y of this one: with one buffer for T, layer two must be able to finish without the second
    // epilogue, that is both its accumulators must hold the whole tile)
    p.ahead = p.db && (p.dbt || p.n_t2 <= 2) ? 1 : 0;
    p.off_ring = (uint32_t)at; at += (size_t)p.stages * p.stage_bytes;
    p.off_w2 = (uint32_t)at; at += (size_t)p.w2_slots * kCtBN2 * 128;
    p.off_t = (uint32_t)at; at += (size_t)(p.dbt ? 2 : 1) * p.n_c2 * kCtChunk;
    p.off_staging = (uint32_t)at; at += (size_t)ct_groups(halo) * p.staging_bytes;
    p.off_tail = (uint32_t)at;
    const size_t smem = at + (halo ? sizeof(CtTail<3>) : sizeof(CtTail<2>));

    // kernels by type of the pair, width of Y (32 bits or the narrow form) and how layer one is staged
    typedef void (*Kernel)(const CtParams);
    static const Kernel kernels[2][2][3] = {{{chain_tc_kernel<false, 4, false, false>, chain_tc_kernel<false, 4, true, false>, chain_tc_kernel<false, 4, true, true>},
                                             {chain_tc_kernel<false, 2, false, false>, chain_tc_kernel<false, 2, true, false>, chain_tc_kernel<false, 2, true, true>}},
                                            {{chain_tc_kernel<true, 4, false, false>, chain_tc_kernel<true, 4, true, false>, chain_tc_kernel<true, 4, true, true>},
                                             {chain_tc_kernel<true, 1, false, false>, chain_tc_kernel<true, 1, true, false>, chain_tc_kernel<true, 1, true, true>}}};
    static bool opted[kGtMaxDevices] = {};
    if (!opted[dev]) {
        for (int t = 0; t < 12; ++t) BSP_CUDA_OK(cudaFuncSetAttribute(kernels[t / 6][t / 3 % 2][t % 3], cudaFuncAttributeMaxDynamicSharedMemorySize, kCtSmem));
        opted[dev] = true;
    }
    // bytes of an operand row of layer one in shared memory, and its swizzle
    const int row_bytes = halo && p.kbytes < 128 ? 32 : 128;
    const CUtensorMapSwizzle swizzle = row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_32B;
    GtEncodeFn enc = gt_encode();
    if (!enc) return BSP_ERR_CUDA;
    {
        const cuuint64_t row = (cuuint64_t)wd1.I * esz;
        const cuuint64_t gdim[4] = {row, (cuuint64_t)xd.J, (cuuint64_t)xd.L, (cuuint64_t)xd.N};
        const cuuint64_t gstr[3] = {row, row * xd.J, row * xd.J * xd.L};
        const cuuint32_t box[4] = {(cuuint32_t)row_bytes, (cuuint32_t)(halo ? p.halo_w : T.Wt * p.sw), (cuuint32_t)(halo ? p.halo_rows : T.Ht * p.sh), (cuuint32_t)T.Nt};
        const cuuint32_t estr[4] = {1, (cuuint32_t)p.sw, (cuuint32_t)p.sh, 1};
        if (enc(&p.tmx, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void *>(X), gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return BSP_ERR_CUDA;
    }
    {
        const cuuint64_t row = (cuuint64_t)wd1.I * esz;
        const cuuint64_t gdim[3] = {row, (cuuint64_t)(wd1.H * wd1.K), (cuuint64_t)wd1.O};
        const cuuint64_t gstr[2] = {row, row * wd1.H * wd1.K};
        const cuuint32_t box[3] = {(cuuint32_t)row_bytes, 1, (cuuint32_t)p.O1p};
        const cuuint32_t estr[3] = {1, 1, 1};
        if (enc(&p.tmw1, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint8_t *>((const uint8_t *)packed1 + L1.off_payload), gdim, gstr, box,
                estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return BSP_ERR_CUDA;
    }
    {
        const cuuint64_t row = (cuuint64_t)wd2.I * esz;
        const cuuint64_t gdim[3] = {row, 1, (cuuint64_t)wd2.O};
        const cuuint64_t gstr[2] = {row, row};
        const cuuint32_t box[3] = {128, 1, (cuuint32_t)kCtBN2};
        const cuuint32_t estr[3] = {1, 1, 1};
        if (enc(&p.tmw2, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint8_t *>((const uint8_t *)packed2 + L2.off_payload), gdim, gstr, box,
                estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return BSP_ERR_CUDA;
    }
    {
        const cuuint64_t row = (cuuint64_t)wd2.O * ey;
        const cuuint64_t gdim[4] = {row, (cuuint64_t)p.Nw, (cuuint64_t)p.M, (cuuint64_t)xd.N};
        const cuuint64_t gstr[3] = {row, row * p.Nw, row * p.Nw * p.M};
        const cuuint32_t box[4] = {128, (cuuint32_t)T.Wt, (cuuint32_t)T.Ht, (cuuint32_t)T.Nt};
        const cuuint32_t estr[4] = {1, 1, 1, 1};
        if (enc(&p.tmy, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, Y, gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return BSP_ERR_CUDA;
    }
    const int grid = p.n_tiles * p.parts < n_sm[dev] ? p.n_tiles * p.parts : n_sm[dev];      // (several parts: one wave)
    BSP_CUDA_OK(launch_after(kernels[wd1.wtype == BSP_I8 ? 1 : 0][ey == 4 ? 0 : 1][halo ? (eights ? 2 : 1) : 0], dim3((unsigned)grid), dim3(64u + 128u * ct_groups(halo)), smem, st, p));
    return BSP_OK;
}

}  // namespace bsp
