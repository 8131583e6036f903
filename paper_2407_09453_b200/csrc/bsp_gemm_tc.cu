// Block-sparse products Y = W*X + b on 5th-generation tensor cores, one kernel for all of them: the matrix product
// Y[p][o] = b[o] + sum over kept blocks of W-bar X (a fully connected layer, "GEMM is a 1x1 convolution") and the NHWC
// convolution with any taps, strides and zero padding, as an implicit GEMM.  tcgen05.mma with the accumulators in
// tensor memory: bf16 -> fp32 (kind::f16), int8 -> int32 (kind::i8), fp32 as TF32 -> fp32 (kind::tf32); fused bias;
// fp32, bf16, int32 or requantised int8 output.  Introduction (Y = W*X + b), Section "Block Sparsity in a Matrix" and
// Section "Compiler and its Code generation" (8-bit tensors with power-of-two scales) of the paper.
//
// The kernel reads the packed form Gamma (.) W in the layout of W, [O][H][K][I] (zeroed blocks stored as zeros), so
// that both operands arrive by tiled TMA loads under the 128-byte swizzle.  A persistent CTA owns tiles of up to 128
// output positions (a box of Wt x Ht positions of Nt images; 128 consecutive positions for a matrix product) x BN
// output channels (BN <= 256).  The reduction runs over taps x 128-byte chunks of input channels: per K-stage one
// thread issues two loads, the activation box shifted by the tap (out-of-bounds positions arrive as zeros: the
// padding; strides are the tensor map's element strides) and BN x 128 bytes of that tap's weights; one elected lane
// of the MMA warp issues four MMAs of 128 x BN x 32 bytes; two accumulator buffers of 256 columns (or four of 128) let the epilogue of
// a tile (tensor memory -> registers -> + bias -> convert -> swizzled shared memory -> global memory, by TMA stores of
// the tile's box) overlap the MMAs of the next one.  Layers that leave most SMs idle take tiles of 64 or 32 positions,
// multiplied with M = 64; layers of several waves may take boxes of parts of several images; stride-1 layers with taps
// and few input channels keep their weights in shared memory and load a tile's activations once (kHalo, kEights); large products
// run on pairs of CTAs (kPairs).  The arithmetic skips nothing: a
// tensor-core instruction covers 128 x BN x 16 entries of the operands at once, far more than a block, and feeding it
// compact blocks (cp.async expansion of the block-CSR payload in shared memory, or TMA gather loads of 128-byte
// cores) was measured two to five times slower than these dense loads.
//
// Warps: 0 producer and 1 MMA issuer (each runs its loop as a whole, converged warp with warp-uniform values; one
// elected lane issues), 2-9 epilogue in two groups of four (warp w reads the tensor-memory lanes 32 (w % 4) ..; the groups
// take turns with the tiles and share the last one).  Barriers per stage: full (one
// arrival that announces the bytes of both loads) and empty (tcgen05.commit); per accumulator buffer: acc_full (commit)
// and acc_empty (4 warps).  Every wait is bounded; on expiry BSP_ERR_TIMEOUT is latched, the roles wind down, loads
// in flight are awaited (bounded) and tensor memory is freed.
#include <type_traits>
#include "bsp_tc.cuh"

namespace bsp {
namespace {

struct GtParams {
    CUtensorMap tmx;          // X as bytes: (I * esz, J, L, N), box 128 bytes x Wt x Ht x Nt positions (in steps of the strides), 128-byte swizzle
    CUtensorMap tmw;          // Gamma (.) W as bytes: (I * esz, H K, O), box 128 bytes x 1 tap x BN channels, 128-byte swizzle
    CUtensorMap tmy;          // Y as bytes: (O * ey, N_w, M, N), box 128 bytes x Wt x Ht x Nt positions (a tile), 128-byte swizzle
    const void *bias;         // float32 or int32 [O], may be NULL
    const int32_t *shift;     // int8 output only: right shift per output channel, 0..31
    const uint8_t *packed;
    int *status;
    int O, I, P, H, K, bo, bi, wtype;
    int early_type;           // what the look at the header before the wait takes for wtype: -1 where loads may not go by it (packed_spans)
    int BN, n_tiles_n, n_tiles, n_tile_pairs, n_ks;
    int stages, stage_bytes;
    // position tiles: Wt x Ht output positions of Nt images (at most 128), tiles_x x tiles_y of them per Nt images
    int N, M, Nw, Wt, Ht, Nt, tiles_x, tiles_y, rows_tile;
    int sh, sw, ph, pw, cpt;          // strides, padding, 128-byte channel chunks per tap
    int a_bytes;                      // bytes of one activation box
    uint8_t *Y;
    int ey;
    int half_rows;                    // kTaps: tiles of at most 64 positions, multiplied with M = 64
    int narrow;                       // kTaps, bfloat16 output: tiles of 32 channels, whose rows of Y are 64 bytes
    int small_acc;                    // int8: the sums of products are at most 2^29
    // kHalo: bytes of the resident weights, pitch and rows of an image's box, position tiles, planes of 32-byte rows and their pitch
    int w_bytes, halo_w, halo_rows, n_pos, planes, plane_bytes;
    uint32_t m_ntn, m_tx, m_ty;       // floor(2^32 / d) of n_tiles_n, tiles_x, tiles_y (division by multiplication)
    int kbytes, a_stride;             // bytes of K per row of a stage: 128, or 64 for layers with at most 64 bytes of input channels; bytes of the activation part of a stage
};

// What follows the ring and the two staging buffers in shared memory.  (All of it is dynamic, so that the ring starts on
// the 1024-byte boundary that the swizzled tiles need without room for rounding: four 48 KB stages, the staging buffers
// and this fill the 227 KB of a CTA.)
constexpr int kGtHaloTaps = 30;
template <typename S>
struct GtTail {
    uint64_t full[kGtMaxStages], empty[kGtMaxStages], acc_full[4], acc_empty[4], w_full[kGtHaloTaps];
    uint32_t tmem;
    uint32_t fail, refused;
    // per epilogue group: bias, 2^(shift - 1) and shift of its round's channels
    __align__(16) uint32_t bias[2][128], half[2][128];
    __align__(16) S shift[2][128];
};
constexpr int kGtGemmSmem = 227 * 1024;
static_assert(4 * (kGtABytes + 256 * 128) + 8 * kGtStagingBytes + sizeof(GtTail<uint8_t>) <= kGtGemmSmem, "four stages at 256 channels");
constexpr int kGtTailBytes = (int)sizeof(GtTail<uint8_t>), kGtTailWords = (int)sizeof(GtTail<uint32_t>);

// First output position (image, row, column) of position tile mt.
__device__ __forceinline__ void gt_tile_origin(const GtParams &p, int mt, int &n0, int &y0, int &x0)
{
    int r, tx, ty, ni;
    gt_divmod(mt, p.tiles_x, p.m_tx, r, tx);
    gt_divmod(r, p.tiles_y, p.m_ty, ni, ty);
    x0 = tx * p.Wt; y0 = ty * p.Ht; n0 = ni * p.Nt;
}

// kWT: operand type; kEy: bytes of an output element (4: float32 or int32, 2: bfloat16, 1: int8); kMode: how operands are staged.
// kTaps loads an activation box and a weight tile per K-stage.  kPairs is the same on pairs of CTAs.  kHalo is for stride-1
// layers with taps whose input channels fit one stage and whose weights fit shared memory: the weights of the CTA's channel
// tile are loaded once and stay, the activations of a position tile arrive in ONE load with the border that its taps reach,
// and a tap is a view of that box shifted by whole rows (the swizzle goes by the shared-memory address).  Nine loads of
// shifted boxes and nine weight tiles per tile had kept such layers at the pace of the TMA unit (about 1.5 cycles per row).
// kEights is kHalo on tiles of eight columns (apart, so that kHalo's descriptors stay constants).
constexpr int kTaps = 0, kPairs = 1, kHalo = 2, kEights = 3;
template <int kWT, int kEy, int kMode>
__global__ void __launch_bounds__(kGtThreads, 1) gemm_tc_kernel(const __grid_constant__ GtParams p)
{
    constexpr bool kPair = kMode == kPairs, kFour = kMode >= kHalo && kEy == 1;
    extern __shared__ __align__(1024) uint8_t smem[];
    using Shift = std::conditional_t<kFour, uint32_t, uint8_t>;      // (words: int8 64->64 at 224 x 224, batch 32, 74.9 -> 72.0 us)
    GtTail<Shift> &tail = *(GtTail<Shift> *)(smem + (kMode >= kHalo ? p.w_bytes : 0) + (size_t)p.stages * p.stage_bytes + 8 * kGtStagingBytes);
    uint64_t *s_full = tail.full, *s_empty = tail.empty, *s_acc_full = tail.acc_full, *s_acc_empty = tail.acc_empty;
    volatile uint32_t &s_fail = tail.fail;

    // (the warp's number, the tensor-memory base and the go-ahead below come through a shuffle, which makes them uniform to
    // the compiler: the role branches and the loops under them are then warp-uniform code.  Without it every MMA cost about
    // 100 cycles of issue and every poll 150, against 48 / 64 / 127 for the MMA itself at 64 / 128 / 256 channels and 90.)
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    const int S = p.stages, n_ks = p.n_ks, BN = p.BN;
    const uint32_t ring = sm32(smem) + (kMode >= kHalo ? (uint32_t)p.w_bytes : 0u);
    const uint32_t staging = ring + (uint32_t)(S * p.stage_bytes);
    // Work items: tiles, or for CTA pairs two position tiles side by side on one channel tile (CTA r of the pair takes
    // position tile 2 mp + r; a pair past an odd count loads zeros and stores nothing).
    uint32_t rank = 0;
    if constexpr (kPair) asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(rank));
    // kHalo: a CTA keeps one channel tile and walks position tiles.
    const int ntn = p.n_tiles_n;
    // Two accumulators of 256 columns; kHalo with int8 output: four of 128 where a tile is no wider, because the requantising epilogue
    // hands one back late (64->128 at 112x112, batch 32, 30.7 -> 28.2 us; other outputs and kTaps gained nothing).
    const uint32_t acc_log = kFour && BN <= 128 ? 2u : 1u, acc_mask = (1u << acc_log) - 1u;
    const int t_first = kMode == kTaps ? (int)blockIdx.x : kPair ? (int)(blockIdx.x >> 1) : (int)blockIdx.x / ntn;
    const int t_step = kMode == kTaps ? (int)gridDim.x : kPair ? (int)(gridDim.x >> 1) : (int)gridDim.x / ntn;
    const int t_count = kMode == kTaps ? p.n_tiles : kPair ? p.n_tile_pairs : p.n_pos;
    // position tile (of this CTA, in a pair) and channel tile of a work item
    auto tile_of = [&](int tile, int &mt, int &tn) {
        if constexpr (kMode >= kHalo) { mt = tile; tn = (int)blockIdx.x - t_first * ntn; }
        else {
            gt_divmod(tile, ntn, p.m_ntn, mt, tn);
            if constexpr (kPair) mt = 2 * mt + (int)rank;
        }
    };
    // barriers of the pair's leader (CTA 0), as shared::cluster addresses
    uint32_t lead_full0 = sm32(&s_full[0]), lead_acc_empty0 = sm32(&s_acc_empty[0]);
    if constexpr (kPair) {
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;\n" : "=r"(lead_full0) : "r"(sm32(&s_full[0])));
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;\n" : "=r"(lead_acc_empty0) : "r"(sm32(&s_acc_empty[0])));
    }

    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&s_full[s])), "r"(1) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&s_empty[s])), "r"(1) : "memory");
        }
        for (int b = 0; b < (kFour ? 4 : 2); ++b) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&s_acc_full[b])), "r"(1) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&s_acc_empty[b])), "r"(kPair ? 8 : 4) : "memory");
        }
        if constexpr (kMode >= kHalo)
            for (int t = 0; t < p.n_ks; ++t) asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm32(&tail.w_full[t])), "r"(1) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(&p.tmx) : "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(&p.tmw) : "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(&p.tmy) : "memory");
    }
    if (warp == 0) {
        if constexpr (kPair) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(sm32(&tail.tmem)), "r"(kGtTmemCols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(sm32(&tail.tmem)), "r"(kGtTmemCols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
        }
    }
    auto header_ok = [&](int type) { return gt_header_ok(p.packed, type, p.O, p.I, p.H, p.K, p.bo, p.bi); };
    // (the CTAs of a pair must come to the same decision, and large products have no use for it)
    const bool early = !kPair && tid == 0 && header_ok(p.early_type);
    wait_for_previous<false>();
    if (warp == 0) let_next_start();                  // (behind its allocation)
    if (tid == 0) {
        const bool ok = early || header_ok(p.wtype);
        const bool placed = (ring & 1023u) == 0u;
        s_fail = ok && placed ? 0u : 2u;
        if (!ok) atomicMax(p.status, (int)BSP_ERR_INDEX);
        else if (!placed) atomicMax(p.status, (int)BSP_ERR_CUDA);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    gt_sync_all<kPair>();                   // (a pair: both CTAs' barriers are initialised before either signals the other)
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, tail.tmem, 0);
    const bool run = __shfl_sync(0xFFFFFFFFu, s_fail, 0) == 0u;

    if (warp == 0) {
        // ================= producer =================
        // The whole warp runs the loop with warp-uniform values; one elected lane arms the barrier and issues the loads.
        if (run) {
            const uint32_t full0 = sm32(&s_full[0]), empty0 = sm32(&s_empty[0]);
            // (a pair: each CTA loads its own activation box and its half of the weight tile, all four loads announce their
            // bytes on the leader's barrier, which the leader arms with the total)
            const uint32_t stage_bytes = (uint32_t)p.stage_bytes;
            const uint32_t tx = (uint32_t)(p.a_bytes + (kMode >= kHalo ? 0 : BN >> (kPair ? 1 : 0)) * p.kbytes) * (kPair ? 2u : 1u);
            const int cpt128 = p.cpt * 128, Kw = p.K;
            // (a fresh barrier counts as released: the wait on parity 1 of the first round returns at once)
            uint32_t slot = 0, epar = 1, issued = 0, dst = ring;
            bool ok = true, free_now = true;
            for (int tile = t_first; tile < t_count && ok; tile += t_step) {
                int mt, tn;
                tile_of(tile, mt, tn);
                const int ch0 = tn * BN + (kPair ? (int)rank * (BN >> 1) : 0);
                int n0, y0, x0;
                gt_tile_origin(p, mt, n0, y0, x0);
                if constexpr (kMode >= kHalo) {
                    if (s_fail) { ok = false; break; }
                    if (!free_now && !__all_sync(0xFFFFFFFFu, gt_poll(empty0 + slot * 8u, epar))) { ok = false; break; }
                    const bool wrap = slot + 1u == (uint32_t)S;
                    const uint32_t next_free = gt_test(empty0 + (wrap ? 0u : slot + 1u) * 8u, wrap ? epar ^ 1u : epar);
                    // (the second plane's load is predicated off where one plane holds all channels, or rows are 128 bytes)
                    asm volatile("{\n .reg .pred e, e1;\n elect.sync _|e, 0xFFFFFFFF;\n setp.ne.b32 e1, %8, 0;\n and.pred e1, e1, e;\n"
                                 " @e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n"
                                 " @e cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%2], [%3, {%4, %5, %6, %7}], [%0];\n"
                                 " @e1 cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%9], [%3, {%10, %5, %6, %7}], [%0];\n}\n"
                                 ::"r"(full0 + slot * 8u), "r"(tx), "r"(dst), "l"(&p.tmx), "r"(0), "r"(x0 - p.pw), "r"(y0 - p.ph), "r"(n0),
                                   "r"(p.planes - 1), "r"(dst + (uint32_t)p.plane_bytes), "r"(32) : "memory");
                    ++issued;
                    free_now = __all_sync(0xFFFFFFFFu, next_free != 0u);
                    if (wrap) { slot = 0; epar ^= 1u; dst = ring; } else { ++slot; dst += stage_bytes; }
                    if (tile == t_first)
                        for (int t = 0; t < n_ks; ++t)
                            asm volatile("{\n .reg .pred e, e1;\n elect.sync _|e, 0xFFFFFFFF;\n setp.ne.b32 e1, %7, 0;\n and.pred e1, e1, e;\n"
                                         " @e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n"
                                         " @e cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%2], [%3, {%4, %5, %6}], [%0];\n"
                                         " @e1 cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%8], [%3, {%9, %5, %6}], [%0];\n}\n"
                                         ::"r"(sm32(&tail.w_full[t])), "r"((uint32_t)(BN * p.kbytes)), "r"(sm32(smem) + (uint32_t)(t * BN * p.kbytes)), "l"(&p.tmw), "r"(0), "r"(t), "r"(ch0),
                                           "r"(p.planes - 1), "r"(sm32(smem) + (uint32_t)(t * BN * p.kbytes + BN * 32)), "r"(32) : "memory");
                } else {
                // input position of the tile's first output position at tap (0, 0); a tap is a shift of the box, positions
                // outside the image read as zeros (the padding)
                const int xi0 = x0 * p.sw - p.pw;
                int c128 = 0, kx = xi0, hy = y0 * p.sh - p.ph, tap = 0, kk = 0;
                if (s_fail) { ok = false; break; }
                for (int ks = 0; ks < n_ks; ++ks) {
                    if (!free_now && !__all_sync(0xFFFFFFFFu, gt_poll(empty0 + slot * 8u, epar))) { ok = false; break; }
                    const bool wrap = slot + 1u == (uint32_t)S;
                    const uint32_t bar_next = empty0 + (wrap ? 0u : slot + 1u) * 8u, par_next = wrap ? epar ^ 1u : epar;
                    uint32_t next_free;
                    if constexpr (kPair) {
                        asm volatile("{\n .reg .pred e, l, f, v;\n elect.sync _|e, 0xFFFFFFFF;\n setp.eq.u32 l, %13, 0;\n and.pred l, l, e;\n"
                                     " @l mbarrier.arrive.expect_tx.shared::cta.b64 _, [%1], %2;\n"
                                     " @e cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%3], [%4, {%5, %6, %7, %8}], [%14];\n"
                                     " mbarrier.test_wait.parity.shared::cta.b64 f, [%15], %16;\n"
                                     " @e cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%9], [%10, {%5, %11, %12}], [%14];\n"
                                     " vote.sync.all.pred v, f, 0xFFFFFFFF;\n selp.b32 %0, 1, 0, v;\n}\n"
                                     : "=r"(next_free) : "r"(full0 + slot * 8u), "r"(tx), "r"(dst), "l"(&p.tmx), "r"(c128), "r"(kx), "r"(hy), "r"(n0),
                                       "r"(dst + (uint32_t)p.a_stride), "l"(&p.tmw), "r"(tap), "r"(ch0), "r"(rank), "r"(lead_full0 + slot * 8u), "r"(bar_next), "r"(par_next) : "memory");
                    } else {
                        asm volatile("{\n .reg .pred e, f, v;\n elect.sync _|e, 0xFFFFFFFF;\n"
                                     " @e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%1], %2;\n"
                                     " @e cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%3], [%4, {%5, %6, %7, %8}], [%1];\n"
                                     " mbarrier.test_wait.parity.shared::cta.b64 f, [%13], %14;\n"
                                     " @e cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%9], [%10, {%5, %11, %12}], [%1];\n"
                                     " vote.sync.all.pred v, f, 0xFFFFFFFF;\n selp.b32 %0, 1, 0, v;\n}\n"
                                     : "=r"(next_free) : "r"(full0 + slot * 8u), "r"(tx), "r"(dst), "l"(&p.tmx), "r"(c128), "r"(kx), "r"(hy), "r"(n0),
                                       "r"(dst + (uint32_t)p.a_stride), "l"(&p.tmw), "r"(tap), "r"(ch0), "r"(bar_next), "r"(par_next) : "memory");
                    }
                    ++issued;
                    free_now = next_free != 0u;
                    if (wrap) { slot = 0; epar ^= 1u; dst = ring; } else { ++slot; dst += stage_bytes; }
                    // next K-stage: the next 128-byte chunk of channels, then the next tap (columns first)
                    c128 += 128;
                    if (c128 == cpt128) {
                        c128 = 0; ++tap; ++kx;
                        if (++kk == Kw) { kk = 0; kx = xi0; ++hy; }
                    }
                }
                }
            }
            if (!ok && lane == 0) {
                // winding down after a wait that ran out: the loads already issued still write into this CTA's shared
                // memory, so the barriers of the stages in flight are awaited (bounded) before the CTA may leave
                atomicExch((uint32_t *)&tail.fail, 1u);
                // (the follower of a pair has no barrier of its own to watch: its loads announce themselves to the leader;
                // both CTAs meet at the cluster barrier before they leave)
                if (kMode >= kHalo && issued > 0)
                    for (int t = 0; t < n_ks; ++t) gt_poll(sm32(&tail.w_full[t]), 0u);
                for (uint32_t back = 0; back < (uint32_t)S && back < issued && rank == 0; ++back) {
                    const uint32_t it = issued - 1u - back;
                    gt_poll(full0 + (it % (uint32_t)S) * 8u, (it / (uint32_t)S) & 1u);
                }
            }
        }
    } else if (kMode >= kHalo && warp == 1) {
        // ================= MMA issuer of kHalo =================
        if (run) {
            const uint32_t dfmt = kWT == BSP_I8 ? 2u : 1u, abfmt = kWT == BSP_F32 ? 2u : 1u;
            const uint32_t idesc = (dfmt << 4) | (abfmt << 7) | (abfmt << 10) | ((uint32_t)(BN >> 3) << 17) | ((128u >> 4) << 24);
            const uint32_t full0 = sm32(&s_full[0]), empty0 = sm32(&s_empty[0]);
            const uint32_t stage16 = (uint32_t)p.stage_bytes >> 4;
            // One tile's MMAs.  kWide: rows of 128 bytes, else planes of 32-byte rows; kFirst: the CTA's first tile, whose taps
            // wait for their weights.  (Apart, so that the loop over the taps has no branch but its own: one on kWide inside
            // it cost 10 %.)
            auto issue = [&](auto wide_c, auto first_c, uint32_t d, uint32_t a_tap) -> bool {
                constexpr bool kWide = decltype(wide_c)::value, kFirst = decltype(first_c)::value;
                constexpr uint64_t shape = kWide ? kGtDesc : kGtDesc32;
                const uint32_t row16 = kWide ? 8u : 2u, w_tap16 = (uint32_t)(BN * p.kbytes) >> 4, row_step = (uint32_t)(p.halo_w - p.K) * row16;
                const uint64_t plane_a = (uint64_t)(p.plane_bytes >> 4), plane_b = (uint64_t)(BN * 32 >> 4);
                const uint32_t two = (uint32_t)p.planes - 1u;
                uint64_t da = (kMode == kEights ? gt_desc_groups(shape, (uint32_t)p.halo_w * row16) : shape) | (uint64_t)a_tap, db = shape | (uint64_t)(sm32(smem) >> 4);
                uint32_t acc = 0u;
                int t = 0;
#pragma unroll 1
                for (int h = 0; h < p.H; ++h, da += row_step)
#pragma unroll 1
                    for (int k = 0; k < p.K; ++k, ++t, da += row16, db += w_tap16) {
                        if constexpr (kFirst) {
                            if (!__all_sync(0xFFFFFFFFu, gt_poll(sm32(&tail.w_full[t]), 0u))) return false;
                            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                        }
                        if constexpr (kWide) gt_issue_tap<kWT>(d, da, db, idesc, acc);
                        else gt_issue_planes<kWT>(d, da, db, plane_a, plane_b, two, idesc, acc);
                        acc = 1u;
                    }
                return true;
            };
            auto run_tiles = [&](auto wide_c) -> bool {
                uint32_t slot = 0, par = 0, tile_i = 0;
                for (int tile = t_first; tile < t_count; tile += t_step, ++tile_i) {
                    const uint32_t buf = tile_i & acc_mask, use = tile_i >> acc_log, d = tmem + (buf << (9 - acc_log));
                    bool ok = gt_poll(sm32(&s_acc_empty[buf]), (use & 1u) ^ 1u) && gt_poll(full0 + slot * 8u, par) && s_fail == 0u;
                    if (!__all_sync(0xFFFFFFFFu, ok)) return false;
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    const uint32_t a_tap = (ring >> 4) + slot * stage16;
                    if (tile_i == 0) ok = issue(wide_c, std::true_type(), d, a_tap);
                    else issue(wide_c, std::false_type(), d, a_tap);
                    if (!ok) return false;
                    gt_commit_elected<false>(empty0 + slot * 8u);
                    gt_commit_elected<false>(sm32(&s_acc_full[buf]));
                    if (++slot == (uint32_t)S) { slot = 0; par ^= 1u; }
                }
                return true;
            };
            const bool ok = p.kbytes == 128 ? run_tiles(std::true_type()) : run_tiles(std::false_type());
            if (!ok && lane == 0) atomicExch((uint32_t *)&tail.fail, 1u);
        }
    } else if (warp == 1) {
        // ================= MMA issuer =================
        // The whole warp runs the loop (so that its address arithmetic stays warp-uniform); one elected lane issues.
        if (run && rank == 0) {               // (of a pair, the leader issues for both CTAs)
            // instruction descriptor: D fp32 (int32 for int8), A and B bf16 / signed int8 / tf32, K-major both, M = 128
            // (256 over a pair, 64 for low tiles), N = BN
            const uint32_t dfmt = kWT == BSP_I8 ? 2u : 1u, abfmt = kWT == BSP_F32 ? 2u : 1u;
            const uint32_t idesc = (dfmt << 4) | (abfmt << 7) | (abfmt << 10) | ((uint32_t)(BN >> 3) << 17) |
                                   (((kPair ? 256u : kMode == kTaps && p.half_rows ? 64u : 128u) >> 4) << 24);
            const uint32_t full0 = sm32(&s_full[0]), empty0 = sm32(&s_empty[0]);
            const uint32_t stage16 = (uint32_t)p.stage_bytes >> 4, astride16 = (uint32_t)p.a_stride >> 4;
            const uint64_t desc0 = p.kbytes == 64 ? kGtDesc64 : kGtDesc;
            const uint32_t nk = (uint32_t)p.kbytes >> 5;            // MMAs per stage: 32 bytes of K each
            uint32_t slot = 0, par = 0, a16 = ring >> 4, tile_i = 0;
            bool ok = true, full_now = false;
            for (int tile = t_first; tile < t_count && ok; tile += t_step, ++tile_i) {
                const uint32_t buf = tile_i & 1u, use = tile_i >> 1;
                if (!gt_poll(sm32(&s_acc_empty[buf]), (use & 1u) ^ 1u) || s_fail != 0u) ok = false;   // (a fresh barrier counts as released)
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint32_t d = tmem + buf * 256u;
                for (int ks = 0; ks < n_ks; ++ks) {
                    if (!full_now && !gt_poll_stage(full0 + slot * 8u, par)) { ok = false; break; }
                    const bool wrap = slot + 1u == (uint32_t)S;
                    const uint64_t da = desc0 | (uint64_t)(a16 & 0x3FFFu), db = desc0 | (uint64_t)((a16 + astride16) & 0x3FFFu);
                    full_now = gt_issue_stage<kWT, kPair>(d, da, db, idesc, empty0 + slot * 8u, ks != 0 ? 1u : 0u, nk,
                                                          full0 + (wrap ? 0u : slot + 1u) * 8u, wrap ? par ^ 1u : par) != 0u;
                    if (wrap) { slot = 0; par ^= 1u; a16 = ring >> 4; } else { ++slot; a16 += stage16; }
                }
                if (ok) gt_commit_elected<kPair>(sm32(&s_acc_full[buf]));
            }
            if (!ok && lane == 0) atomicExch((uint32_t *)&tail.fail, 1u);
        }
    } else {
        // ================= epilogue (warps 2-9) =================
        // Two groups of four warps: group g drains every second tile of the CTA, so the
        // epilogues of two consecutive tiles run side by side.  The last tile of a CTA (often its only one) is shared, each
        // group taking every second of its 128-byte rounds: 1x1 256->1024 at 14x14, batch 64, 14.1 -> 12.9 us; sharing every
        // tile instead cost 10 % where a CTA has many small ones (8-bit 3x3 64->64 at 224x224, int32 output).
        if (run) {
            const int q = warp & 3;                              // quarter of the tensor-memory lanes this warp reaches
            const int grp = (warp - 2) >> 2;
            constexpr int cpr = 128 / kEy;                       // output channels per round (128 bytes of a row)
            const bool narrow = kMode == kTaps && kEy == 2 && p.narrow != 0;
            // the group's staging buffer: 128 rows of 128 bytes
            const uint32_t sg = staging + (uint32_t)(grp * 4 * kGtStagingBytes);
            const bool issuer = q == 0 && lane == 0;             // one thread of the group issues its stores
            // this lane's row of the staging buffer: the lane's row of the tile, or in kHalo the place of its output in the box
            int row = q * 32 + lane;
            if constexpr (kMode == kTaps)                        // (with M = 64, 16 rows in the first half of each quarter)
                if (p.half_rows) row = lane < 16 ? q * 16 + lane : -1;
            if constexpr (kMode >= kHalo) row = gt_halo_row(row, kMode == kEights, p.Wt, p.Ht, p.Nt, p.halo_w, p.halo_rows);
            // Constants of a round's channels: the group's thread c holds channel c of the next round and puts them into shared
            // memory once the group has read the current ones, so that the trip to memory is never waited for.
            uint32_t *bias = tail.bias[grp], *half = tail.half[grp];
            Shift *shift = tail.shift[grp];
            const int ct = ((warp - 2) & 3) * 32 + lane;
            bool mine = true;                                    // (the look that decides, by one thread, on its way while the tile is made)
            if (!kPair && tid == 64) mine = header_ok(p.wtype);
            const uint32_t *bias_of = from_here((const uint32_t *)p.bias);       // raw bits: float32 or int32
            const int32_t *shift_of = from_here(p.shift);
            uint32_t next_bias = 0u, next_shift = 1u;
            int have = -1;                                       // first channel of the round whose constants are in shared memory
            bool small = false, mine_small = false, fresh = false;
            auto fetch = [&](int ch0) {
                if (ct >= cpr) return;
                next_bias = bias_of != nullptr && ch0 + ct < p.O ? load_free(bias_of + ch0 + ct) : 0u;
                if constexpr (kEy == 1) next_shift = ch0 + ct < p.O ? (uint32_t)load_free(shift_of + ch0 + ct) & 31u : 1u;
            };
            auto place = [&](int ch0) {                          // (between two barriers of the group)
                have = ch0;
                fresh = true;
                if constexpr (kEy == 1)
                    mine_small = p.small_acc != 0 && next_shift != 0u && next_shift != 31u && (int)next_bias <= (1 << 29) && (int)next_bias >= -(1 << 29);
                if (ct >= cpr) return;
                bias[ct] = next_bias;
                if constexpr (kEy == 1) { half[ct] = (1u << next_shift) >> 1; shift[ct] = (Shift)next_shift; }
            };
            uint32_t tile_i = 0;
            bool ok = true, store = true;
            if constexpr (!kPair) {
                if (tid == 64) {
                    tail.refused = mine ? 0u : 1u;
                    if (!mine) atomicMax(p.status, (int)BSP_ERR_INDEX);
                }
                asm volatile("bar.sync 3, 256;\n" ::: "memory");
                store = tail.refused == 0u;
            }
            for (int tile = t_first; tile < t_count; tile += t_step, ++tile_i) {
                const bool last = tile + t_step >= t_count, shared_tile = last && BN > cpr;
                if (!shared_tile && (int)(tile_i & 1u) != grp) continue;
                const int c_first = shared_tile ? grp * cpr : 0, c_step = shared_tile ? 2 * cpr : cpr;
                const uint32_t buf = tile_i & acc_mask, use = tile_i >> acc_log;
                int mt, tn;
                tile_of(tile, mt, tn);
                const int n0 = tn * BN;
                int in0, y0, x0;
                gt_tile_origin(p, mt, in0, y0, x0);
                // (here every thread of the group is past the barrier of its last round: its constants may be replaced)
                const bool replace = have != n0 + c_first;       // the first tile, or an order of rounds that was not foreseen
                if (replace) { fetch(n0 + c_first); place(n0 + c_first); }
                // A wait that ran out is latched below; the group goes on (its warps meet at barriers) and waits no more.
                if (s_fail) ok = false;
                if (ok && !gt_wait(sm32(&s_acc_full[buf]), use & 1u)) ok = false;
                // int8: the staging buffer was handed to a TMA store; the issuing thread waits until it has been read
                if (kEy == 1 && issuer) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
                if (kEy == 1 ? !fresh : replace) gt_group_sync(1 + grp);
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (buf << (9 - acc_log));
                // the channels of the round after the last one of this tile: those of the group's next tile
                int after = n0 + c_first;
                if (!last && kMode < kHalo && ntn > 1) {
                    int m2, t2;
                    const int next = tile + 2 * t_step < t_count ? tile + 2 * t_step : tile + t_step;
                    gt_divmod(next, ntn, p.m_ntn, m2, t2);
                    after = t2 * BN + (next + t_step >= t_count && BN > cpr ? grp * cpr : 0);
                }
                // the accumulator buffer has been read: hand it back to the MMA issuer (before the round is staged, where that can be)
                auto hand_back = [&]() {
                    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        if constexpr (kPair)
                            asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];\n" ::"r"(lead_acc_empty0 + buf * 8u) : "memory");
                        else
                            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(sm32(&s_acc_empty[buf])) : "memory");
                    }
                };
                for (int c0 = c_first; c0 < BN; c0 += c_step) {
                    const bool hand = !last && c0 + c_step >= BN;
                    const int left = (p.O - n0 < BN ? p.O - n0 : BN) - c0;          // channels from here on
                    const int next_ch = c0 + c_step < BN ? n0 + c0 + c_step : after;
                    if (next_ch != have) fetch(next_ch);
                    const uint32_t tcol = tbase + (uint32_t)c0, srow = sg + (uint32_t)row * (narrow ? 64u : 128u), sw = narrow ? ((uint32_t)row >> 1) & 3u : (uint32_t)row & 7u;
                    if constexpr (kEy == 1) {
                        if (c0 != c_first) {
                            if (issuer) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
                            if (!fresh) gt_group_sync(1 + grp);
                        }
                        if (fresh) small = gt_group_all(1 + grp, mine_small);
                        fresh = false;
                        gt_epilogue_int8<false>(tcol, bias, half, shift, small, left, 0, srow, sw, row >= 0);
                        if (hand) hand_back();
                    } else {
                        // (loads and arithmetic run while the last store reads the staging buffer)
                        uint32_t out[32];
                        gt_epilogue_round<kWT == BSP_I8, kEy, false>(tcol, bias, left, 0, out);
                        if (hand) hand_back();
                        if (issuer) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
                        gt_group_sync(1 + grp);
                        if (next_ch != have) place(next_ch);
                        gt_store_round(srow, sw, row >= 0, out, narrow ? 4u : 8u);
                    }
                    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                    gt_group_sync(1 + grp);
                    if (kEy == 1 && next_ch != have) place(next_ch);
                    // one store of the tile's box: 128 bytes of every row; what lies past the last channel, column, row or image
                    // of Y is clipped (rows of the buffer beyond the box are not part of the store)
                    if (issuer && left > 0 && store) {
                        asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];\n"
                                     ::"l"(&p.tmy), "r"(sg), "r"((n0 + c0) * kEy), "r"(x0), "r"(y0), "r"(in0) : "memory");
                        asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
                    }
                }
            }
            if (issuer) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");      // (the stores have read this CTA's memory)
            if (!ok && lane == 0) atomicExch((uint32_t *)&tail.fail, 1u);
        }
    }

    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    gt_sync_all<kPair>();                   // (a pair: neither CTA leaves while the other may still signal its barriers)
    if (s_fail == 1u && tid == 0) atomicMax(p.status, (int)BSP_ERR_TIMEOUT);
    if (warp == 0) {
        if constexpr (kPair) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kGtTmemCols) : "memory");
        else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kGtTmemCols) : "memory");
    }
}

}  // namespace


// True if the kernel can run this layer: rows of X, W and Y that are multiples of 16 bytes (tensor-map strides), a
// position count that fits 32 bits, and a position tile whose box the tensor map can express.
bool gemm_tc_eligible(const bsp_wdesc &wd, const bsp_xdesc &xd0, bsp_dtype ytype)
{
    const bsp_xdesc xd = gt_flatten(wd, xd0);
    if (!packed_layout(wd).enabled) return false;
    if (ytype != BSP_F32 && ytype != BSP_BF16 && ytype != BSP_I32 && ytype != BSP_I8) return false;
    const int ey = ytype == BSP_BF16 ? 2 : (ytype == BSP_I8 ? 1 : 4);
    if (((long long)wd.O * ey) % 16 != 0) return false;
    const int M = (xd.L + 2 * xd.pad_h - wd.H) / xd.stride_h + 1, Nw = (xd.J + 2 * xd.pad_w - wd.K) / xd.stride_w + 1;
    if (M <= 0 || Nw <= 0) return false;
    if ((long long)xd.N * M * Nw > 0x7FFFFFFF || (long long)xd.N * xd.L * xd.J > 0x7FFFFFFF) return false;
    if ((long long)xd.N * M * Nw * wd.O * ey >= (1LL << 46)) return false;
    return xd.stride_h <= 256 && xd.stride_w <= 256;       // (a box of one position then fits: gt_pick_tile)
}

bsp_status launch_gemm_tc(const bsp_wdesc &wd, const bsp_xdesc &xd0, const void *packed, const void *X,
                          const void *bias, const int32_t *shift, void *Y, bsp_dtype ytype, void *ws, cudaStream_t st)
{
    const bsp_xdesc xd = gt_flatten(wd, xd0);
    const PackedLayout L = packed_layout(wd);
    if (!L.enabled) return BSP_ERR_SHAPE;
    const int esz = elem_bytes(wd.wtype);
    const int ey = ytype == BSP_BF16 ? 2 : (ytype == BSP_I8 ? 1 : 4);
    const int HK = wd.H * wd.K;
    if (ytype == BSP_I8 && shift == nullptr) return BSP_ERR_NULL;
    GtParams p = {};
    p.bias = bias; p.shift = shift; p.packed = (const uint8_t *)packed;
    p.status = (int *)ws;
    p.O = wd.O; p.I = wd.I; p.H = wd.H; p.K = wd.K; p.bo = wd.bo; p.bi = wd.bi;
    p.wtype = wd.wtype; p.ey = ey; p.Y = (uint8_t *)Y;
    p.small_acc = (long long)wd.I * HK * 128 * 128 <= (1 << 29) ? 1 : 0;
    p.N = xd.N; p.sh = xd.stride_h; p.sw = xd.stride_w; p.ph = xd.pad_h; p.pw = xd.pad_w;
    p.M = (xd.L + 2 * xd.pad_h - wd.H) / xd.stride_h + 1;
    p.Nw = (xd.J + 2 * xd.pad_w - wd.K) / xd.stride_w + 1;
    const long long P = (long long)xd.N * p.M * p.Nw;
    p.P = (int)P;
    GtTile T = gt_pick_tile(xd.N, p.M, p.Nw, p.sh, p.sw);
    if (T.tiles <= 0) return BSP_ERR_SHAPE;
    static int n_sm[kGtMaxDevices] = {};
    int dev = 0;
    BSP_CUDA_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kGtMaxDevices) return BSP_ERR_CUDA;
    if (n_sm[dev] == 0) BSP_CUDA_OK(cudaDeviceGetAttribute(&n_sm[dev], cudaDevAttrMultiProcessorCount, dev));
    if (T.tiles * ((wd.O + 255) / 256) > n_sm[dev]) T = gt_pick_packed(T, xd.N, p.M, p.Nw, p.sh, p.sw);
    // layers with at most 64 bytes of input channels per position stage 64-byte rows (64-byte swizzle, two MMAs a stage)
    p.kbytes = (long long)wd.I * esz <= 64 ? 64 : 128;
    p.cpt = (int)(((long long)wd.I * esz + 127) / 128);
    p.n_ks = HK * p.cpt;
    // kernels by operand type (in the order of bsp_dtype), width of the output (32 bits or the narrow form) and mode
    typedef void (*Kernel)(const GtParams);
    static const Kernel kernels[3][2][4] = {
        {{gemm_tc_kernel<BSP_F32, 4, kTaps>, gemm_tc_kernel<BSP_F32, 4, kPairs>, gemm_tc_kernel<BSP_F32, 4, kHalo>, gemm_tc_kernel<BSP_F32, 4, kEights>},
         {gemm_tc_kernel<BSP_F32, 2, kTaps>, gemm_tc_kernel<BSP_F32, 2, kPairs>, gemm_tc_kernel<BSP_F32, 2, kHalo>, gemm_tc_kernel<BSP_F32, 2, kEights>}},
        {{gemm_tc_kernel<BSP_BF16, 4, kTaps>, gemm_tc_kernel<BSP_BF16, 4, kPairs>, gemm_tc_kernel<BSP_BF16, 4, kHalo>, gemm_tc_kernel<BSP_BF16, 4, kEights>},
         {gemm_tc_kernel<BSP_BF16, 2, kTaps>, gemm_tc_kernel<BSP_BF16, 2, kPairs>, gemm_tc_kernel<BSP_BF16, 2, kHalo>, gemm_tc_kernel<BSP_BF16, 2, kEights>}},
        {{gemm_tc_kernel<BSP_I8, 4, kTaps>, gemm_tc_kernel<BSP_I8, 4, kPairs>, gemm_tc_kernel<BSP_I8, 4, kHalo>, gemm_tc_kernel<BSP_I8, 4, kEights>},
         {gemm_tc_kernel<BSP_I8, 1, kTaps>, gemm_tc_kernel<BSP_I8, 1, kPairs>, gemm_tc_kernel<BSP_I8, 1, kHalo>, gemm_tc_kernel<BSP_I8, 1, kEights>}}};
    static_assert(BSP_F32 == 0 && BSP_BF16 == 1 && BSP_I8 == 2, "the table is indexed by type");
    const Kernel *kernel = kernels[wd.wtype][ey == 4 ? 0 : 1];
    static bool opted[kGtMaxDevices] = {};
    if (!opted[dev]) {
        for (int t = 0; t < 24; ++t)
            BSP_CUDA_OK(cudaFuncSetAttribute(kernels[t / 8][t / 4 % 2][t % 4], cudaFuncAttributeMaxDynamicSharedMemorySize, kGtGemmSmem));
        opted[dev] = true;
    }
    // Channels per tile: the widest tile keeps the tensor pipe busiest (a stage costs about 256 + 2 BN cycles of operand
    // fetch from shared memory), but a layer with few position tiles fills more SMs with narrower ones: the width with
    // the lowest waves x stage cost wins.  kHalo competes where it applies, with cycles per tile for both: a K-stage costs
    // its MMAs (32 + BN / 4 cycles of operand reads or BN / 2 of arithmetic per 32 bytes of K) or, loaded per tap, 1.5
    // cycles per row of its two boxes; kHalo pays only the MMAs, on tiles that the border makes a few more.
    const int staging = 8 * kGtStagingBytes, nk = p.kbytes / 32;
    const GtHaloTile Th = gt_pick_halo(xd.N, p.M, p.Nw, wd.H, wd.K);
    const bool halo_ok = HK > 1 && HK <= kGtHaloTaps && p.cpt == 1 && p.sh == 1 && p.sw == 1 && Th.tiles > 0;
    // (up to 64 bytes of channels lie in planes of 32-byte rows: MMAs on 64-byte rows took 90 cycles instead of 67 at 128
    // channels and 72 instead of 59 at 64)
    const int halo_kb = (long long)wd.I * esz <= 32 ? 32 : p.kbytes, planes = halo_kb == 128 ? 1 : halo_kb / 32;
    const int plane_bytes = halo_ok ? (Th.Nt * (Th.Ht + wd.H - 1) * (Th.Wt + wd.K - 1) * (halo_kb / planes) + 1023) / 1024 * 1024 : 0;
    const int halo_bytes = planes * plane_bytes, halo_tail = ytype == BSP_I8 ? kGtTailWords : kGtTailBytes;
    int mode = kTaps, halo_bn = 0;
    double taps_cycles = -1.0, halo_cycles = -1.0;
    {
        const int step = 64;
        const int widest = (gemm_tile_n(wd.O) + step - 1) / step * step;
        long long best_cost = -1;
        for (int bn = widest; bn >= step; bn -= step) {
            if (bn != widest && bn != 128 && bn != 64) continue;
            // (a round of the int8 output stores 128 channels: a tile that is not a multiple of that must be the only one)
            if (ytype == BSP_I8 && bn % 128 != 0 && bn < wd.O) continue;
            const long long ntn = (wd.O + bn - 1) / bn, tiles = T.tiles * ntn;
            const long long waves = (tiles + n_sm[dev] - 1) / n_sm[dev], cost = waves * (256 + 2 * bn);
            const double mma = nk * (bn >= 128 ? (32 + bn / 4 > bn / 2 ? 32 + bn / 4 : bn / 2) : 32 + bn / 4);
            if (best_cost < 0 || cost < best_cost) {
                best_cost = cost; p.BN = bn;
                const double loads = 1.5 * (T.Wt * T.Ht * T.Nt + bn);
                taps_cycles = waves * (p.n_ks * (mma > loads ? mma : loads) + 400.0);
            }
            if (halo_ok && ntn <= n_sm[dev] && HK * bn * halo_kb + 2 * halo_bytes + staging + halo_tail <= kGtGemmSmem) {
                const long long hw = (Th.tiles + n_sm[dev] / ntn - 1) / (n_sm[dev] / ntn);
                const double c = hw * (HK * mma * halo_kb / p.kbytes + 400.0);
                if (halo_cycles < 0 || c < halo_cycles) { halo_cycles = c; halo_bn = bn; }
            }
        }
    }
    // A layer that leaves most SMs idle takes lower position tiles, for as long as its tiles stay on SMs of their own: what it
    // waits for is the pace of one SM, 1.5 cycles a row of its two boxes and, in tiles of up to 64 positions, MMAs with M = 64
    // that read half as much of the activations.  (Measured: 3x3 176->64 at 27x27 9.2 -> 6.3 us, of which M = 64 is 1.0;
    // 3x3 128->128 at 28x28 5.8 -> 5.4; a product of 64 positions, K = 2048, 7.4 -> 6.9.  Sharing the K-stages of a tile over a
    // cluster of CTAs instead took 9.9 us for that one: a kernel on all SMs cannot start before the one ahead of it ends.)
    for (int rows = kGtBM / 2; rows >= 32; rows /= 2) {
        const GtTile low = gt_pick_tile(xd.N, p.M, p.Nw, p.sh, p.sw, rows);
        const long long ntn = (wd.O + p.BN - 1) / p.BN;
        if (low.tiles <= 0 || low.tiles * ntn > n_sm[dev]) break;
        const double mma = nk * (16 + p.BN / 4 > p.BN / 2 ? 16 + p.BN / 4 : p.BN / 2), loads = 1.5 * (low.Wt * low.Ht * low.Nt + p.BN);
        const double cycles = p.n_ks * (mma > loads ? mma : loads) + 400.0;
        if (cycles >= taps_cycles) break;
        T = low;
        taps_cycles = cycles;
    }
    // ... and tiles of 32 channels, where these still have SMs of their own: half of the weights to load per CTA, and MMAs of 24 cycles
    // instead of 32.  (A product of 64 positions, 2048->1000, 6.58 -> 6.25 us; fp32, 100 positions, 9.17 -> 8.97.)
    if (ytype != BSP_I8 && p.BN == 64 && T.Wt * T.Ht * T.Nt <= 64 && T.tiles * ((wd.O + 31) / 32) <= n_sm[dev]) p.BN = 32;
    if (halo_cycles >= 0 && halo_cycles < taps_cycles) { mode = kHalo; p.BN = halo_bn; T = Th; }
    p.half_rows = mode == kTaps && T.Wt * T.Ht * T.Nt <= 64 ? 1 : 0;
    p.narrow = mode == kTaps && p.BN == 32 && ey == 2 ? 1 : 0;
    p.Wt = T.Wt; p.Ht = T.Ht; p.Nt = T.Nt; p.rows_tile = T.Wt * T.Ht * T.Nt;
    p.tiles_x = (p.Nw + T.Wt - 1) / T.Wt; p.tiles_y = (p.M + T.Ht - 1) / T.Ht;
    p.n_tiles_n = (wd.O + p.BN - 1) / p.BN;
    if (T.tiles * p.n_tiles_n > 0x7FFFFFFF - 4096) return BSP_ERR_SHAPE;      // (tile counters step by up to twice the grid)
    p.n_tiles = (int)(T.tiles * p.n_tiles_n);
    p.n_pos = (int)T.tiles;
    // Large products run on CTA pairs: two position tiles side by side on one 256-channel tile, every CTA loading its
    // own activations and half of the weights (the operand fetch per SM and MMA falls from 12 KB to 8 KB).
    // (Tiles of a few K-stages are bound by their epilogue, and there the pair's cross-CTA hand-shakes only cost.)
    if (mode == kTaps && p.kbytes == 128 && p.BN == 256 && p.n_ks >= 8 && (long long)p.n_tiles >= 4LL * n_sm[dev] && n_sm[dev] >= 2) mode = kPairs;
    const bool pair = mode == kPairs;
    p.n_tile_pairs = (int)(((T.tiles + 1) / 2) * p.n_tiles_n);
    p.m_ntn = gt_magic(p.n_tiles_n); p.m_tx = gt_magic(p.tiles_x); p.m_ty = gt_magic(p.tiles_y);
    p.a_stride = kGtBM * p.kbytes;
    p.a_bytes = p.rows_tile * p.kbytes;
    p.stage_bytes = p.a_stride + (pair ? p.BN / 2 : p.BN) * p.kbytes;
    if (mode == kHalo) {
        p.kbytes = halo_kb; p.planes = planes; p.plane_bytes = plane_bytes;
        p.halo_w = T.Wt + wd.K - 1; p.halo_rows = T.Ht + wd.H - 1;
        p.w_bytes = HK * p.BN * p.kbytes;
        p.a_bytes = T.Nt * p.halo_rows * p.halo_w * p.kbytes;
        p.stage_bytes = halo_bytes;
    }
    const int tail_bytes = mode == kHalo ? halo_tail : kGtTailBytes;
    int stages = (kGtGemmSmem - staging - tail_bytes - p.w_bytes) / p.stage_bytes;
    if (stages > kGtMaxStages) stages = kGtMaxStages;
    if (stages < 2) return BSP_ERR_SHAPE;
    p.stages = stages;
    const size_t smem = (size_t)p.w_bytes + (size_t)stages * p.stage_bytes + staging + (size_t)tail_bytes;

    // bytes of an operand row in shared memory, and its swizzle
    const int row_bytes = mode == kHalo && p.kbytes < 128 ? 32 : p.kbytes;
    const CUtensorMapSwizzle swizzle = row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : (row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
    GtEncodeFn enc = gt_encode();
    if (!enc) return BSP_ERR_CUDA;
    {
        const cuuint64_t row = (cuuint64_t)wd.I * esz;
        const cuuint64_t gdim[4] = {row, (cuuint64_t)xd.J, (cuuint64_t)xd.L, (cuuint64_t)xd.N};
        const cuuint64_t gstr[3] = {row, row * xd.J, row * xd.J * xd.L};
        // a box spans Wt * s_w x Ht * s_h input positions in steps of the strides: Wt x Ht positions arrive
        const cuuint32_t box[4] = {(cuuint32_t)row_bytes, (cuuint32_t)(mode == kHalo ? p.halo_w : T.Wt * p.sw),
                                   (cuuint32_t)(mode == kHalo ? p.halo_rows : T.Ht * p.sh), (cuuint32_t)T.Nt};
        const cuuint32_t estr[4] = {1, (cuuint32_t)p.sw, (cuuint32_t)p.sh, 1};
        if (enc(&p.tmx, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void *>(X), gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return BSP_ERR_CUDA;
    }
    {
        const cuuint64_t row = (cuuint64_t)wd.I * esz;
        const cuuint64_t gdim[3] = {row, (cuuint64_t)HK, (cuuint64_t)wd.O};
        const cuuint64_t gstr[2] = {row, row * HK};
        const cuuint32_t box[3] = {(cuuint32_t)row_bytes, 1, (cuuint32_t)(pair ? p.BN / 2 : p.BN)};
        const cuuint32_t estr[3] = {1, 1, 1};
        if (enc(&p.tmw, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint8_t *>((const uint8_t *)packed + L.off_payload), gdim, gstr, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return BSP_ERR_CUDA;
    }
    {
        const cuuint64_t row = (cuuint64_t)wd.O * ey;
        const cuuint64_t gdim[4] = {row, (cuuint64_t)p.Nw, (cuuint64_t)p.M, (cuuint64_t)xd.N};
        const cuuint64_t gstr[3] = {row, row * p.Nw, row * p.Nw * p.M};
        const cuuint32_t box[4] = {p.narrow ? 64u : 128u, (cuuint32_t)T.Wt, (cuuint32_t)T.Ht, (cuuint32_t)T.Nt};
        const cuuint32_t estr[4] = {1, 1, 1, 1};
        if (enc(&p.tmy, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, Y, gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                p.narrow ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return BSP_ERR_CUDA;
    }

    p.early_type = !pair && packed_spans(wd, packed) ? (int)wd.wtype : -1;
    if (pair) {
        const int pairs = p.n_tile_pairs < n_sm[dev] / 2 ? p.n_tile_pairs : n_sm[dev] / 2;
        BSP_CUDA_OK(launch_after_clusters(kernel[kPairs], dim3((unsigned)(2 * pairs)), dim3(kGtThreads), smem, st, 2, 1, p));
        return BSP_OK;
    }
    int grid = p.n_tiles < n_sm[dev] ? p.n_tiles : n_sm[dev];
    if (mode == kHalo) grid = grid / p.n_tiles_n * p.n_tiles_n;
    BSP_CUDA_OK(launch_after(kernel[mode == kHalo && Th.eights ? kEights : mode], dim3((unsigned)grid), dim3(kGtThreads), smem, st, p));
    return BSP_OK;
}

}  // namespace bsp
