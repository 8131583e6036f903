// Internal declarations shared by the CUDA translation units of libbsp.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include "bsp.h"

namespace bsp {

constexpr uint32_t kPackedMagic = 0x42535032u;   // "BSP2"

// First 256 bytes of the packed buffer, written on the device by bsp_compact and checked by the product kernel
// before it stores anything (and before it loads from a buffer that may end before the descriptor's weights do: gt_header_ok).
struct PackedHeader {
    uint32_t magic;
    int32_t dtype, O, I, H, K, bo, bi;
    int32_t forms;           // kForm* bits of what the buffer holds
    int64_t off_payload;     // byte offset of the packed weights
};
static_assert(sizeof(PackedHeader) <= 256, "the packed header is the first 256 bytes");

// The packed form: Gamma (.) W in the layout of W, [O][H][K][I], weights of zeroed blocks written as zeros, so that
// tiles of it arrive by tiled TMA loads.  A K-stage of the product kernel is 128 bytes of the input channels of one
// tap (64 bf16, 128 int8, 32 fp32).
constexpr int kFormDense = 4;

struct PackedLayout {
    bool enabled;            // rows of input channels are multiples of 16 bytes and O a multiple of 8
    size_t off_payload, total_bytes;
};

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }
inline int elem_bytes(bsp_dtype t) { return t == BSP_I8 ? 1 : (t == BSP_BF16 ? 2 : 4); }

PackedLayout packed_layout(const bsp_wdesc &wd);

// Whether the allocation that `packed` lies in reaches as far as a packed buffer of this descriptor: loads by it then stay in mapped memory,
// whatever the buffer holds.  (False where the driver cannot say; 0.1 us.)
bool packed_spans(const bsp_wdesc &wd, const void *packed);

// Workspace: the first 256 bytes hold the latched status word (word 0) and the counts of CTAs that have arrived and that are done
// of the single-launch kernels (words kWsSyncWord, kWsSyncWord + 1), zero between launches; scratch starts after them.
constexpr size_t kWsHeader = 256;
constexpr int kWsSyncWord = 2;
// Scratch of the cooperative select after the scores in the mask workspace: three histograms of 2048 words, 8 counter words,
// one word per CTA, and in what is left a list of candidate keys with the numbers of their blocks.
constexpr int kSelectMaxCtas = 1024;
constexpr int kSelectHist = 3 * 2048;
constexpr size_t kSelectScratch = 98336;
constexpr int kSelectList = (int)((kSelectScratch - (kSelectHist + 8 + kSelectMaxCtas) * 4) / 12 / 512 * 512);

// Host-side validation of a weight descriptor, shared by every entry point.
bsp_status check_wdesc(const bsp_wdesc *wd);

bsp_status launch_mask(const bsp_wdesc &wd, const void *W, bsp_norm norm, bsp_scope scope, int64_t n_zero,
                       uint8_t *gamma, void *scores, bool keep_scores, void *ws, cudaStream_t st);
bsp_status launch_compact(const bsp_wdesc &wd, const void *W, const uint8_t *gamma, int32_t *row_ptr,
                          int32_t *col_idx, void *payload, void *packed, int64_t capacity_blocks, void *ws,
                          cudaStream_t st);
bsp_status launch_count(const uint8_t *gamma, int64_t n, unsigned long long *out, cudaStream_t st);

// A failed CUDA call becomes BSP_ERR_CUDA; with BSP_DEBUG set in the environment its text goes to stderr.
void report_cuda_error(cudaError_t e, const char *expr, const char *file, int line);

bool gemm_tc_eligible(const bsp_wdesc &wd, const bsp_xdesc &xd, bsp_dtype ytype);
bool chain_tc_eligible(const bsp_wdesc &wd1, const bsp_wdesc &wd2, const bsp_xdesc &xd, bsp_dtype ytype);
bsp_status launch_chain_tc(const bsp_wdesc &wd1, const void *packed1, const bsp_wdesc &wd2, const void *packed2,
                           const bsp_xdesc &xd, const void *X, const void *bias1, const int32_t *shift1, int relu,
                           const void *bias2, const int32_t *shift2, void *Y, bsp_dtype ytype, void *ws, cudaStream_t st);
bsp_status launch_gemm_tc(const bsp_wdesc &wd, const bsp_xdesc &xd, const void *packed, const void *X,
                          const void *bias, const int32_t *shift, void *Y, bsp_dtype ytype, void *ws, cudaStream_t st);
// Output channels per CTA tile of the product kernel (a multiple of 64, at most 256).
inline int gemm_tile_n(int O)
{
    const int tiles = (O + 255) / 256;
    return (((O + tiles - 1) / tiles) + 63) / 64 * 64;
}

// Programmatic dependent launch: a kernel launched by launch_after() may start while the kernel before it on the stream
// still runs, once every CTA of that one has called let_next_start() or left.  Until wait_for_previous() returns - the
// kernel before it has then completed and its writes are visible - it takes nothing from global memory (it sets up
// barriers, tensor memory and descriptors; the tensor-core kernels look at a header, see gt_header_ok).  It lets its own successor start only after that, so at most two kernels of a
// stream overlap, and no successor can hold a line in L1 that was read before the kernel in between wrote it.  (Launched
// one after another without this, the kernels of a stream started in steps of about 2 us.)
// What an earlier kernel may have written is read by plain loads or __ldcg, through pointers without __restrict__: __ldg and
// const __restrict__ promise data that nobody writes while the kernel runs, and it runs before wait_for_previous() returns.
// In a kernel that owns tensor memory the warp that allocates it signals, behind the allocation, and no other: the first thread
// of a CTA to signal speaks for the whole CTA, and while the allocating warp still waits for columns, a CTA of the successor on
// the same SM could take them and hold them until this kernel ends, and neither would move.  (Behind the CTA barrier instead
// the signal came 0.1 us later, and with it the next kernel.)
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
// kLetNext = false: the next kernel starts when this one has ended (still without the gap between launches), or calls
// let_next_start() later.
template <bool kLetNext = true>
__device__ __forceinline__ void wait_for_previous()
{
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    if constexpr (kLetNext) let_next_start();
}

// Loads that the compiler may move and hoist like those of read-only data, but coherent, and not above the from_here() that
// their address came through: for what an earlier kernel wrote and nobody writes after the wait.  (Plain loads stay between
// the stores, atomics and volatile statements around them: bfloat16 728 x 1408 x 1472 at 75 % 10.6 us with __ldg, 12.4 plain.)
template <typename T>
__device__ __forceinline__ const T *from_here(const T *p)
{
    asm volatile("" : "+l"(p));
    return p;
}
__device__ __forceinline__ uint32_t load_free(const uint32_t *p) { uint32_t v; asm("ld.global.b32 %0, [%1];\n" : "=r"(v) : "l"(p)); return v; }
__device__ __forceinline__ int32_t load_free(const int32_t *p) { return (int32_t)load_free((const uint32_t *)p); }
__device__ __forceinline__ uint32_t load_free(const uint8_t *p) { uint32_t v; asm("ld.global.u8 %0, [%1];\n" : "=r"(v) : "l"(p)); return v; }
__device__ __forceinline__ uint2 load_free(const uint2 *p)
{
    uint2 v;
    asm("ld.global.v2.b32 {%0, %1}, [%2];\n" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ uint4 load_free(const uint4 *p)
{
    uint4 v;
    asm("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
template <int kBytes = 0>                                 // (kBytes past p: part of the instruction)
__device__ __forceinline__ float4 load_free(const float4 *p)
{
    float4 v;
    asm("ld.global.v4.f32 {%0, %1, %2, %3}, [%4 + %5];\n" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p), "n"(kBytes));
    return v;
}

template <typename... P, typename... A>
cudaError_t launch_after_clusters(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, int cluster_x, int cluster_z, A... args)
{
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster_x; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = (unsigned)cluster_z;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cfg.attrs = attr; cfg.numAttrs = cluster_x * cluster_z > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args)
{
    return launch_after_clusters(kernel, grid, block, smem, st, 1, 1, args...);
}

#define BSP_CUDA_OK(expr)                                            \
    do {                                                             \
        cudaError_t e_ = (expr);                                     \
        if (e_ != cudaSuccess) {                                     \
            bsp::report_cuda_error(e_, #expr, __FILE__, __LINE__);   \
            return BSP_ERR_CUDA;                                     \
        }                                                            \
    } while (0)

}  // namespace bsp
