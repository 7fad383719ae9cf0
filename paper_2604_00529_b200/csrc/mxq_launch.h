// Internal interface between the C ABI (argument checks, mxq_api.cu) and the per-operation
// translation units that instantiate and launch the kernels.  Arguments are already validated.
#pragma once
#include <cstddef>
#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

#include "../../include/mxq.h"
#include "mxq_debug.cuh"

namespace mxq {

// Grid size that gives every warp tile a warp of its own (`threads` per CTA); 0 when the tensor
// would need more CTAs than a grid can hold (beyond 2^40 elements: reported as MXQ_ERR_SIZE).
inline int grid_for_tiles(size_t ntiles, int threads)
{
    const size_t warps = (size_t)threads / 32;
    const size_t need = (ntiles + warps - 1) / warps;
    if (need > (size_t)0x7FFFFFFF) return 0;
    return (int)(need ? need : 1);
}

// The same for kernels whose CTA covers `per_cta` consecutive lane units.
inline int grid_for_units(size_t nunits, size_t per_cta)
{
    const size_t need = (nunits + per_cta - 1) / per_cta;
    return need > (size_t)0x7FFFFFFF ? 0 : (int)need;
}

// Are `ctas` CTAs of 128 threads too few to keep the chip busy (under eight per SM of its 148)?  A launch is then
// bound by how long one thread takes, and the shape with half the work per thread is faster.
inline bool grid_is_small(size_t ctas) { return ctas < (size_t)148 * 8; }

int launch_quantize(const void* src, int dtype, size_t n, int fmt, int block, void* codes, uint8_t* scales,
                    cudaStream_t stream);
int launch_fake_quant(const void* src, int dtype, size_t n, int fmt, int block, int mode, void* dst,
                      cudaStream_t stream);
int launch_slice_scale(const void* codes, const uint8_t* scales, size_t n, int block, int src_fmt, int dst_fmt,
                       void* out_codes, uint8_t* out_scales, cudaStream_t stream);
// One 8-bit anchor -> 2 ... kSetTargetsMax DIFFERENT lower formats in one pass (one kernel per set of formats).
struct SsOut;
constexpr int kSetTargetsMax = 4;
bool slice_scale_set_anchor(int src_fmt);                   // the sources that have these kernels
int launch_slice_scale_set(const uint8_t* codes, const uint8_t* scales, size_t n, int block, int src_fmt, int ntargets,
                           const int* fmts, const SsOut* outs, cudaStream_t stream);
int launch_slice_scale_set_e4m3(const uint8_t* codes, const uint8_t* scales, size_t n, int block, int ntargets,
                                const int* fmts, const SsOut* outs, cudaStream_t stream);
// Two different lower formats of up to kSsPairItemsMax anchors in one launch (items: a HOST array with tile_begin
// filled in, tiles counted by ss_pair_batched_tiles).
struct SsPairDeviceItem;
constexpr int kSsPairItemsMax = 256;
int launch_slice_scale_pair_batched(const SsPairDeviceItem* items_host, int count, size_t total_tiles, int src_fmt, int fmt1,
                                    int fmt2, cudaStream_t stream);
int launch_slice_scale_pair_batched_e4m3(const SsPairDeviceItem* items_host, int count, size_t total_tiles, int fmt1,
                                         int fmt2, cudaStream_t stream);
size_t ss_pair_batched_tiles(size_t nunits);
// The same two operations with the scale bytes written in 128 x 4 tiles (block 32, kblocks block-columns
// per row; bytes of a tile that the matrix does not cover are written as 0).
int launch_quantize_tiled(const void* src, int dtype, size_t n, int fmt, void* codes, uint8_t* tiled,
                          uint32_t kblocks, cudaStream_t stream);
int launch_slice_scale_tiled(const void* codes, const uint8_t* scales, size_t n, int src_fmt, int dst_fmt,
                             void* out_codes, uint8_t* out_tiled, uint32_t kblocks, cudaStream_t stream);
int launch_dequantize(const void* codes, const uint8_t* scales, size_t n, int fmt, int block, void* dst, int dtype,
                      cudaStream_t stream);
// Fused fake-quant over up to kFqBatchItemsMax tensors in one launch; `items_host` is a HOST array
// whose tile_begin fields are filled in.
struct FqDeviceItem;
constexpr int kFqBatchItemsMax = 512;
int launch_fake_quant_batched(const FqDeviceItem* items_host, int count, size_t total_tiles, int dtype, int fmt,
                              int block, int mode, cudaStream_t stream);
size_t fq_batched_tiles(size_t nunits);
int launch_copy(const void* src, size_t nbytes, void* dst, cudaStream_t stream);
// Q_f and the reconstruction over up to 512 tensors in one launch; `items_host` is a HOST array whose
// tile_begin fields are filled in (tiles counted by q_batched_tiles / dq_batched_tiles of each tensor's
// lane units: n / elements-per-32-bytes of the source for Q_f and for FP32 outputs, n / 32 for BF16 outputs).
struct QDeviceItem;
struct DqDeviceItem;
constexpr int kQBatchItemsMax = 512;
constexpr int kDqBatchItemsMax = 512;
int launch_quantize_batched(const QDeviceItem* items_host, int count, size_t total_tiles, int dtype, int fmt, int block,
                            cudaStream_t stream);
int launch_dequantize_batched(const DqDeviceItem* items_host, int count, size_t total_tiles, int fmt, int block, int dtype,
                              cudaStream_t stream);
size_t q_batched_tiles(size_t nunits);
size_t dq_batched_tiles(size_t nunits);

// Batched Slice-and-Scale over a device-resident item table and its coarse tile index (see
// mxq_kernels.cuh: SsDeviceItem, TileIndex); used by the fixed-table entry point.
struct SsDeviceItem;
struct TileIndex;
int launch_slice_scale_batched(const SsDeviceItem* items_dev, const TileIndex* index_dev, int count, size_t total_tiles,
                               int src_fmt, int dst_fmt, cudaStream_t stream);
// The same launch with the items (a HOST array here) passed in the kernel's parameter space; count
// must not exceed kSsParamItemsMax.
constexpr int kSsParamItemsMax = 512;
int launch_slice_scale_batched_params(const SsDeviceItem* items_host, int count, size_t total_tiles, int src_fmt,
                                      int dst_fmt, cudaStream_t stream);
// The batched launch with tiled scale outputs: up to kSsTiledItemsMax items (a HOST array, tile_begin
// filled in) in the kernel's parameter space.
struct SsTiledDeviceItem;
constexpr int kSsTiledItemsMax = 256;
int launch_slice_scale_tiled_batched(const SsTiledDeviceItem* items_host, int count, size_t total_tiles, int src_fmt,
                                     int dst_fmt, cudaStream_t stream);
// tiles one tensor of `nunits` lane units occupies in the batched kernel's tile space
size_t ss_batched_tiles(size_t nunits);
size_t ss_tiled_batched_tiles(const SsTiledDeviceItem& item);      // the same with the padding of its scale tiles

// Item tables ride in the kernel parameters, and a launch pays for their size (host time per launch next to a
// B200: 2.3 us with 64 bytes of parameters, 2.4 with 4 KB, 3.6 with 16 KB, 5.0 - 5.5 with 32 KB).  So every batched
// kernel exists with a small table, for the sets of a few layers, and with the largest one.
constexpr int kSmallBatchItems = 64;
template <int KMAX, class FN>
inline int with_item_capacity(int count, FN&& fn)
{
    if (count > KMAX) return MXQ_ERR_SIZE;
    if (count <= kSmallBatchItems) return fn(std::integral_constant<int, kSmallBatchItems>{});
    return fn(std::integral_constant<int, KMAX>{});
}

// The table block of a batched kernel: `count` items (a HOST array with tile_begin filled in) and the tile index.
template <class BLK, class ITEM>
inline void fill_item_block(BLK& blk, const ITEM* items, int count, size_t total_tiles)
{
    constexpr int K = (int)(sizeof(blk.items) / sizeof(blk.items[0]));
    for (int i = 0; i < count; ++i) blk.items[i] = items[i];
    for (int i = count; i < K; ++i) blk.items[i] = ITEM{};
    build_tile_index(blk.index, items, count, total_tiles);
}

// Expands the body once per element format with NAME bound to mxq::Fmt<id>.
#define MXQ_DISPATCH_FORMAT_AS(fmt, NAME, ...)                                      \
    switch (fmt) {                                                                  \
    case MXQ_INT8: { using NAME = ::mxq::Fmt<MXQ_INT8>; __VA_ARGS__; } break;           \
    case MXQ_INT7: { using NAME = ::mxq::Fmt<MXQ_INT7>; __VA_ARGS__; } break;           \
    case MXQ_INT6: { using NAME = ::mxq::Fmt<MXQ_INT6>; __VA_ARGS__; } break;           \
    case MXQ_INT5: { using NAME = ::mxq::Fmt<MXQ_INT5>; __VA_ARGS__; } break;           \
    case MXQ_INT4: { using NAME = ::mxq::Fmt<MXQ_INT4>; __VA_ARGS__; } break;           \
    case MXQ_INT3: { using NAME = ::mxq::Fmt<MXQ_INT3>; __VA_ARGS__; } break;           \
    case MXQ_INT2: { using NAME = ::mxq::Fmt<MXQ_INT2>; __VA_ARGS__; } break;           \
    case MXQ_FP8_E4M3: { using NAME = ::mxq::Fmt<MXQ_FP8_E4M3>; __VA_ARGS__; } break;   \
    case MXQ_FP7_E3M3: { using NAME = ::mxq::Fmt<MXQ_FP7_E3M3>; __VA_ARGS__; } break;   \
    case MXQ_FP6_E3M2: { using NAME = ::mxq::Fmt<MXQ_FP6_E3M2>; __VA_ARGS__; } break;   \
    case MXQ_FP6_E2M3: { using NAME = ::mxq::Fmt<MXQ_FP6_E2M3>; __VA_ARGS__; } break;   \
    case MXQ_FP5_E2M2: { using NAME = ::mxq::Fmt<MXQ_FP5_E2M2>; __VA_ARGS__; } break;   \
    case MXQ_FP4_E2M1: { using NAME = ::mxq::Fmt<MXQ_FP4_E2M1>; __VA_ARGS__; } break;   \
    default: return MXQ_ERR_FORMAT;                                                 \
    }
#define MXQ_DISPATCH_FORMAT(fmt, ...) MXQ_DISPATCH_FORMAT_AS(fmt, F, __VA_ARGS__)

// Launches `kern` on `stream` with programmatic stream serialization allowed (see pdl_release /
// pdl_acquire in mxq_access.cuh).  Returns MXQ_OK or MXQ_ERR_CUDA.
template <class... KArgs, class... Args>
inline int launch_kernel(void (*kern)(KArgs...), int grid, int threads, cudaStream_t stream, const Args&... args)
{
    if (grid <= 0) return MXQ_ERR_SIZE;
#ifdef MXQ_DEBUG
    if (debug_upload(stream) != 0) {                      // the byte ranges this launch may touch
        (void)cudaGetLastError();
        return MXQ_ERR_CUDA;
    }
#endif
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // (the arguments go by address: an item table is copied once, into the launch itself)
    auto launch = [&](const KArgs&... a) {
        void* p[] = {const_cast<void*>(static_cast<const void*>(&a))...};
        return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(kern), p);
    };
    if (launch(args...) != cudaSuccess) {
        (void)cudaGetLastError();
        return MXQ_ERR_CUDA;
    }
    return MXQ_OK;
}

}  // namespace mxq
