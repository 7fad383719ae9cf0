// Launchers of Slice-and-Scale (Eq. 4-5): one tensor per launch, and the batched form that
// converts a whole set of tensors in one launch.
#include "mxq_kernels.cuh"
#include "mxq_launch.h"

namespace mxq {
namespace {

constexpr int kU = 2;
constexpr int kThreads = 128;

// One function template per operation: inside a template the branch that an illegal (source, target)
// pair would take is discarded, so kernels are instantiated for the legal pairs only.
template <class FH, class FL>
int run_single(const void* codes, const uint8_t* scales, size_t n, int block, void* out_codes, uint8_t* out_scales,
               cudaStream_t stream)
{
    if constexpr (ss_pair_ok(FH::id, FL::id)) {
        const size_t nunits = n / 32, nscales = n / (size_t)block;
        size_t ntiles = (nunits + 32 * kU - 1) / (32 * kU);
        auto kern = slice_scale_kernel<FH, FL, kU, kThreads>;
        if (block == 16) kern = slice_scale_kernel<FH, FL, kU, kThreads, uint8_t*, true>;
        // E4M3 to more than four bits with one unit per thread where two leave the chip idle: E2M3 of 2^23 codes 4.6 -> 4.0 us,
        // block 16 5.2 -> 4.1, of 2^22.1 codes 3.25 -> 2.9 and 5.7 -> 3.1; 2^24 codes 5.8 -> 6.2.  E2M1 and the MXINT conversions do
        // not gain (2^23 codes 3.0 -> 3.6, MXINT8 -> MXINT4 2.9 -> 3.4).
        if constexpr (FH::id == MXQ_FP8_E4M3 && FL::bits > 4) {
            if (grid_is_small((ntiles + kThreads / 32 - 1) / (kThreads / 32))) {
                kern = block == 16 ? slice_scale_kernel<FH, FL, 1, kThreads, uint8_t*, true> : slice_scale_kernel<FH, FL, 1, kThreads>;
                ntiles = (nunits + 31) / 32;
            }
        }
        // MXINT8 in about one wave: the kernel with fewer resident CTAs (measured at slice_scale_is_small); to 3 bits, up to four CTAs per
        // SM, one unit per thread (2^14 codes 1.6 -> 1.4 us, 2^20 1.8 -> 1.6, 2^22 2.9 -> 2.55; 2^22.25 3.0 -> 3.05).
        if constexpr (slice_scale_has_small<FH, FL>()) {
            const size_t ctas = (ntiles + kThreads / 32 - 1) / (kThreads / 32);
            if (slice_scale_is_small<FL>(ctas))
                kern = block == 16 ? slice_scale_kernel<FH, FL, kU, kThreads, uint8_t*, true, true>
                                   : slice_scale_kernel<FH, FL, kU, kThreads, uint8_t*, false, true>;
            if constexpr (FL::bits == 3) {
                if (ctas <= (size_t)148 * 4) {
                    kern = block == 16 ? slice_scale_kernel<FH, FL, 1, kThreads, uint8_t*, true> : slice_scale_kernel<FH, FL, 1, kThreads>;
                    ntiles = (nunits + 31) / 32;
                }
            }
        }
        return launch_kernel(kern, grid_for_tiles(ntiles, kThreads), kThreads, stream, static_cast<const uint8_t*>(codes),
                             scales, nunits, nscales, static_cast<uint8_t*>(out_codes), out_scales);
    } else {
        return MXQ_ERR_PAIR;
    }
}

template <class FH, class FL>
int run_single_tiled(const void* codes, const uint8_t* scales, size_t n, void* out_codes, const TiledScales& out_tiled,
                     cudaStream_t stream)
{
    if constexpr (ss_pair_ok(FH::id, FL::id) && FL::kind == KIND_FP) {
        auto kern = slice_scale_kernel<FH, FL, kU, kThreads, TiledScales>;
        const size_t nunits = n / 32;
        const size_t ctas = (nunits + kThreads * kU - 1) / (kThreads * kU) + tiled_pad_ctas(out_tiled, kThreads);
        return launch_kernel(kern, grid_for_units(ctas, 1), kThreads, stream, static_cast<const uint8_t*>(codes),
                             scales, nunits, nunits, static_cast<uint8_t*>(out_codes), out_tiled);
    } else {
        return MXQ_ERR_PAIR;
    }
}

template <class FH, class FL>
int run_table(const SsDeviceItem* items_dev, const TileIndex* index_dev, int count, size_t total_tiles,
              cudaStream_t stream)
{
    if constexpr (ss_pair_ok(FH::id, FL::id)) {
        auto kern = slice_scale_batched_kernel<FH, FL, kU, kThreads>;
        return launch_kernel(kern, grid_for_units(total_tiles, 1), kThreads, stream, items_dev, index_dev);
    } else {
        return MXQ_ERR_PAIR;
    }
}

template <class FH, class FL>
int run_params(const SsDeviceItem* items_host, int count, size_t total_tiles, cudaStream_t stream)
{
    if constexpr (ss_pair_ok(FH::id, FL::id)) {
        return with_item_capacity<kSsParamItemsMax>(count, [&](auto k) {
            constexpr int K = decltype(k)::value;
            SsItemBlock<K> blk;
            fill_item_block(blk, items_host, count, total_tiles);
            auto kern = slice_scale_batched_param_kernel<FH, FL, kU, kThreads, K>;
            if constexpr (slice_scale_has_small<FH, FL>() && FL::bits != 4 && K == kSmallBatchItems) {
                if (slice_scale_is_small<FL>(total_tiles)) kern = slice_scale_batched_param_kernel<FH, FL, kU, kThreads, K, true>;
            }
            return launch_kernel(kern, grid_for_units(total_tiles, 1), kThreads, stream, blk);
        });
    } else {
        return MXQ_ERR_PAIR;
    }
}

template <class FH, class FL>
int run_tiled_params(const SsTiledDeviceItem* items_host, int count, size_t total_tiles, cudaStream_t stream)
{
    if constexpr (ss_pair_ok(FH::id, FL::id) && FL::kind == KIND_FP) {
        return with_item_capacity<kSsTiledItemsMax>(count, [&](auto k) {
            constexpr int K = decltype(k)::value;
            SsTiledItemBlock<K> blk;
            fill_item_block(blk, items_host, count, total_tiles);
            auto kern = slice_scale_tiled_batched_kernel<FH, FL, kU, kThreads, K>;
            return launch_kernel(kern, grid_for_units(total_tiles, 1), kThreads, stream, blk);
        });
    } else {
        return MXQ_ERR_PAIR;
    }
}

}  // namespace

size_t ss_tiled_batched_tiles(const SsTiledDeviceItem& item)
{
    return ss_batched_tiles(item.nunits) + tiled_pad_ctas(item.out_scales, kThreads);
}

size_t ss_batched_tiles(size_t nunits) { return (nunits + kThreads * kU - 1) / (kThreads * kU); }

int launch_slice_scale(const void* codes, const uint8_t* scales, size_t n, int block, int src_fmt, int dst_fmt,
                       void* out_codes, uint8_t* out_scales, cudaStream_t stream)
{
    MXQ_DISPATCH_FORMAT_AS(src_fmt, FH, {
        MXQ_DISPATCH_FORMAT_AS(dst_fmt, FL, { return run_single<FH, FL>(codes, scales, n, block, out_codes, out_scales, stream); });
    });
    return MXQ_ERR_FORMAT;
}

int launch_slice_scale_tiled(const void* codes, const uint8_t* scales, size_t n, int src_fmt, int dst_fmt,
                             void* out_codes, uint8_t* out_tiled, uint32_t kblocks, cudaStream_t stream)
{
    const TiledScales sink = make_tiled_scales(out_tiled, kblocks, (uint32_t)(n / 32 / kblocks));
    MXQ_DISPATCH_FORMAT_AS(src_fmt, FH, {
        MXQ_DISPATCH_FORMAT_AS(dst_fmt, FL, { return run_single_tiled<FH, FL>(codes, scales, n, out_codes, sink, stream); });
    });
    return MXQ_ERR_FORMAT;
}

int launch_slice_scale_tiled_batched(const SsTiledDeviceItem* items_host, int count, size_t total_tiles, int src_fmt,
                                     int dst_fmt, cudaStream_t stream)
{
    MXQ_DISPATCH_FORMAT_AS(src_fmt, FH, {
        MXQ_DISPATCH_FORMAT_AS(dst_fmt, FL, { return run_tiled_params<FH, FL>(items_host, count, total_tiles, stream); });
    });
    return MXQ_ERR_FORMAT;
}

int launch_slice_scale_batched(const SsDeviceItem* items_dev, const TileIndex* index_dev, int count, size_t total_tiles,
                               int src_fmt, int dst_fmt, cudaStream_t stream)
{
    MXQ_DISPATCH_FORMAT_AS(src_fmt, FH, {
        MXQ_DISPATCH_FORMAT_AS(dst_fmt, FL, { return run_table<FH, FL>(items_dev, index_dev, count, total_tiles, stream); });
    });
    return MXQ_ERR_FORMAT;
}

int launch_slice_scale_batched_params(const SsDeviceItem* items_host, int count, size_t total_tiles, int src_fmt,
                                      int dst_fmt, cudaStream_t stream)
{
    MXQ_DISPATCH_FORMAT_AS(src_fmt, FH, {
        MXQ_DISPATCH_FORMAT_AS(dst_fmt, FL, { return run_params<FH, FL>(items_host, count, total_tiles, stream); });
    });
    return MXQ_ERR_FORMAT;
}

}  // namespace mxq
