// Launcher of the reconstruction V^ = X P (Sec. 3.3, Notation).
#include "mxq_kernels.cuh"
#include "mxq_launch.h"

namespace mxq {
namespace {

constexpr int kU = 2;
constexpr int kThreads = 128;

template <class F, class T>
int run(const void* codes, const uint8_t* scales, size_t n, int block, void* dst, cudaStream_t stream)
{
    if constexpr (T::size == 4) {
        // FP32 output: lane units of 32 output bytes
        auto kern = dequantize_wide_kernel<F, T, kU, kThreads>;
        const size_t nunits = n / T::epl;
        int shift = 0;
        while ((T::epl << shift) < block) ++shift;        // units per scale = block / epl (block >= 16 >= epl)
        return launch_kernel(kern, grid_for_tiles((nunits + 32 * kU - 1) / (32 * kU), kThreads), kThreads, stream,
                             static_cast<const uint8_t*>(codes), scales, nunits, shift, static_cast<uint8_t*>(dst));
    } else {
        // 16-bit output: lane units of 32 codes, two per thread, but one where two leave the chip idle (see
        // grid_is_small): 2^22.1 codes from L2 to BF16, MXINT4 5.8 -> 3.2 us, E2M3 6.5 -> 3.2, and behind the conversion that wrote
        // them (both launches) MXINT4 unchanged, E2M3 7.7 ... 13 -> 6.0; 2^23 codes E2M3 5.8 -> 4.2 and 11.6 -> 8.6, but MXINT4
        // 7.2 -> 8.1: 4-bit codes and narrower keep two from half that size on.  2^24 codes: 2 - 5 % slower.
        const size_t ctas = (n / 32 + kThreads * kU - 1) / (kThreads * kU);
        const bool one = grid_is_small(F::bits > 4 ? ctas : 2 * ctas);
        auto kern = one ? dequantize_kernel<F, T, 1, kThreads> : dequantize_kernel<F, T, kU, kThreads>;
        const size_t nunits = n / 32, per_tile = one ? 32 : 32 * kU;
        const size_t ntiles = (nunits + per_tile - 1) / per_tile;
        int shift = 0, per_unit = 1;
        if (block == 16) per_unit = 2;
        else while ((32 << shift) < block) ++shift;
        return launch_kernel(kern, grid_for_tiles(ntiles, kThreads), kThreads, stream,
                             static_cast<const uint8_t*>(codes), scales, nunits, shift, per_unit,
                             static_cast<uint8_t*>(dst));
    }
}

// shift / scales-per-unit of the kernel that writes T (see run above)
template <class T>
void scale_geometry(int block, int& shift, int& per_unit)
{
    shift = 0;
    per_unit = 1;
    if constexpr (T::size == 4) {
        while ((T::epl << shift) < block) ++shift;
    } else {
        if (block == 16) per_unit = 2;
        else while ((32 << shift) < block) ++shift;
    }
}

template <class F, class T>
int run_batched(const DqDeviceItem* items_host, int count, size_t total_tiles, int block, cudaStream_t stream)
{
    int shift, per_unit;
    scale_geometry<T>(block, shift, per_unit);
    return with_item_capacity<kDqBatchItemsMax>(count, [&](auto k) {
        constexpr int K = decltype(k)::value;
        DqItemBlock<K> blk;
        fill_item_block(blk, items_host, count, total_tiles);
        auto kern = dequantize_batched_kernel<F, T, kU, kThreads, K>;
        return launch_kernel(kern, grid_for_units(total_tiles, 1), kThreads, stream, blk, shift, per_unit);
    });
}

}  // namespace

size_t dq_batched_tiles(size_t nunits) { return (nunits + kThreads * kU - 1) / (kThreads * kU); }

int launch_dequantize_batched(const DqDeviceItem* items_host, int count, size_t total_tiles, int fmt, int block, int dtype,
                              cudaStream_t stream)
{
    MXQ_DISPATCH_FORMAT(fmt, {
        if (dtype == MXQ_F32) return run_batched<F, F32>(items_host, count, total_tiles, block, stream);
        return run_batched<F, BF16>(items_host, count, total_tiles, block, stream);
    });
    return MXQ_ERR_FORMAT;
}

int launch_dequantize(const void* codes, const uint8_t* scales, size_t n, int fmt, int block, void* dst, int dtype,
                      cudaStream_t stream)
{
    MXQ_DISPATCH_FORMAT(fmt, {
        if (dtype == MXQ_F32) return run<F, F32>(codes, scales, n, block, dst, stream);
        return run<F, BF16>(codes, scales, n, block, dst, stream);
    });
    return MXQ_ERR_FORMAT;
}

}  // namespace mxq
