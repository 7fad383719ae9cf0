// Launcher of the batched fused fake-quant (Eq. 6 over a whole set of tensors in one launch).
#include "mxq_kernels.cuh"
#include "mxq_launch.h"

namespace mxq {
namespace {

constexpr int kU = 1;
// Consecutive warp tiles of one tensor per warp: 1 / 2 / 4 take 547 / 498 / 542 us (BF16, MXINT4 through the anchor) and
// 539 / 499 / 543 us (BF16, E2M3) over four decoder layers.  FP32 takes 990 ... 1042 us with 1, changing from run to run
// within a process, and 1008 ... 1015 with 2; alone in a process 1006 ... 1012 and 1008 ... 1010: no difference to keep two forms for.
constexpr int kR = 2;
constexpr int kThreads = 128;

template <class T, class F, int BLOCK, int MODE>
int run(const FqDeviceItem* items_host, int count, size_t total_tiles, cudaStream_t stream)
{
    if constexpr (BLOCK < T::epl) {
        return MXQ_ERR_BLOCK;
    } else {
        return with_item_capacity<kFqBatchItemsMax>(count, [&](auto k) {
            constexpr int K = decltype(k)::value;
            FqItemBlock<K> blk;
            fill_item_block(blk, items_host, count, total_tiles);
            auto kern = fake_quant_batched_kernel<T, F, BLOCK, MODE, kU, kR, kThreads, K>;
            return launch_kernel(kern, grid_for_units(total_tiles, 1), kThreads, stream, blk);
        });
    }
}

template <class T, class F, int MODE>
int by_block(int block, const FqDeviceItem* items_host, int count, size_t total_tiles, cudaStream_t stream)
{
    switch (block) {
    case 16: return run<T, F, 16, MODE>(items_host, count, total_tiles, stream);
    case 32: return run<T, F, 32, MODE>(items_host, count, total_tiles, stream);
    case 64: return run<T, F, 64, MODE>(items_host, count, total_tiles, stream);
    case 128: return run<T, F, 128, MODE>(items_host, count, total_tiles, stream);
    default: return MXQ_ERR_BLOCK;
    }
}

template <class T, class F>
int by_mode(int mode, int block, const FqDeviceItem* items_host, int count, size_t total_tiles, cudaStream_t stream)
{
    constexpr bool anchor = F::id == MXQ_INT8 || F::id == MXQ_FP8_E4M3;
    if (mode == MXQ_FQ_DIRECT || anchor) return by_block<T, F, MXQ_FQ_DIRECT>(block, items_host, count, total_tiles, stream);
    if constexpr (!anchor) return by_block<T, F, MXQ_FQ_VIA_ANCHOR>(block, items_host, count, total_tiles, stream);
    return MXQ_ERR_FORMAT;
}

}  // namespace

size_t fq_batched_tiles(size_t nunits) { return (nunits + kThreads * kU * kR - 1) / (kThreads * kU * kR); }

int launch_fake_quant_batched(const FqDeviceItem* items_host, int count, size_t total_tiles, int dtype, int fmt,
                              int block, int mode, cudaStream_t stream)
{
    MXQ_DISPATCH_FORMAT(fmt, {
        if (dtype == MXQ_F32) return by_mode<F32, F>(mode, block, items_host, count, total_tiles, stream);
        return by_mode<BF16, F>(mode, block, items_host, count, total_tiles, stream);
    });
    return MXQ_ERR_FORMAT;
}

}  // namespace mxq
