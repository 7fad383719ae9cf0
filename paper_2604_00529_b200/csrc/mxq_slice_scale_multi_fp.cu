// The several-target Slice-and-Scale kernels of the E4M3 anchor (see mxq_slice_scale_multi.cu).
#include "mxq_slice_scale_set.cuh"

namespace mxq {

int launch_slice_scale_set_e4m3(const uint8_t* codes, const uint8_t* scales, size_t n, int block, int ntargets,
                                const int* fmts, const SsOut* outs, cudaStream_t stream)
{
    return launch_set<Fmt<MXQ_FP8_E4M3>>(codes, scales, n, block, ntargets, fmts, outs, stream);
}

int launch_slice_scale_pair_batched_e4m3(const SsPairDeviceItem* items_host, int count, size_t total_tiles, int fmt1,
                                         int fmt2, cudaStream_t stream)
{
    return launch_pair_batched<Fmt<MXQ_FP8_E4M3>>(items_host, count, total_tiles, fmt1, fmt2, stream);
}

}  // namespace mxq
