// Launchers of the several-target Slice-and-Scale (Eq. 4-5 applied to one read of the anchor), and the kernels of
// the MXINT8 anchor; those of the E4M3 anchor are in mxq_slice_scale_multi_fp.cu.
#include "mxq_slice_scale_set.cuh"

namespace mxq {

bool slice_scale_set_anchor(int src_fmt) { return src_fmt == MXQ_INT8 || src_fmt == MXQ_FP8_E4M3; }

int launch_slice_scale_set(const uint8_t* codes, const uint8_t* scales, size_t n, int block, int src_fmt, int ntargets,
                           const int* fmts, const SsOut* outs, cudaStream_t stream)
{
    if (src_fmt == MXQ_INT8) return launch_set<Fmt<MXQ_INT8>>(codes, scales, n, block, ntargets, fmts, outs, stream);
    if (src_fmt == MXQ_FP8_E4M3) return launch_slice_scale_set_e4m3(codes, scales, n, block, ntargets, fmts, outs, stream);
    return MXQ_ERR_PAIR;
}

size_t ss_pair_batched_tiles(size_t nunits) { return (nunits + kSetTile - 1) / kSetTile; }

int launch_slice_scale_pair_batched(const SsPairDeviceItem* items_host, int count, size_t total_tiles, int src_fmt, int fmt1,
                                    int fmt2, cudaStream_t stream)
{
    if (src_fmt == MXQ_INT8) return launch_pair_batched<Fmt<MXQ_INT8>>(items_host, count, total_tiles, fmt1, fmt2, stream);
    if (src_fmt == MXQ_FP8_E4M3)
        return launch_slice_scale_pair_batched_e4m3(items_host, count, total_tiles, fmt1, fmt2, stream);
    return MXQ_ERR_PAIR;
}

}  // namespace mxq
