// Host side of the several-target Slice-and-Scale: from a set of target formats to its kernel.  Included by one
// translation unit per anchor family.
#pragma once
#include <array>
#include <utility>

#include "mxq_kernels.cuh"
#include "mxq_launch.h"

namespace mxq {

constexpr int kSetU = 2;
constexpr int kSetThreads = 128;
constexpr int kSetTile = kSetU * kSetThreads;      // lane units per CTA

// The lower formats of an anchor in the order of the set's bit mask.
template <class FH>
struct SetFormats;
template <>
struct SetFormats<Fmt<MXQ_INT8>> {
    static constexpr int fmt[] = {MXQ_INT7, MXQ_INT6, MXQ_INT5, MXQ_INT4, MXQ_INT3, MXQ_INT2};
    static constexpr int count = 6;
};
template <>
struct SetFormats<Fmt<MXQ_FP8_E4M3>> {
    static constexpr int fmt[] = {MXQ_FP7_E3M3, MXQ_FP6_E3M2, MXQ_FP6_E2M3, MXQ_FP5_E2M2, MXQ_FP4_E2M1};
    static constexpr int count = 5;
};

constexpr int set_size(unsigned mask)
{
    int n = 0;
    for (; mask; mask &= mask - 1) ++n;
    return n;
}

// index in the family's list of the I-th member of the set
constexpr int set_member(unsigned mask, int i)
{
    for (int b = 0;; ++b)
        if ((mask >> b & 1u) && i-- == 0) return b;
}

template <class FH>
constexpr int set_index(int fmt)
{
    for (int b = 0; b < SetFormats<FH>::count; ++b)
        if (SetFormats<FH>::fmt[b] == fmt) return b;
    return -1;
}

struct SetArgs {
    const uint8_t* codes;
    const uint8_t* scales;
    size_t n;
    int block;
    const SsOut* outs;         // by index in SetFormats
    cudaStream_t stream;
};

template <class FH, unsigned MASK, size_t... I>
int run_set(const SetArgs& a, std::index_sequence<I...>)
{
    constexpr int N = sizeof...(I);
    const SsOuts<N> outs{{a.outs[set_member(MASK, (int)I)]...}};
    auto kern = slice_scale_set_kernel<FH, kSetU, kSetThreads, Fmt<SetFormats<FH>::fmt[set_member(MASK, (int)I)]>...>;
    const size_t nunits = a.n / 32, nscales = a.n / (size_t)a.block;
    return launch_kernel(kern, grid_for_units(nunits, kSetTile), kSetThreads, a.stream, a.codes, a.scales, nunits, nscales, outs);
}

template <class FH, unsigned MASK>
int run_set_of(const SetArgs& a)
{
    if constexpr (set_size(MASK) >= 2 && set_size(MASK) <= kSetTargetsMax)
        return run_set<FH, MASK>(a, std::make_index_sequence<(size_t)set_size(MASK)>{});
    else
        return MXQ_ERR_PAIR;
}

// The function of every set, indexed by its mask.
template <class FH, size_t... M>
constexpr auto set_table(std::index_sequence<M...>)
{
    return std::array<int (*)(const SetArgs&), sizeof...(M)>{&run_set_of<FH, (unsigned)M>...};
}

// `ntargets` different lower formats of the anchor FH (2 ... kSetTargetsMax) in one pass.
template <class FH>
int launch_set(const uint8_t* codes, const uint8_t* scales, size_t n, int block, int ntargets, const int* fmts,
               const SsOut* outs, cudaStream_t stream)
{
    static constexpr auto table = set_table<FH>(std::make_index_sequence<(size_t)1 << SetFormats<FH>::count>{});
    SsOut by_index[SetFormats<FH>::count] = {};
    unsigned mask = 0;
    for (int k = 0; k < ntargets; ++k) {
        const int i = set_index<FH>(fmts[k]);
        if (i < 0 || (mask >> i & 1u)) return MXQ_ERR_PAIR;
        mask |= 1u << i;
        by_index[i] = outs[k];
    }
    return table[mask](SetArgs{codes, scales, n, block, by_index, stream});
}

// Two different lower formats of a set of anchors; the items' first output belongs to the format that comes first in
// SetFormats when `swap` is false, to the other one when it is true.
template <class FH, unsigned MASK>
int run_pair_batched(const SsPairDeviceItem* items_host, int count, size_t total_tiles, bool swap, cudaStream_t stream)
{
    if constexpr (set_size(MASK) == 2) {
        return with_item_capacity<kSsPairItemsMax>(count, [&](auto k) {
            constexpr int K = decltype(k)::value;
            SsPairItemBlock<K> blk;
            fill_item_block(blk, items_host, count, total_tiles);
            if (swap)
                for (int i = 0; i < count; ++i) std::swap(blk.items[i].out[0], blk.items[i].out[1]);
            auto kern = slice_scale_pair_batched_kernel<FH, Fmt<SetFormats<FH>::fmt[set_member(MASK, 0)]>,
                                                        Fmt<SetFormats<FH>::fmt[set_member(MASK, 1)]>, kSetU, kSetThreads, K>;
            return launch_kernel(kern, grid_for_units(total_tiles, 1), kSetThreads, stream, blk);
        });
    } else {
        return MXQ_ERR_PAIR;
    }
}

template <class FH, size_t... M>
constexpr auto pair_table(std::index_sequence<M...>)
{
    return std::array<int (*)(const SsPairDeviceItem*, int, size_t, bool, cudaStream_t), sizeof...(M)>{
        &run_pair_batched<FH, (unsigned)M>...};
}

template <class FH>
int launch_pair_batched(const SsPairDeviceItem* items_host, int count, size_t total_tiles, int fmt1, int fmt2,
                        cudaStream_t stream)
{
    static constexpr auto table = pair_table<FH>(std::make_index_sequence<(size_t)1 << SetFormats<FH>::count>{});
    const int a = set_index<FH>(fmt1), b = set_index<FH>(fmt2);
    if (a < 0 || b < 0 || a == b) return MXQ_ERR_PAIR;
    return table[1u << a | 1u << b](items_host, count, total_tiles, a > b, stream);
}

}  // namespace mxq
