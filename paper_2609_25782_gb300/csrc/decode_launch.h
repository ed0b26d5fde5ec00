// Which kernels a decode call runs: a rule on its sizes, the SMs and the room for
// partials, as host code of its own, so that it can be checked without a GPU.
#pragma once

#include <algorithm>

#include "kvt_internal.h"

#ifdef __CUDACC__
#define KVT_BOTH __host__ __device__
#else
#define KVT_BOTH
#endif

namespace kvt {

constexpr int kAccs = 8;   // running softmax states of a split (decode_kernels.cu)
// The merge of a session's splits folds four chains (contiguous quarters of
// the splits, in split order) and then merges the chains in order; that order
// depends on the split count only, whichever kernel runs it. One warp merges
// up to kRegMergeMax splits from registers (four per chain); the split kernel
// merges sessions of up to kSplitKernelMerge splits itself in long grids.
constexpr int kMergeChains = 4;
constexpr int kRegMergeMax = 16;
constexpr int kSplitKernelMerge = 4;

#ifndef KVT_WAVE_MARGIN
#define KVT_WAVE_MARGIN 0.1   // last-wave fill gain that moves a grid to 2 CTAs per SM
#endif

// Partial rows per split of a grid whose splits are shared by `sub` CTAs: one
// per half where each of two CTAs holds one, one per accumulator for eight.
KVT_BOTH constexpr int parts_per_split(int sub) {
    return sub <= 2 ? sub : kAccs;
}

// Partial rows that a pool of `rows` rows for unshared splits (max_batch x Hq x
// splits) allocates, so that every call which decode_shape lets share its splits
// has room: 8 rows of a split at up to two CTAs per SM, or 2 at up to three.
inline int64_t shared_part_rows(int64_t rows, int num_sms, int group) {
    const int64_t wave = static_cast<int64_t>(num_sms) * group;
    return std::max({rows, std::min(8 * rows, 2 * wave), std::min(2 * rows, 3 * wave)});
}

struct DecodeShape {
    int32_t sub;               // CTAs that share a split: 1, 2 or 8
    int32_t per_sm;            // CTAs per SM that the kernel's ring is sized for
    int32_t pace;              // DecodeArgs::pace
    int32_t merge_max_splits;  // DecodeArgs::merge_max_splits
    bool one_split;            // no session has more than one split
    bool by_length;            // the longest sessions first
    bool wide;                 // tables of more than kRegMergeMax splits
    bool combine;              // a combine kernel follows
};

// a: sizes, tables' width and room for partials; splits: of that width.
inline DecodeShape decode_shape(const DecodeArgs &a, int splits, int num_sms, bool overlap_previous) {
    // CTAs of the grid (an upper bound: splits past a session's own count
    // exit at once) against the SMs decide the ring depth.
    const int64_t ctas = static_cast<int64_t>(splits) * a.s.Hkv * a.nlayers * a.B;
    // Beyond two CTAs per SM, 2 per SM still wins when it fills its last wave
    // clearly better than 3 per SM (a grid just above one 3-per-SM wave).
    auto fill = [&](int per_sm) {
        const double w = static_cast<double>(ctas) / (per_sm * static_cast<double>(num_sms));
        return w / static_cast<double>(static_cast<int64_t>(w) + (w > static_cast<int64_t>(w)));
    };
    // Splits shared by several CTAs. A grid of few CTAs leaves SMs idle, and
    // each of its CTAs draws 512 KB or more through one SM (6 us) with its
    // warps in each other's way; shared, a CTA has less to draw, holds more of
    // it before the previous call ends, and is gone sooner, so the next call's
    // CTAs start their copies sooner. The combine reads 2 or 8 states per split
    // instead of one. us per layer, unshared and shared:
    //   8 (one warp each, its ring the whole of a 64-tile split), at most two
    //     per SM: 1 x 3 001 8.04 and 5.14, 1 x 8K 8.51 and 5.70, 4 x 1 280 8.26
    //     and 5.10 (shared by 4 of two warps, one per SM: 6.85 and 6.51)
    //   2, at most one per SM: 1 x 16 391 9.97 and 8.72 (two CTAs per SM with
    //     half the ring 10.0, four of a shorter split 10.6)
    //   2, two per SM: 8 x 4K 13.1 and 12.4, 2 x 16K 13.3 and 12.6, 5 x 5K 11.6
    //     and 10.9 (three per SM 14.0, 14.0, 12.1)
    //   2, three per SM: 8 x 5K 17.1 and 15.7, 10 x 4K 17.4 and 15.7, 3 x 16K
    //     19.3 and 18.3; not the long splits of tables wider than 32K tokens
    //     (1 x 100K 34.3 and 35.0), which do share at two per SM (1 x 40K 16.8
    //     and 16.1)
    // Sessions of one split need no combine unshared, and do not share: from a
    // graph it would still pay for one to four of them above 512 tokens (1 x 1K
    // 6.04 and 5.10, but 8 x 1K 6.67 and 6.94, 48 x 1 000 18.4 and 21.0), while
    // direct calls would pay for the second launch. A caller's scratch may have
    // no room for the extra rows.
    const int64_t sms = num_sms;
    const int64_t rows1 = static_cast<int64_t>(splits) * a.s.Hq * a.nlayers * a.B;
    auto fits = [&](int sub, int per_sm) {
        return sub * ctas <= per_sm * sms && parts_per_split(sub) * rows1 <= a.part_rows;
    };
    const bool wide = splits > kRegMergeMax;   // long splits, and a combine in batches
    DecodeShape d = {};
    d.sub = 1;
    d.wide = wide;
    d.one_split = splits == 1;
    if (splits > 1 && !wide && fits(8, 2)) {
        d.sub = 8;
        d.per_sm = 2;
    } else if (splits > 1 && (fits(2, 1) || fits(2, 2) || (!wide && fits(2, 3)))) {
        d.sub = 2;
        d.per_sm = fits(2, 1) ? 1 : fits(2, 2) ? 2 : 3;
    } else if (d.one_split && ctas <= sms) {
        d.per_sm = 1;
    } else {
        d.per_sm = ctas <= 2 * sms || fill(2) > fill(3) + KVT_WAVE_MARGIN ? 2 : 3;
    }
    // An overlapped call whose CTAs are all resident at once fills its rings
    // while the previous call still merges: 20-30 MB of copies queued in front
    // of that call's partials, this call's q and the end of the grid between
    // them. Paced to one tile per warp (two with four warps per SM), the copies
    // still keep HBM busy and the chain behind them is shorter. us per layer,
    // unpaced and paced: one session of 16 391 tokens 8.64 and 7.98, 32K 13.6
    // and 12.7; 8 x 4K 15.0 and 13.2, 12 x 2K 12.1 and 11.4; 4 x 16K 24.1 and
    // 23.1. Rings that cover a whole split (8 CTAs per split) showed no
    // difference, and in grids of more than one wave the later CTAs lose by it
    // (8 x 16K 44.4 and 45.1). Calls without a combine (40 x 1 000 16.0 and
    // 16.9) and unshared long splits (1 x 100K) take no part.
    if (overlap_previous && d.sub == 2)
        d.pace = d.per_sm == 1 ? 2 : 1;
    else if (overlap_previous && d.sub == 1 && splits > 1 && !wide && ctas <= 2 * sms)
        d.pace = 1;
    // A grid of several waves ends when its last long splits do, with most SMs
    // waiting: where splits differ in length (tables wider than 16K tokens) the
    // longest sessions go out first. 48 layers of 16 sessions of 2K-30K tokens
    // 3 920 -> 3 822 us, of 32 of 8K-32K 9 188 -> 9 043, 24 layers of 12 of
    // 4K-60K 2 601 -> 2 531. Equal splits only lose by it, the block ids then
    // waiting for the ranks (24 of 1K-14K 2 879 and 2 920); a lane ranks one
    // session, so up to 32.
    d.by_length = a.nlayers == 1 && a.B > 1 && a.B <= 32 && d.sub == 1 && ctas > 3 * sms &&
                  split_tiles(a.max_blocks * a.s.bt) > KVT_SPLIT_MIN_TILES;
    // Which sessions the split kernel merges itself (the bits are the same
    // either way): those of up to kSplitKernelMerge splits, in grids of at
    // least 8 CTAs per SM. There, many groups finish at different times and
    // their merges spread over the grid. In shorter grids each CTA's arrival
    // (an atomic round trip holding its SM slot) and the tail merges cost more
    // than the combine launch (measured on GB300 against merging everything in
    // the combine: 256 x 4K-token sessions per layer +1.3 %, 8 x 4K all
    // layers +1.6 %; one 4K- or 16K-token session per layer -7 % / -5 % and
    // 32 x 4K -5 % when shorter grids merged too).
    d.merge_max_splits = ctas >= 8 * sms ? kSplitKernelMerge : 0;
    d.combine = d.sub > 1 || (splits > 1 && splits > d.merge_max_splits);
    return d;
}

}  // namespace kvt
