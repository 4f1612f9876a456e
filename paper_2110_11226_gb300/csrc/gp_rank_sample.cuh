// gp_rank_sample.cuh -- the buckets of the rank fitness (gp_rank.cu): their sizes
// and the rows whose values become the splitters between them.  Plain
// functions of integers, on the host and on the device.
#pragma once

#include <stdint.h>

namespace gpk {

constexpr int kBucketCap = 6144;
constexpr int kBucketAim = kBucketCap / 3;
constexpr int kMaxBuckets = 2048;
constexpr int kOversample = 16;  // sampled keys per bucket

#ifndef __CUDACC__
#define GP_RANK_FN inline
#else
#define GP_RANK_FN __host__ __device__ __forceinline__
#endif

GP_RANK_FN int pow2_at_least(int v) {
    int p = 1;
    while (p < v) p *= 2;
    return p;
}

// a few thousand rows are one bucket, taken straight from the predictions
GP_RANK_FN int bucket_count(int64_t n) {
    if (n <= kBucketCap) return 1;
    const int64_t nb = (n + kBucketAim - 1) / kBucketAim;
    return (int)(nb < kMaxBuckets + 1 ? nb : kMaxBuckets + 1);
}

// Row of sample i: one of each of 2^log2_samples equal strata of the rows, drawn
// by an integer hash (the finalizer of MurmurHash3).  Rows often follow one another by a
// rule -- grids, time series -- and every 64th or 128th row of a table with a
// period that shares a factor with that stride meets a few of its values
// only: of a 1024 x 1024 grid's fast axis 8, with 130,048 rows between two
// of them, where a bucket holds 6144.
GP_RANK_FN int64_t sample_row(int i, int64_t n, int log2_samples) {
    uint32_t h = (uint32_t)i;
    h = (h ^ (h >> 16)) * 0x85ebca6bu;
    h = (h ^ (h >> 13)) * 0xc2b2ae35u;
    h ^= h >> 16;
    const int64_t lo = (int64_t)i * n >> log2_samples, hi = (int64_t)(i + 1) * n >> log2_samples;
    return lo + (int64_t)((uint64_t)h * (uint64_t)(hi - lo) >> 32);
}

// Rows of blocks of a launch over the listed ones of n_seg segments, with x
// blocks per segment: the host does not know how many are listed, so as many
// as fill the device (4 blocks per SM) and no more, as most often none is and
// each block reads a zero.  With 4 rows whatever x is, 1024 programs of 16384
// rows (4 blocks each), all listed, took 10.7 ms, now 1.29 (the sort alone
// 0.90); with none listed 0.56 both.
GP_RANK_FN int64_t listed_rows(int64_t n_seg, int64_t x) {
    constexpr int64_t kBlocks = 4 * 152;
    int64_t rows = (kBlocks + x - 1) / x;
    rows = rows < 4 ? 4 : rows;
    return rows < n_seg ? rows : n_seg;
}

#undef GP_RANK_FN

}  // namespace gpk
