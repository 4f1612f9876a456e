// sample_row, the bucket sizes and listed_rows for test_rank_sample.py
#include "gp_rank_sample.cuh"
extern "C" {
int buckets(int64_t n) { return gpk::bucket_count(n); }
int capacity() { return gpk::kBucketCap; }
int samples(int64_t n) { return gpk::pow2_at_least(gpk::bucket_count(n) * gpk::kOversample); }
int64_t row(int i, int64_t n) { return gpk::sample_row(i, n, __builtin_ctz(samples(n))); }
int64_t listed_rows(int64_t n_seg, int64_t x) { return gpk::listed_rows(n_seg, x); }
}
