// sample_row and the bucket sizes for test_rank_sample.py
#include "gp_rank_sample.cuh"
extern "C" {
int buckets(int64_t n) { return gpk::bucket_count(n); }
int capacity() { return gpk::kBucketCap; }
int samples(int64_t n) { return gpk::pow2_at_least(gpk::bucket_count(n) * gpk::kOversample); }
int64_t row(int i, int64_t n) { return gpk::sample_row(i, n, __builtin_ctz(samples(n))); }
}
