// gp_rank.cu -- Spearman's rank correlation fitness (Sec. III-C3: ranks of
// the values, then Karl Pearson's coefficient of the ranks).
//
// Unlike the fused metrics this one needs every prediction of a program at
// once: a batch of programs is predicted into [B][N], each segment is sorted
// by value (a stable LSD radix sort, 8-bit digits in 4 passes, of
// order-preserving 32-bit keys with the row index as payload; the first
// pass reads the predictions themselves), ties get the mean of their
// positions, and the weighted moments of the rank pairs are summed in FP64
// with a fixed partition.  Without weights, and up to 4M rows, the values are
// ranked bucket by bucket instead (below), and the sort is what remains for
// segments that the buckets' sample misjudged.  The target's ranks are sorted
// once per call.  Ranks are kept doubled (first + last position, 1-based),
// which is an integer; the correlation does not see the factor 2.
#include <algorithm>
#include <type_traits>

#include "gp_internal.cuh"
#include "gp_rank_sample.cuh"

namespace gpk {
namespace {

// rank pass: 2048 sorted keys per block
constexpr int kTileItems = 8;                          // per thread
constexpr int kTileThreads = 256;
constexpr int kTile = kTileItems * kTileThreads;

// LSD radix sort: 8-bit digits, 4 passes over tiles of 4096 keys, which
// the histogram kernel reads as 256 threads x 16 keys (key r * 256 + t of
// the tile to thread t) and the scatter as 512 threads x 8
constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortItems = 16;
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kRadixBits = 8;
constexpr int kBins = 1 << kRadixBits;
constexpr int kPasses = 32 / kRadixBits;

// order-preserving key of a float (-0 and +0 become the same key)
__device__ __forceinline__ uint32_t float_key(float f) {
    if (f == 0.0f) f = 0.0f;
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// key of item m of a segment: pass 0 reads the float values, later passes
// the keys of the previous pass
template <bool FROM_FLOAT>
__device__ __forceinline__ uint32_t load_key(const void *src, int64_t m) {
    if (FROM_FLOAT) return float_key(static_cast<const float *>(src)[m]);
    return static_cast<const uint32_t *>(src)[m];
}

// The segments that a kernel's blocks work on: all of them, one per
// blockIdx.y, or, with a list on the device, the *count listed ones of them,
// taken in turn by the gridDim.y rows of blocks.
struct Segs {
    const int32_t *list;
    const int32_t *count;
    int all;
    unsigned rows(int64_t x) const { return (unsigned)(list ? listed_rows(all, x) : all); }
};
template <class F>
__device__ __forceinline__ void each_segment(const Segs &sg, F body) {
    const int n = sg.list ? *sg.count : sg.all;
    for (int i = blockIdx.y; i < n; i += gridDim.y) {
        body(sg.list ? sg.list[i] : i);
        __syncthreads();  // the next one reuses the shared memory
    }
}

// digit counts of one tile: hist[seg][digit][tile].  Each thread loads its
// 16 keys first (independent loads), then counts them into its warp's own
// histogram; a warp whose 32 keys share one digit adds once.
template <bool FROM_FLOAT>
__global__ void __launch_bounds__(kSortThreads) hist_kernel(const void *__restrict__ src, int64_t n,
                                                            int n_tiles, int shift, int32_t *hist,
                                                            uint32_t *nan_flag, Segs sg) {
    __shared__ int32_t wh[kSortWarps][kBins];
    each_segment(sg, [&](int seg) {
    const int tile = blockIdx.x, t = threadIdx.x;
    const int lane = t & 31, warp = t >> 5;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) wh[w][t] = 0;
    const int64_t t0 = (int64_t)tile * kSortTile;
    const int tl = (int)min((int64_t)kSortTile, n - t0);
    const int64_t so = (int64_t)seg * n + t0;
    uint32_t d[kSortItems];
    bool nan = false;
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const int i = r * kSortThreads + t;
        uint32_t k = 0;
        if (i < tl) {
            if (FROM_FLOAT) {
                const float f = static_cast<const float *>(src)[so + i];
                nan |= f != f;
                k = float_key(f);
            } else {
                k = static_cast<const uint32_t *>(src)[so + i];
            }
        }
        d[r] = i < tl ? (k >> shift) & (kBins - 1) : (uint32_t)kBins;  // kBins: not counted
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const uint32_t d0 = __shfl_sync(0xffffffffu, d[r], 0);
        if (__all_sync(0xffffffffu, d[r] == d0)) {
            if (lane == 0 && d0 < kBins) atomicAdd(&wh[warp][d0], 32);
        } else if (d[r] < kBins) {
            atomicAdd(&wh[warp][d[r]], 1);
        }
    }
    if (FROM_FLOAT && __any_sync(0xffffffffu, nan) && lane == 0) atomicOr(nan_flag + seg, 1u);
    __syncthreads();
    int32_t c = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) c += wh[w][t];
    hist[((int64_t)seg * kBins + t) * n_tiles + tile] = c;
    });
}

// per (segment, digit), one warp: exclusive scan of the tile counts in
// place, and the digit's total in tot[seg][digit]
__global__ void __launch_bounds__(256) tile_scan_kernel(int32_t *hist, int32_t *tot, int n_tiles,
                                                        Segs sg) {
    const int lane = threadIdx.x & 31;
    const int digit = (int)(blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5));  // < kBins
    each_segment(sg, [&](int seg) {
    const int64_t row = (int64_t)seg * kBins + digit;
    int32_t *h = hist + row * n_tiles;
    int32_t carry = 0;
    for (int base = 0; base < n_tiles; base += 32) {
        const int i = base + lane;
        const int32_t v = i < n_tiles ? h[i] : 0;
        int32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (i < n_tiles) h[i] = carry + x - v;
        carry += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) tot[row] = carry;
    });
}

// exclusive scan of one value per thread over the block (blockDim.x
// threads, wsum: one entry per warp)
__device__ __forceinline__ int32_t block_exclusive_scan(int32_t v, int32_t *wsum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    int32_t before = 0;
    for (int q = 0; q < warp; ++q) before += wsum[q];
    __syncthreads();
    return before + x - v;
}

// the scatter's tile: 512 threads x 8 keys (warp w owns keys [256 w, 256 w + 256))
constexpr int kScatThreads = 512;
constexpr int kScatWarps = kScatThreads / 32;
constexpr int kScatItems = kSortTile / kScatThreads;

// lanes of the warp whose digit equals this lane's (8-bit digits): one
// ballot per bit, as CUB does it, or the match instruction
template <bool BALLOT>
__device__ __forceinline__ unsigned digit_peers(uint32_t d) {
    if constexpr (BALLOT) {
        unsigned peers = 0xffffffffu;
#pragma unroll
        for (int b = 0; b < kRadixBits; ++b) {
            const bool bit = (d >> b) & 1u;
            const unsigned m = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? m : ~m;
        }
        return peers;
    } else {
        return __match_any_sync(0xffffffffu, d);
    }
}

constexpr bool kBallotPeers = true;

// Stable scatter of one tile by one digit.  The tile is ranked in shared
// memory first (warp-level digit groups in key order, then a scan over
// (digit, warp)), staged in sorted order, and written out run by run so
// that neighbouring threads store to neighbouring addresses.  Padding
// beyond a ragged tile's end takes digit 255 and, being last in key order,
// sorted positions >= the tile length, which are not written.  Pass 0
// reads float values and produces the payload: the row index, or, when
// vals is given, vals[row] (a per-row table shared by the segments).  Two
// blocks per SM (64 registers); three, at 40 registers with spills, ran
// the rank fitness 3% slower.
template <bool FROM_FLOAT>
__global__ void __launch_bounds__(kScatThreads, 2) scatter_kernel(
    const void *__restrict__ src, const uint32_t *__restrict__ vals, int64_t n, int n_tiles,
    int shift, const int32_t *__restrict__ offs, const int32_t *__restrict__ tot,
    uint32_t *keys_out, uint32_t *vals_out, Segs sg) {
    __shared__ uint32_t sk[kSortTile];
    __shared__ uint32_t sv[kSortTile];
    __shared__ int32_t wcnt[kScatWarps][kBins];
    __shared__ int32_t dstart[kBins];
    __shared__ int32_t gbase[kBins];
    __shared__ int32_t wsum[kScatWarps];
    each_segment(sg, [&](int seg) {
    const int tile = blockIdx.x, t = threadIdx.x;
    const int lane = t & 31, warp = t >> 5;
    const int64_t t0 = (int64_t)tile * kSortTile;
    const int tl = (int)min((int64_t)kSortTile, n - t0);
    const int64_t so = (int64_t)seg * n;
    for (int i = t; i < kScatWarps * kBins; i += kScatThreads) (&wcnt[0][0])[i] = 0;
    // the digit totals and this tile's digit offsets, loaded ahead of the keys
    const int32_t my_tot = t < kBins ? tot[(int64_t)seg * kBins + t] : 0;
    const int32_t my_off = t < kBins ? offs[((int64_t)seg * kBins + t) * n_tiles + tile] : 0;
    uint32_t kk[kScatItems], vv[kScatItems];
#pragma unroll
    for (int r = 0; r < kScatItems; ++r) {
        const int i = warp * (kScatItems * 32) + r * 32 + lane;
        const bool in = i < tl;
        kk[r] = in ? load_key<FROM_FLOAT>(src, so + t0 + i) : 0xffffffffu;
        if (FROM_FLOAT) vv[r] = vals ? (in ? vals[t0 + i] : 0u) : (uint32_t)(t0 + i);
        else vv[r] = in ? vals[so + t0 + i] : 0u;
    }
    // global position of this tile's first item of digit t: the digit's
    // start in the segment plus the same digit in earlier tiles
    const int32_t dbase = block_exclusive_scan(my_tot, wsum);
    if (t < kBins) gbase[t] = dbase + my_off;
    // the lanes holding one digit in a round form a group; its lowest lane
    // reserves the group's places with one atomic (predicated, so that the
    // rounds' atomics issue back to back; shared-memory atomics of one warp
    // keep their order) and hands the old count to the others afterwards
    const unsigned lt = (1u << lane) - 1u;
    uint32_t old[kScatItems];
    int32_t off[kScatItems];
    unsigned char lead[kScatItems];
#pragma unroll
    for (int r = 0; r < kScatItems; ++r) {
        const uint32_t d = (kk[r] >> shift) & (kBins - 1);
        const unsigned peers = digit_peers<kBallotPeers>(d);
        const int leader = __ffs(peers) - 1;
        const uint32_t addr = (uint32_t)__cvta_generic_to_shared(&wcnt[warp][d]);
        old[r] = 0u;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.eq.u32 p, %1, %2;\n\t"
            "@p atom.shared.add.u32 %0, [%3], %4;\n\t}"
            : "+r"(old[r])
            : "r"((uint32_t)lane), "r"((uint32_t)leader), "r"(addr), "r"((uint32_t)__popc(peers))
            : "memory");
        lead[r] = (unsigned char)leader;
        off[r] = __popc(peers & lt);
    }
#pragma unroll
    for (int r = 0; r < kScatItems; ++r)
        off[r] += (int32_t)__shfl_sync(0xffffffffu, old[r], lead[r]);
    __syncthreads();
    // digit t: warps' exclusive prefixes, then the digits' starts in the tile
    int32_t run = 0;
    if (t < kBins) {
#pragma unroll
        for (int w = 0; w < kScatWarps; ++w) {
            const int32_t c = wcnt[w][t];
            wcnt[w][t] = run;
            run += c;
        }
    }
    const int32_t ds = block_exclusive_scan(run, wsum);
    if (t < kBins) dstart[t] = ds;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kScatItems; ++r) {
        const uint32_t d = (kk[r] >> shift) & (kBins - 1);
        const int pos = dstart[d] + wcnt[warp][d] + off[r];
        sk[pos] = kk[r];
        sv[pos] = vv[r];
    }
    __syncthreads();
#pragma unroll 4
    for (int pos = t; pos < tl; pos += kScatThreads) {
        const uint32_t k = sk[pos];
        const uint32_t d = (k >> shift) & (kBins - 1);
        const int64_t g = so + gbase[d] + (pos - dstart[d]);
        keys_out[g] = k;
        vals_out[g] = sv[pos];
    }
    });
}

// first index in [lo, hi) of k with k[i] >= v (k ascending)
__device__ int64_t lower_bound_u32(const uint32_t *k, int64_t lo, int64_t hi, uint32_t v) {
    while (lo < hi) {
        const int64_t mid = lo + (hi - lo) / 2;
        if (k[mid] < v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

__device__ int64_t upper_bound_u32(const uint32_t *k, int64_t lo, int64_t hi, uint32_t v) {
    while (lo < hi) {
        const int64_t mid = lo + (hi - lo) / 2;
        if (k[mid] <= v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Tie-group ends at the tile edges: edge[seg][tile] = (first position of
// the group of the tile's first key, last position of the group of its last
// key).  One thread per tile; the binary search runs only when the group
// crosses the edge, which keeps the rank pass free of dependent global loads.
__global__ void __launch_bounds__(256) edges_kernel(const uint32_t *__restrict__ keys, int64_t n,
                                                    int n_tiles, int2 *edge, Segs sg) {
    const int tile = blockIdx.x * blockDim.x + threadIdx.x;
    each_segment(sg, [&](int seg) {
    if (tile >= n_tiles) return;
    const uint32_t *k = keys + (int64_t)seg * n;
    const int64_t t0 = (int64_t)tile * kTile;
    const int64_t t1 = min(n, t0 + kTile);  // one past the tile's last key
    const uint32_t first = k[t0], last = k[t1 - 1];
    const int64_t lo = (t0 > 0 && k[t0 - 1] == first) ? lower_bound_u32(k, 0, t0, first) : t0;
    const int64_t hi = (t1 < n && k[t1] == last) ? upper_bound_u32(k, t1, n, last) - 1 : t1 - 1;
    edge[(int64_t)seg * n_tiles + tile] = make_int2((int)lo, (int)hi);
    });
}

// Doubled average rank of every sorted position (first + last + 2, 1-based
// positions of its tie group).  Groups inside a tile are found with
// ballots over the sorted keys in shared memory; a group that reaches the
// tile's edge takes its end from edge[] (edges_kernel).  Ranks enter the sums centred on
// n + 1 (their unweighted mean): exact integers, zero for every row of a
// constant program, and sums without the cancellation of uncentred squares.
// mode 0 (the target): r2[row] = rank, and part = (sum w, sum w b,
// sum w b^2) of the tile; mode 1 (programs): part = (sum w a, sum w a^2,
// sum w a b), b = the target's centred rank of the row, read from r2y by
// the row in vals or, with vals_are_ranks (unweighted rows), carried in
// vals itself by the sort.  Unweighted and
// with n <= 2^29 a thread's sums are exact 64-bit integers; otherwise FP64.
// One FP64 triple per (segment, tile), added in a fixed order.
__global__ void __launch_bounds__(kTileThreads) rank_kernel(
    const uint32_t *__restrict__ keys, const uint32_t *__restrict__ vals, int64_t n, int n_tiles,
    int mode, const int2 *__restrict__ edge, uint32_t *r2, const uint32_t *__restrict__ r2y,
    const float *__restrict__ w, double *part, int vals_are_ranks, Segs sg) {
    constexpr int kSegs = kTile / 32;  // 32-position segments of the tile
    __shared__ uint32_t sk[kTile];
    __shared__ int16_t sfirst[kTile], slast[kTile];
    __shared__ int seg_first[kSegs], seg_last[kSegs];
    __shared__ double red[3][kTileThreads / 32];
    each_segment(sg, [&](int seg) {
    const int tile = blockIdx.x, t = threadIdx.x;
    const int lane = t & 31;
    const uint32_t *k = keys + (int64_t)seg * n;
    const uint32_t *vl = vals + (int64_t)seg * n;
    const int64_t t0 = (int64_t)tile * kTile;
    const int tl = (int)min((int64_t)kTile, n - t0);
    // the tile's keys: independent loads issued together
    uint32_t kv[kTileItems];
#pragma unroll
    for (int it = 0; it < kTileItems; ++it) {
        const int q = it * kTileThreads + t;
        kv[it] = q < tl ? k[t0 + q] : 0u;
    }
#pragma unroll
    for (int it = 0; it < kTileItems; ++it) {
        const int q = it * kTileThreads + t;
        if (q < tl) sk[q] = kv[it];
    }
    const int2 eg = edge[(int64_t)seg * n_tiles + tile];
    // the rows of this thread's items, then their target ranks: independent
    // loads issued together
    uint32_t rows[kTileItems], rb[kTileItems];
#pragma unroll
    for (int it = 0; it < kTileItems; ++it) {
        const int q = it * kTileThreads + t;
        rows[it] = q < tl ? vl[t0 + q] : 0u;
    }
#pragma unroll
    for (int it = 0; it < kTileItems; ++it) {
        const int q = it * kTileThreads + t;
        rb[it] = (mode == 1 && q < tl) ? (vals_are_ranks ? rows[it] : r2y[rows[it]]) : 0u;
    }
    __syncthreads();
    // tie groups inside the tile: the warp's 32 positions q = it * 256 + t
    // are consecutive, so ballots of the group-start and group-end flags
    // give each position the latest start at or before it and the earliest
    // end at or after it within its 32-position segment; a segment without
    // one takes it from the segments before (after) it, scanned by warp 0
    const unsigned le = (2u << lane) - 1u, ge = ~((1u << lane) - 1u);
#pragma unroll
    for (int it = 0; it < kTileItems; ++it) {
        const int q = it * kTileThreads + t;
        const int sgi = q >> 5;
        const bool in = q < tl;
        const uint32_t v = in ? sk[q] : 0u;
        const bool start = in && (q == 0 || sk[q - 1] != v);
        const bool end = in && (q == tl - 1 || sk[q + 1] != v);
        const unsigned bs = __ballot_sync(0xffffffffu, start);
        const unsigned be = __ballot_sync(0xffffffffu, end);
        if (in) {
            sfirst[q] = (int16_t)((bs & le) ? (sgi << 5) + 31 - __clz(bs & le) : -1);
            slast[q] = (int16_t)((be & ge) ? (sgi << 5) + __ffs(be & ge) - 1 : -1);
        }
        if (lane == 0) {
            seg_first[sgi] = bs ? (sgi << 5) + 31 - __clz(bs) : -1;
            seg_last[sgi] = be ? (sgi << 5) + __ffs(be) - 1 : INT_MAX;
        }
    }
    __syncthreads();
    if (t < 32) {
        // exclusive prefix max of the segments' latest starts, exclusive
        // suffix min of their earliest ends (two segments per lane)
        const int a0 = seg_first[2 * t], a1 = seg_first[2 * t + 1];
        const int b0 = seg_last[2 * t], b1 = seg_last[2 * t + 1];
        int x = max(a0, a1);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (t >= o) x = max(x, y);
        }
        int before = __shfl_up_sync(0xffffffffu, x, 1);
        if (t == 0) before = -1;
        int z = min(b0, b1);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_down_sync(0xffffffffu, z, o);
            if (t + o < 32) z = min(z, y);
        }
        int after = __shfl_down_sync(0xffffffffu, z, 1);
        if (t == 31) after = INT_MAX;
        __syncwarp();
        seg_first[2 * t] = before;
        seg_first[2 * t + 1] = max(before, a0);
        seg_last[2 * t + 1] = after;
        seg_last[2 * t] = min(after, b1);
    }
    __syncthreads();
    const bool exact = w == nullptr && n <= ((int64_t)1 << 29);
    long long is[3] = {0, 0, 0};
    double s[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int it = 0; it < kTileItems; ++it) {
        const int q = it * kTileThreads + t;
        if (q >= tl) break;
        int lq = sfirst[q], uq = slast[q];
        if (lq < 0) lq = seg_first[q >> 5];
        if (uq < 0) uq = seg_last[q >> 5];
        const int64_t first = lq == 0 ? (int64_t)eg.x : t0 + lq;
        const int64_t last = uq == tl - 1 ? (int64_t)eg.y : t0 + uq;
        const uint32_t rank2 = (uint32_t)(first + last + 2);
        const uint32_t row = rows[it];
        const int a = (int)((int64_t)rank2 - (n + 1));  // |a| <= n - 1
        if (mode == 0) r2[row] = rank2;
        const int b = mode == 0 ? 1 : (int)((int64_t)rb[it] - (n + 1));
        if (exact) {
            // mode 0: (count, sum a, sum a^2); mode 1: (sum a, sum a^2, sum a b)
            is[0] += mode == 0 ? 1 : a;
            is[1] += mode == 0 ? a : (long long)a * a;
            is[2] += (long long)a * (mode == 0 ? a : b);
        } else {
            const double wv = w ? (double)w[row] : 1.0;
            const double ad = (double)a;
            const double wa = wv * ad;
            if (mode == 0) {
                s[0] += wv;
                s[1] += wa;
                s[2] = fma(wa, ad, s[2]);
            } else {
                s[0] += wa;
                s[1] = fma(wa, ad, s[1]);
                s[2] = fma(wa, (double)b, s[2]);
            }
        }
    }
    if (exact) {
#pragma unroll
        for (int j = 0; j < 3; ++j) s[j] = (double)is[j];
    }
    // fixed butterfly inside each warp, then the warps in order
#pragma unroll
    for (int j = 0; j < 3; ++j) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s[j] += __shfl_xor_sync(0xffffffffu, s[j], o);
    }
    if ((t & 31) == 0) {
#pragma unroll
        for (int j = 0; j < 3; ++j) red[j][t >> 5] = s[j];
    }
    __syncthreads();
    if (t < 3) {
        double v = 0.0;
        for (int q = 0; q < kTileThreads / 32; ++q) v += red[t][q];
        part[((int64_t)seg * n_tiles + tile) * 3 + t] = v;
    }
    });
}

// sum of tile triples in a fixed order: lane-strided, then lanes in order
__device__ __forceinline__ void sum_tiles(const double *p, int n_tiles, double (&S)[3]) {
    const int lane = threadIdx.x & 31;
    double s[3] = {0.0, 0.0, 0.0};
    for (int i = lane; i < n_tiles; i += 32)
#pragma unroll
        for (int j = 0; j < 3; ++j) s[j] += p[(int64_t)i * 3 + j];
#pragma unroll
    for (int j = 0; j < 3; ++j) S[j] = 0.0;
    for (int l = 0; l < 32; ++l)
#pragma unroll
        for (int j = 0; j < 3; ++j) S[j] += __shfl_sync(0xffffffffu, s[j], l);
}

// the sums of a's ranks that the bucket path collects: exact integers, the
// two products as limbs v = hi 2^32 + lo
struct RankSums {
    unsigned long long a, a2lo, a2hi, ablo, abhi;
};

__device__ __forceinline__ double limbs(unsigned long long hi, unsigned long long lo) {
    return (double)(long long)hi * 4294967296.0 + (double)(long long)lo;
}

// one warp per segment: |r| of the ranks from the program's sums -- exact
// (sums; kept: segments of the bucket path) or per tile -- and the target's
// totals (sum w, sum w b, sum w b^2)
__global__ void __launch_bounds__(256) spearman_final_kernel(
    const double *part, const RankSums *sums, const int32_t *listed, const double *total, int n_seg,
    int n_tiles, const uint32_t *nan_flag, float *out, double *out64) {
    const int lane = threadIdx.x & 31;
    const int seg = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    if (seg >= n_seg) return;
    double P[3];
    if (sums && !listed[seg]) {
        const RankSums s = sums[seg];
        P[0] = (double)(long long)s.a;
        P[1] = limbs(s.a2hi, s.a2lo);
        P[2] = limbs(s.abhi, s.ablo);
    } else {
        sum_tiles(part + (int64_t)seg * n_tiles * 3, n_tiles, P);
    }
    if (lane != 0) return;
    const double sw = total[0];
    const double ma = P[0] / sw, mb = total[1] / sw;
    const double va = P[1] / sw - ma * ma, vb = total[2] / sw - mb * mb;
    const double cov = P[2] / sw - ma * mb;
    double f;
    if (nan_flag[seg] || !isfinite(va) || !isfinite(vb) || !isfinite(cov)) f = __longlong_as_double(0x7ff8000000000000LL);
    else if (!(va > 0.0) || !(vb > 0.0)) f = 0.0;
    else f = fabs(cov) / sqrt(va * vb);
    out[seg] = (float)f;
    if (out64) out64[seg] = f;
}

// the target's totals after its tile sums
__global__ void __launch_bounds__(32) target_total_kernel(const double *tpart, int n_tiles,
                                                          double *total) {
    double T[3];
    sum_tiles(tpart, n_tiles, T);
    if (threadIdx.x < 3) total[threadIdx.x] = T[threadIdx.x];
}

// Sorts each of n_seg segments of n float values into keys (order-preserving
// integers) with the row index as payload, or payload[row] when a per-row
// table is given; the result is in keys/vals.
// hist holds n_seg * 256 * n_tiles counts, tot n_seg * 256.
cudaError_t radix_sort_values(const float *v, uint32_t *keys, uint32_t *vals, uint32_t *keys2,
                              uint32_t *vals2, int64_t n, int32_t *hist, int32_t *tot,
                              uint32_t *nan_flag, const uint32_t *payload, const Segs &sg,
                              cudaStream_t st) {
    const int n_tiles = (int)((n + kSortTile - 1) / kSortTile);
    const dim3 grid(n_tiles, sg.rows(n_tiles)), scan_grid(kBins / 8, sg.rows(kBins / 8));
    for (int pass = 0; pass < kPasses; ++pass) {
        const int shift = pass * kRadixBits;
        // pass 0: values -> keys2; then keys2 -> keys -> keys2 -> keys
        const uint32_t *ki = (pass & 1) ? keys2 : keys;
        const uint32_t *vi = (pass & 1) ? vals2 : vals;
        uint32_t *ko = (pass & 1) ? keys : keys2;
        uint32_t *vo = (pass & 1) ? vals : vals2;
        if (pass == 0) {
            hist_kernel<true><<<grid, kSortThreads, 0, st>>>(v, n, n_tiles, shift, hist, nan_flag, sg);
        } else {
            hist_kernel<false><<<grid, kSortThreads, 0, st>>>(ki, n, n_tiles, shift, hist, nullptr, sg);
        }
        tile_scan_kernel<<<scan_grid, 256, 0, st>>>(hist, tot, n_tiles, sg);
        if (pass == 0) {
            scatter_kernel<true><<<grid, kScatThreads, 0, st>>>(v, payload, n, n_tiles, shift, hist,
                                                                tot, ko, vo, sg);
        } else {
            scatter_kernel<false><<<grid, kScatThreads, 0, st>>>(ki, vi, n, n_tiles, shift, hist,
                                                                 tot, ko, vo, sg);
        }
    }
    return cudaGetLastError();  // 4 passes: the result is in keys/vals
}

// ---- ranks by buckets --------------------------------------------------
// Without weights the coefficient needs each value's rank only next to the
// target's rank of its row, so no segment has to be sorted as a whole:
//   splitter_kernel   a sorted sample of the segment's keys (sample_row) gives
//                     splitters for buckets of about kBucketAim keys
//   partition_kernel  every key goes, with the target's rank of its row, to
//                     its bucket (of at most kBucketCap places).  Keys equal
//                     to a splitter -- every value frequent enough to fill a
//                     bucket is one -- need no place: they share one rank, so
//                     their number and the sum of their targets' ranks do,
//                     counted per tile in shared memory
//   base_kernel       first position of every bucket; the splitters' shares
//   local_kernel      a bucket in shared memory: 4096 equal bins over its key
//                     range, about one key each, then a key's rank is the
//                     bin's start plus the smaller keys in the bin (a bin
//                     of one value that repeats: the bin's start)
// The sums are integers and exact, so no order shows in them.  A segment
// with an overfull bucket (the sample misjudged it) is listed, and the radix
// sort below runs for the listed segments alone.
// Bound by the global traffic of the partition (4 B read, 8 B written as runs
// of about 6 keys, 8 B read) and shared-memory atomics; the radix sort moves
// 84 B a key and spends about 800 instructions on it.  512 programs x 1M rows:
// 20.5 -> 9.75 ms; a batch of 164 programs x 2^20 rows takes 0.71 ms of
// predictions, 0.12 of splitters, 1.09 of partition (tiles of 4096 keys or
// other block sizes: 6 to 23% more) and 1.43 of local ranks.
constexpr int kPartThreads = 512, kPartItems = 16, kPartTile = kPartThreads * kPartItems;
constexpr int kLocThreads = 512, kLocItems = kBucketCap / kLocThreads, kLocBins = 4096;
constexpr int kLocKeys = 8192;   // kBucketCap to a power of two, for the bitonic sort
constexpr int kTogether = 4;   // lanes with one key that add their sum at once
constexpr int kBusy = 32;      // keys in one bin that make a look for bins of one value worth it
constexpr int kCrowded = 128;  // keys in one bin of several values that make the bucket sort

// weighted sums are FP64 and need a fixed order; beyond kMaxBuckets the
// partition's runs get too short
static inline bool bucket_path(const float *w, int64_t n) {
    return w == nullptr && bucket_count(n) <= kMaxBuckets;
}

// per segment of a batch
struct Buckets {
    int nb, p2;               // buckets; splitters padded to a power of two
    uint32_t *split;          // [seg][p2], ascending, then 0xffffffff
    int32_t *cnt, *eqc;       // [seg][nb] keys in the bucket, equal to its splitter
    unsigned long long *eqb;  // [seg][nb] sum of the targets' centred ranks of the latter
    int32_t *base;            // [seg][nb] first position
    RankSums *sums;           // [seg]
    int32_t *listed;          // [seg] 1: left to the radix sort
    int32_t *list, *count;    // those segments
    uint2 *kv;                // [seg][nb][kBucketCap]
};

// ascending bitonic sort of p2 keys in shared memory by the whole block
__device__ void bitonic_sort(uint32_t *k, int p2) {
    for (int size = 2; size <= p2; size *= 2)
        for (int d = size / 2; d > 0; d /= 2) {
            __syncthreads();
            for (int i = threadIdx.x; i < p2 / 2; i += blockDim.x) {
                const int lo = 2 * i - (i & (d - 1)), hi = lo + d;
                const uint32_t a = k[lo], b = k[hi];
                const bool up = (lo & size) == 0;
                k[lo] = up ? min(a, b) : max(a, b);
                k[hi] = up ? max(a, b) : min(a, b);
            }
        }
    __syncthreads();
}

__global__ void __launch_bounds__(1024) splitter_kernel(const float *__restrict__ pred, int64_t n,
                                                        int samples, Buckets B, uint32_t *nan_flag) {
    extern __shared__ uint32_t sample[];
    const int seg = blockIdx.x, t = threadIdx.x;
    const float *v = pred + (int64_t)seg * n;
    const int log2_samples = 31 - __clz(samples);
    for (int i = t; i < samples; i += blockDim.x) sample[i] = float_key(v[sample_row(i, n, log2_samples)]);
    for (int j = t; j < B.nb; j += blockDim.x) {
        const int64_t q = (int64_t)seg * B.nb + j;
        B.cnt[q] = 0;
        B.eqc[q] = 0;
        B.eqb[q] = 0ull;
    }
    if (t == 0) {
        B.sums[seg] = RankSums{0ull, 0ull, 0ull, 0ull, 0ull};
        B.listed[seg] = 0;
        nan_flag[seg] = 0u;
        if (seg == 0) *B.count = 0;
    }
    bitonic_sort(sample, samples);
    for (int j = t; j < B.p2; j += blockDim.x)
        B.split[(int64_t)seg * B.p2 + j] =
            j < B.nb - 1 ? sample[((int64_t)(j + 1) * samples) / B.nb] : 0xffffffffu;
}

__global__ void __launch_bounds__(kPartThreads, 2) partition_kernel(
    const float *__restrict__ pred, int64_t n, const uint32_t *__restrict__ r2y, Buckets B,
    uint32_t *nan_flag) {
    extern __shared__ uint32_t smem_part[];
    uint2 *stage = reinterpret_cast<uint2 *>(smem_part);                      // [kPartTile]
    int2 *place = reinterpret_cast<int2 *>(stage + kPartTile);                // [nb] see below
    uint32_t *split = reinterpret_cast<uint32_t *>(place + B.nb);             // [p2]
    uint32_t *tree = split + B.p2;                                            // [p2] see below
    int32_t *cnt = reinterpret_cast<int32_t *>(tree + B.p2);                  // [nb] the tile's counts
    uint16_t *sj = reinterpret_cast<uint16_t *>(cnt + B.nb);                  // [kPartTile] bucket
    __shared__ int32_t wsum[kPartThreads / 32];
    const int seg = blockIdx.y, t = threadIdx.x, lane = t & 31;
    const int64_t t0 = (int64_t)blockIdx.x * kPartTile;
    const int tl = (int)min((int64_t)kPartTile, n - t0);
    const float *v = pred + (int64_t)seg * n + t0;
    uint32_t key[kPartItems];
    int j[kPartItems];
    bool nan = false;
#pragma unroll
    for (int r = 0; r < kPartItems; ++r) {
        const int i = r * kPartThreads + t;
        const float f = i < tl ? v[i] : 0.0f;
        nan |= f != f;
        key[r] = float_key(f);
        j[r] = 1;
    }
    // the splitters as a search tree by levels (node i over nodes 2i and
    // 2i + 1): a level's nodes lie side by side, so the lanes' reads of the
    // upper levels meet no bank twice (a binary search over the sorted array
    // reads addresses 32 apart there, all in one bank)
    for (int i = t; i < B.p2; i += kPartThreads) {
        const uint32_t *sp = B.split + (int64_t)seg * B.p2;
        split[i] = sp[i];
        if (i == 0) continue;  // node 1 is the root
        const int level = 31 - __clz(i);
        tree[i] = sp[(2 * (i - (1 << level)) + 1) * (B.p2 >> (level + 1)) - 1];
    }
    // the tile's keys equal to a splitter: their number (from bit 18) and the
    // upper bits of their targets' ranks, the lower 18 bits.  8192 ranks of at
    // most 2^23, one of them at most that large, fit; the staged keys take their
    // place afterwards
    uint32_t *eq_hi = reinterpret_cast<uint32_t *>(stage), *eq_lo = eq_hi + B.nb;  // [nb] each
    static_assert(2 * kMaxBuckets * sizeof(uint32_t) <= kPartTile * sizeof(uint2), "room for them");
    static_assert(2ll * kMaxBuckets * kBucketAim <= 1 << 23 && kPartTile <= 1 << 13, "ranks of 23 bits");
    for (int i = t; i < B.nb; i += kPartThreads) cnt[i] = 0, eq_hi[i] = eq_lo[i] = 0u;
    if (__any_sync(0xffffffffu, nan) && lane == 0) atomicOr(nan_flag + seg, 1u);
    __syncthreads();
    // the number of splitters below the key
    for (int size = B.p2; size > 1; size /= 2) {
#pragma unroll
        for (int r = 0; r < kPartItems; ++r) j[r] = 2 * j[r] + (tree[j[r]] < key[r] ? 1 : 0);
    }
    int off[kPartItems];  // place in the tile's share of the bucket; -1: none needed
#pragma unroll
    for (int r = 0; r < kPartItems; ++r) {
        const int i = r * kPartThreads + t;
        const bool in = i < tl;
        j[r] = min(j[r] - B.p2, B.nb - 1);
        const bool eq = in && j[r] < B.nb - 1 && split[j[r]] == key[r];
        off[r] = in && !eq ? atomicAdd(&cnt[j[r]], 1) : -1;
        // several lanes equal to one splitter add once, the others by themselves
        // (a turn for each splitter of a warp, with its sums in global memory: 156
        // columns of 1M values of two decimals 12.5 ms, now 2.6; the sort 6.0)
        unsigned em = __ballot_sync(0xffffffffu, eq);
        if (em) {
            const uint32_t rank = eq ? r2y[t0 + i] : 0u;
            bool left = eq;
            while (em) {
                const int src = __ffs(em) - 1;
                const int j0 = __shfl_sync(0xffffffffu, j[r], src);
                const bool mine = left && j[r] == j0;
                const unsigned mm = __ballot_sync(0xffffffffu, mine);
                const int same = __popc(mm);
                if (same < kTogether) break;
                const uint32_t sum = __reduce_add_sync(0xffffffffu, mine ? rank : 0u);  // below 2^29
                if (lane == src) {
                    atomicAdd(&eq_hi[j[r]], (uint32_t)same << 18 | sum >> 18);
                    atomicAdd(&eq_lo[j[r]], sum & 0x3ffffu);
                }
                left = left && !mine;
                em &= ~mm;
            }
            if (left) {
                atomicAdd(&eq_hi[j[r]], 1u << 18 | rank >> 18);
                atomicAdd(&eq_lo[j[r]], rank & 0x3ffffu);
            }
        }
    }
    __syncthreads();
    // place[b]: the first of bucket b's keys in the tile, and from there to
    // their places in the bucket (at most 4 buckets per thread)
    int run = 0, c[kMaxBuckets / kPartThreads];
    const int per = (B.nb + kPartThreads - 1) / kPartThreads;
#pragma unroll
    for (int q = 0; q < kMaxBuckets / kPartThreads; ++q) {
        const int b = t * per + q;
        c[q] = q < per && b < B.nb ? cnt[b] : 0;
        run += c[q];
    }
    int start = block_exclusive_scan(run, wsum);
#pragma unroll
    for (int q = 0; q < kMaxBuckets / kPartThreads; ++q) {
        const int b = t * per + q;
        if (q < per && b < B.nb) {
            const int at = c[q] ? atomicAdd(&B.cnt[(int64_t)seg * B.nb + b], c[q]) : 0;
            place[b] = make_int2(start, at - start);
            const uint32_t hi = eq_hi[b], same = hi >> 18;
            if (same) {  // the ranks centred
                const int64_t g = (int64_t)seg * B.nb + b;
                const int64_t sum = ((int64_t)(hi & 0x3ffffu) << 18) + eq_lo[b];
                atomicAdd(&B.eqc[g], (int32_t)same);
                atomicAdd(&B.eqb[g], (unsigned long long)(sum - (int64_t)same * (n + 1)));
            }
        }
        start += c[q];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kPartItems; ++r) {
        if (off[r] < 0) continue;
        const int pos = place[j[r]].x + off[r];
        stage[pos] = make_uint2(key[r], r2y[t0 + r * kPartThreads + t]);
        sj[pos] = (uint16_t)j[r];
    }
    if (t == kPartThreads - 1) wsum[0] = start;  // the keys staged in all
    __syncthreads();
    const int m = wsum[0];
    uint2 *kv = B.kv + (int64_t)seg * B.nb * kBucketCap;
    for (int pos = t; pos < m; pos += kPartThreads) {
        const int b = sj[pos], at = place[b].y + pos;
        if (at < kBucketCap) kv[(int64_t)b * kBucketCap + at] = stage[pos];
    }
}

// adds to a segment's sums: its a, and products as limbs (exact)
__device__ __forceinline__ void add_sums(RankSums *s, long long a, unsigned long long a2lo,
                                         long long a2hi, unsigned long long ablo, long long abhi) {
    atomicAdd(&s->a, (unsigned long long)a);
    atomicAdd(&s->a2lo, a2lo);
    atomicAdd(&s->a2hi, (unsigned long long)a2hi);
    atomicAdd(&s->ablo, ablo);
    atomicAdd(&s->abhi, (unsigned long long)abhi);
}

constexpr long long kLow32 = 0xffffffffll;

__global__ void __launch_bounds__(256) base_kernel(int64_t n, Buckets B) {
    __shared__ int32_t wsum[8];
    const int seg = blockIdx.x, t = threadIdx.x;
    const int per = (B.nb + 255) / 256;  // <= 8
    int run = 0;
    bool over = false;
    for (int q = 0; q < per; ++q) {
        const int b = t * per + q;
        if (b >= B.nb) break;
        const int64_t at = (int64_t)seg * B.nb + b;
        over |= B.cnt[at] > kBucketCap;
        run += B.cnt[at] + B.eqc[at];
    }
    int pos = block_exclusive_scan(run, wsum);
    over = __syncthreads_or(over);
    if (over && t == 0) {
        B.listed[seg] = 1;
        B.list[atomicAdd(B.count, 1)] = seg;
    }
    for (int q = 0; q < per; ++q) {
        const int b = t * per + q;
        if (b >= B.nb) break;
        const int64_t at = (int64_t)seg * B.nb + b;
        B.base[at] = pos;
        pos += B.cnt[at];
        const int c = B.eqc[at];
        if (c) {  // positions pos .. pos + c - 1 (0-based) share the doubled rank
            const long long a = 2ll * pos + c + 1 - (n + 1), a2 = a * a;
            const long long sb = (long long)B.eqb[at];
            // a sb in 128 bits, as limbs
            const unsigned long long ab = (unsigned long long)(a * sb);
            const long long abhi = (long long)((unsigned long long)__mul64hi(a, sb) << 32 | ab >> 32);
            add_sums(&B.sums[seg], c * a, (unsigned long long)(c * (a2 & kLow32)), c * (a2 >> 32),
                     ab & (unsigned long long)kLow32, abhi);
        }
        pos += c;
    }
}

// DIRECT: the segment is one bucket, read from the predictions themselves
template <bool DIRECT>
__global__ void __launch_bounds__(kLocThreads, 3) local_kernel(
    const float *__restrict__ pred, const uint32_t *__restrict__ r2y, int64_t n, Buckets B,
    uint32_t *nan_flag) {
    __shared__ __align__(16) uint32_t bins[kLocBins + 4];
    extern __shared__ uint32_t keys[];  // [kLocKeys]
    __shared__ int32_t wsum[kLocThreads / 32];
    __shared__ uint32_t s_lo, s_hi;
    __shared__ __align__(8) uint8_t mixed[kLocBins];  // 1: the bin holds several values
    __shared__ long long red[3][kLocThreads / 32];
    const int seg = DIRECT ? blockIdx.x : blockIdx.y, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t q = DIRECT ? 0 : (int64_t)seg * B.nb + blockIdx.x;
    const int m = DIRECT ? (int)n : B.cnt[q];
    if (m == 0 || m > kBucketCap) return;  // overfull: the segment is listed
    const int64_t base = DIRECT ? 0 : B.base[q];
    // the key range: between the bucket's splitters, or, at the segment's
    // ends, the keys' own
    const bool ends = DIRECT || blockIdx.x == 0 || blockIdx.x == B.nb - 1;
    uint32_t lo = 0xffffffffu, hi = 0u;
    if (!ends) {
        lo = B.split[(int64_t)seg * B.p2 + blockIdx.x - 1] + 1u;
        hi = B.split[(int64_t)seg * B.p2 + blockIdx.x] - 1u;
    }
    uint32_t key[kLocItems];
    bool nan = false;
#pragma unroll
    for (int r = 0; r < kLocItems; ++r) {
        if (r * kLocThreads >= m) break;
        const int i = r * kLocThreads + t;
        key[r] = 0u;
        if (i < m) {
            if (DIRECT) {
                const float f = pred[(int64_t)seg * n + i];
                nan |= f != f;
                key[r] = float_key(f);
            } else {
                key[r] = B.kv[q * kBucketCap + i].x;
            }
            if (ends) {
                lo = min(lo, key[r]);
                hi = max(hi, key[r]);
            }
        }
    }
    uint4 *bins4 = reinterpret_cast<uint4 *>(bins);
    static_assert(kLocBins == 8 * kLocThreads, "two uint4 of bins per thread");
    bins4[t] = bins4[kLocThreads + t] = make_uint4(0u, 0u, 0u, 0u);
    reinterpret_cast<uint2 *>(mixed)[t] = make_uint2(0u, 0u);
    if (t == 0) {
        s_lo = 0xffffffffu;
        s_hi = 0u;
    }
    if (DIRECT) nan = __syncthreads_or(nan);
    else __syncthreads();
    if (ends) {
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (lane == 0) {
            atomicMin(&s_lo, lo);
            atomicMax(&s_hi, hi);
        }
        __syncthreads();
        lo = s_lo;
        hi = s_hi;
    }
    // bin = (key - lo) kLocBins / (range + 1), rounded down; key - lo itself
    // when that is below kLocBins (the quotient in FP32, 2^-22 too small, so
    // the largest key stays below the last bin's end)
    const uint32_t range = hi - lo;
    const uint32_t mult =
        range < kLocBins ? 0u
                         : (uint32_t)__fdiv_rd((float)kLocBins * 4294967296.0f * (1.0f - 0x1p-22f),
                                               __uint2float_ru(range));
    auto bin_of = [&](uint32_t k) { return mult ? __umulhi(k - lo, mult) : k - lo; };
    uint32_t off[kLocItems];
#pragma unroll
    for (int r = 0; r < kLocItems; ++r) {
        if (r * kLocThreads >= m) break;
        if (r * kLocThreads + t < m) off[r] = atomicAdd(&bins[bin_of(key[r])], 1u);
    }
    __syncthreads();
    uint32_t most;
    {
        const uint4 u = bins4[2 * t], v = bins4[2 * t + 1];
        const uint32_t c[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
        uint32_t run = 0u, x[8];
        most = 0u;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            x[i] = run;
            run += c[i];
            most = max(most, c[i]);
        }
        const uint32_t at = (uint32_t)block_exclusive_scan((int32_t)run, wsum);
        bins4[2 * t] = make_uint4(at + x[0], at + x[1], at + x[2], at + x[3]);
        bins4[2 * t + 1] = make_uint4(at + x[4], at + x[5], at + x[6], at + x[7]);
        if (t == kLocThreads - 1) bins[kLocBins] = at + run;
    }
    const bool busy = __syncthreads_or(most > kBusy && mult != 0u);
#pragma unroll
    for (int r = 0; r < kLocItems; ++r) {
        if (r * kLocThreads >= m) break;
        if (r * kLocThreads + t < m) keys[bins[bin_of(key[r])] + off[r]] = key[r];
    }
    // Well-filled bins mostly hold one value that repeats, whose keys need no
    // look at the others of the bin and make no bucket sort.  512 columns of
    // 100003 values of two decimals took 2.9 ms with both, the plain sort 2.1,
    // now 1.1; 2000 columns of 6000 distinct values 0.46 -> 0.48 (0.93)
    bool crowded = false;
    if (busy) {
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kLocItems; ++r) {
            if (r * kLocThreads >= m) break;
            if (r * kLocThreads + t >= m) continue;
            const uint32_t bin = bin_of(key[r]);
            if (keys[bins[bin]] != key[r]) mixed[bin] = 1;
        }
        __syncthreads();
        // the thread's 8 bins: one that is mixed and long?
        bool many = false;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            many |= mixed[8 * t + i] && bins[8 * t + i + 1] - bins[8 * t + i] > kCrowded;
        crowded = __syncthreads_or(many);
    }
    if (crowded) {
        const int p2 = 1 << (32 - __clz(max(m - 1, 1)));
        for (int i = m + t; i < p2; i += kLocThreads) keys[i] = 0xffffffffu;
        bitonic_sort(keys, p2);
    }
    __syncthreads();
    long long s[3] = {0, 0, 0};
#pragma unroll
    for (int r = 0; r < kLocItems; ++r) {
        if (r * kLocThreads >= m) break;
        if (r * kLocThreads + t >= m) continue;
        const uint32_t k = key[r];
        int less, same;
        if (crowded) {
            int x = 0, y = m;
            while (x < y) {
                const int mid = (x + y) / 2;
                if (keys[mid] < k) x = mid + 1;
                else y = mid;
            }
            less = x;
            y = m;
            while (x < y) {
                const int mid = (x + y) / 2;
                if (keys[mid] <= k) x = mid + 1;
                else y = mid;
            }
            same = x - less;
        } else if (mult == 0u) {  // one value per bin
            less = (int)bins[k - lo];
            same = (int)bins[k - lo + 1] - less;
        } else {
            const uint32_t bin = bin_of(k);
            const int b0 = (int)bins[bin], b1 = (int)bins[bin + 1];
            less = b0;
            same = b1 - b0;
            if (!busy || mixed[bin]) {
                same = 0;
                for (int x = b0; x < b1; ++x) {
                    less += keys[x] < k;
                    same += keys[x] == k;
                }
            }
        }
        const long long a = 2ll * (base + less) + same + 1 - (n + 1);
        // the target's rank, from the cache: held in a register since the key's
        // load it would cost a resident block
        const int i = r * kLocThreads + t;
        const long long b = (long long)(DIRECT ? r2y[i] : B.kv[q * kBucketCap + i].y) - (n + 1);
        s[0] += a;
        s[1] += a * a;
        s[2] += a * b;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
        if (lane == 0) red[k][warp] = s[k];
    }
    __syncthreads();
    if (t != 0) return;
    for (int w = 1; w < kLocThreads / 32; ++w)
        for (int k = 0; k < 3; ++k) red[k][0] += red[k][w];
    const unsigned long long a2lo = red[1][0] & kLow32, ablo = red[2][0] & kLow32;
    if (DIRECT) {
        B.sums[seg] = RankSums{(unsigned long long)red[0][0], a2lo, (unsigned long long)(red[1][0] >> 32),
                               ablo, (unsigned long long)(red[2][0] >> 32)};
        B.listed[seg] = 0;
        nan_flag[seg] = nan ? 1u : 0u;
    } else {
        add_sums(&B.sums[seg], red[0][0], a2lo, red[1][0] >> 32, ablo, red[2][0] >> 32);
    }
}

size_t partition_smem(const Buckets &B) {
    return (size_t)kPartTile * (sizeof(uint2) + sizeof(uint16_t)) + (size_t)B.p2 * 8 + (size_t)B.nb * 12;
}

cudaError_t bucket_ranks(const float *pred, int n_seg, int64_t n, const uint32_t *r2y,
                         const Buckets &B, uint32_t *nan_flag, cudaStream_t st) {
    const size_t smem_l = kLocKeys * sizeof(uint32_t);
    cudaError_t e = cudaFuncSetAttribute(B.nb == 1 ? local_kernel<true> : local_kernel<false>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_l);
    if (e != cudaSuccess) return e;
    if (B.nb == 1) {
        local_kernel<true><<<n_seg, kLocThreads, smem_l, st>>>(pred, r2y, n, B, nan_flag);
        return cudaGetLastError();
    }
    const int samples = pow2_at_least(B.nb * kOversample);
    const size_t smem_s = (size_t)samples * 4, smem_p = partition_smem(B);
    e = cudaFuncSetAttribute(splitter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem_s);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(partition_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_p);
    if (e != cudaSuccess) return e;
    splitter_kernel<<<n_seg, std::min(1024, samples / 2), smem_s, st>>>(pred, n, samples, B, nan_flag);
    const dim3 tiles((unsigned)((n + kPartTile - 1) / kPartTile), n_seg);
    partition_kernel<<<tiles, kPartThreads, smem_p, st>>>(pred, n, r2y, B, nan_flag);
    base_kernel<<<n_seg, 256, 0, st>>>(n, B);
    local_kernel<false><<<dim3(B.nb, n_seg), kLocThreads, smem_l, st>>>(pred, r2y, n, B, nan_flag);
    return cudaGetLastError();
}

}  // namespace

// scratch of one batch of n_seg segments: keys, vals and their second
// buffers, the tile digit counts, the digit totals, the rank partials and
// the NaN flags
struct RankScratch {
    uint32_t *keys, *vals, *keys2, *vals2;
    int32_t *hist, *tot;
    double *part;
    int2 *edge;
    uint32_t *nan_flag;
    size_t bytes;
};

RankScratch carve_rank(void *scratch, int n_seg, int64_t n, bool buckets, Buckets *B) {
    const int64_t sort_tiles = (n + kSortTile - 1) / kSortTile;
    const int64_t rank_tiles = (n + kTile - 1) / kTile;
    auto al = [](int64_t x) { return (size_t)((x + 255) / 256 * 256); };
    char *b = static_cast<char *>(scratch);
    RankScratch r{};
    size_t o = 0;
    auto take = [&](auto **p, int64_t bytes) {
        *p = reinterpret_cast<std::remove_reference_t<decltype(*p)>>(b + o);
        o += al(bytes);
    };
    take(&r.nan_flag, (int64_t)n_seg * 4);
    size_t end = 0;
    if (buckets) {
        *B = Buckets{};
        B->nb = bucket_count(n);
        B->p2 = pow2_at_least(B->nb);
        take(&B->sums, (int64_t)n_seg * sizeof(RankSums));
        take(&B->listed, (int64_t)n_seg * 4);
        if (B->nb > 1) {
            take(&B->split, (int64_t)n_seg * B->p2 * 4);
            take(&B->cnt, (int64_t)n_seg * B->nb * 4);
            take(&B->eqc, (int64_t)n_seg * B->nb * 4);
            take(&B->eqb, (int64_t)n_seg * B->nb * 8);
            take(&B->base, (int64_t)n_seg * B->nb * 4);
            take(&B->list, (int64_t)n_seg * 4);
            take(&B->count, 4);
            // the buckets lie where the radix sort's arrays do: it runs after
            // they are done with
            B->kv = reinterpret_cast<uint2 *>(b + o);
            end = o + al((int64_t)n_seg * B->nb * kBucketCap * 8);
        } else {
            r.bytes = o;  // one bucket never overflows
            return r;
        }
    }
    take(&r.keys, (int64_t)n_seg * n * 4);
    take(&r.vals, (int64_t)n_seg * n * 4);
    take(&r.keys2, (int64_t)n_seg * n * 4);
    take(&r.vals2, (int64_t)n_seg * n * 4);
    take(&r.hist, (int64_t)n_seg * kBins * sort_tiles * 4);
    take(&r.tot, (int64_t)n_seg * kBins * 4);
    take(&r.part, (int64_t)n_seg * rank_tiles * 3 * 8);
    take(&r.edge, (int64_t)n_seg * rank_tiles * 8);
    r.bytes = std::max(o, end);
    return r;
}

// the radix path's sort, tie groups and rank sums for the segments sg
cudaError_t radix_ranks(const float *v, int64_t n, const RankScratch &r, const uint32_t *payload,
                        int mode, uint32_t *r2, const uint32_t *r2y, const float *w, double *part,
                        uint32_t *nan_flag, const Segs &sg, cudaStream_t st) {
    const int64_t n_tiles = (n + kTile - 1) / kTile;
    cudaError_t e = radix_sort_values(v, r.keys, r.vals, r.keys2, r.vals2, n, r.hist, r.tot, nan_flag,
                                      payload, sg, st);
    if (e != cudaSuccess) return e;
    const unsigned edge_blocks = (unsigned)((n_tiles + 255) / 256);
    edges_kernel<<<dim3(edge_blocks, sg.rows(edge_blocks)), 256, 0, st>>>(r.keys, n, (int)n_tiles, r.edge, sg);
    rank_kernel<<<dim3((unsigned)n_tiles, sg.rows(n_tiles)), kTileThreads, 0, st>>>(
        r.keys, r.vals, n, (int)n_tiles, mode, r.edge, r2, r2y, w, part, payload ? 1 : 0, sg);
    return cudaGetLastError();
}

size_t rank_scratch_bytes(int n_seg, int64_t n, bool weighted) {
    Buckets B;
    const float one = 1.0f;
    // the target's own sort uses the same memory
    return std::max(carve_rank(nullptr, n_seg, n, bucket_path(weighted ? &one : nullptr, n), &B).bytes,
                    carve_rank(nullptr, 1, n, false, &B).bytes);
}

// tile sums, then their totals
size_t target_part_bytes(int64_t n) { return ((size_t)((n + kTile - 1) / kTile) + 1) * 3 * 8; }

cudaError_t target_ranks(const float *y, const float *w, int64_t n, void *scratch, uint32_t *r2y,
                         double *tpart, cudaStream_t st) {
    const int64_t n_tiles = (n + kTile - 1) / kTile;
    Buckets B;
    const RankScratch r = carve_rank(scratch, 1, n, false, &B);
    cudaError_t e = cudaMemsetAsync(r.nan_flag, 0, 4, st);
    if (e != cudaSuccess) return e;
    e = radix_ranks(y, n, r, nullptr, 0, r2y, nullptr, w, tpart, r.nan_flag, Segs{nullptr, nullptr, 1}, st);
    if (e != cudaSuccess) return e;
    target_total_kernel<<<1, 32, 0, st>>>(tpart, (int)n_tiles, tpart + 3 * n_tiles);
    return cudaGetLastError();
}

cudaError_t spearman_batch(const float *pred, int n_seg, int64_t n, const uint32_t *r2y,
                           const double *tpart, const float *w, void *scratch, float *out,
                           double *out64, cudaStream_t st) {
    const int64_t n_tiles = (n + kTile - 1) / kTile;
    const bool buckets = bucket_path(w, n);
    Buckets B{};
    const RankScratch r = carve_rank(scratch, n_seg, n, buckets, &B);
    cudaError_t e = cudaSuccess;
    if (buckets) {
        if ((e = bucket_ranks(pred, n_seg, n, r2y, B, r.nan_flag, st)) != cudaSuccess) return e;
    } else {
        if ((e = cudaMemsetAsync(r.nan_flag, 0, (size_t)n_seg * 4, st)) != cudaSuccess) return e;
    }
    // unweighted rows need only the target's rank of each row: the sort
    // carries it as the payload, so the rank pass reads it in sorted order
    // instead of gathering it by row
    const uint32_t *payload = w == nullptr ? r2y : nullptr;
    if (!buckets || B.nb > 1) {
        const Segs sg = buckets ? Segs{B.list, B.count, n_seg} : Segs{nullptr, nullptr, n_seg};
        e = radix_ranks(pred, n, r, payload, 1, nullptr, r2y, w, r.part, r.nan_flag, sg, st);
        if (e != cudaSuccess) return e;
    }
    spearman_final_kernel<<<(n_seg + 7) / 8, 256, 0, st>>>(r.part, buckets ? B.sums : nullptr, B.listed,
                                                           tpart + 3 * n_tiles, n_seg, (int)n_tiles,
                                                           r.nan_flag, out, out64);
    return cudaGetLastError();
}

}  // namespace gpk
