// gp_mutate.cu -- the mutation step on the device: the next population is
// built from tournament winners without leaving the GPU (the paper mutates
// on the CPU and copies every program back, Sec. III-C2 and III-D2, and
// names avoiding those transfers as future work, Sec. V).
//
// Three launches: one warp per offspring draws its kind and builds the
// child in its own 256-node scratch slot (Sec. II-A crossover, subtree,
// hoist and point mutation, reproduction; the hoisted crossover of
// Sec. III-C2 keeps the child within 20 stack slots and 255 nodes); one
// block turns the children's lengths into offsets; one warp per child
// copies it into the packed output.  Every random word comes from the
// offspring's own Philox4x32-10 stream, word k = Philox(counter = (k/4, t,
// offset lo32, offset hi32), key = seed)[k%4], so the output depends on
// nothing but the inputs.
#include "gp_internal.cuh"

namespace gpk {
namespace {

constexpr int kSlot = 256;  // scratch nodes per offspring

struct Stream {
    uint2 key;
    uint32_t t, c2, c3, k;
    uint4 r;
};

__device__ __forceinline__ uint32_t next_word(Stream &s) {
    if ((s.k & 3) == 0) s.r = philox4x32_10(make_uint4(s.k >> 2, s.t, s.c2, s.c3), s.key);
    const uint32_t w = (s.k & 3) == 0 ? s.r.x : (s.k & 3) == 1 ? s.r.y : (s.k & 3) == 2 ? s.r.z : s.r.w;
    s.k += 1;
    return w;
}

// an index in [0, n) from one word
__device__ __forceinline__ int pick(Stream &s, int n) {
    return (int)(((uint64_t)next_word(s) * (uint64_t)n) >> 32);
}

__device__ __forceinline__ int arity_of(int op) {
    if (op == GP_CONST || op == GP_VAR) return 0;
    if ((op >= GP_ADD && op <= GP_DIV) || op == GP_MAX || op == GP_MIN) return 2;
    if (op >= GP_SQRT && op <= GP_COSH) return 1;
    return -1;
}

// A prefix list in shared memory and, per node, the stack height after it in
// the reverse scan of Sec. III-A: terminals minus binary nodes from it to the
// end, counted 32 nodes at a time with ballots.  The nodes [i, i + size) of a
// subtree end where the height first falls below node i's.
struct List {
    uint2 node[256];    // op | feat << 16, constant
    uint8_t hgt[256];   // 0 at len
};

__device__ __forceinline__ int op_of(const List &l, int m) { return (int16_t)(l.node[m].x & 0xffffu); }

// fills l.hgt[0 .. len]; whether the list is a valid program.  The whole warp
__device__ bool scan_list(List &l, int len, int n_feat) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned ge = full << lane, gt = ge & ~(1u << lane);
    int carry = 0, hw = 0;
    bool ok = true;
    for (int c = (len - 1) >> 5; c >= 0; --c) {
        const int m = c * 32 + lane;
        const bool in = m < len;
        const int op = in ? op_of(l, m) : GP_NUM_OPS, ar = in ? arity_of(op) : 1;
        const unsigned leaf = __ballot_sync(full, ar == 0), bin = __ballot_sync(full, ar == 2);
        const int h = carry + __popc(leaf & ge) - __popc(bin & ge);
        const int before = carry + __popc(leaf & gt) - __popc(bin & gt);
        if (in) {
            const int feat = (int16_t)(l.node[m].x >> 16);
            ok = ok && ar >= 0 && before >= ar && !(op == GP_VAR && (feat < 0 || feat >= n_feat));
            l.hgt[m] = (uint8_t)h;
            hw = max(hw, h);
        }
        carry += __popc(leaf) - __popc(bin);
    }
    if (lane == 0) l.hgt[len] = 0;
    __syncwarp();
    return __all_sync(full, ok) && carry == 1 && __reduce_max_sync(full, hw) <= GP_MAX_STACK;
}

// nodes of the subtree rooted at node i
__device__ int subtree_size(const List &l, int len, int i) {
    const int lane = threadIdx.x & 31;
    for (int m0 = i + 1; m0 <= len; m0 += 32) {
        const int m = m0 + lane;
        const unsigned ends = __ballot_sync(0xffffffffu, m <= len && l.hgt[m] < l.hgt[i]);
        if (ends) return m0 + __ffs(ends) - 1 - i;
    }
    return len - i;  // unreachable for a valid program
}

// the largest height of nodes [m0, m1) (at least 0)
__device__ int highest(const List &l, int m0, int m1) {
    int h = 0;
    for (int m = m0 + (threadIdx.x & 31); m < m1; m += 32) h = max(h, (int)l.hgt[m]);
    return __reduce_max_sync(0xffffffffu, h);
}

// the caller's nodes are only 4-byte aligned
__device__ __forceinline__ uint2 load_node(const gp_node *p, int m) {
    const uint32_t *q = reinterpret_cast<const uint32_t *>(p) + 2 * m;
    return make_uint2(q[0], q[1]);
}

__device__ __forceinline__ uint2 bits_of(const gp_node &nd) {
    return make_uint2((uint32_t)(uint16_t)nd.op | (uint32_t)(uint16_t)nd.feat << 16, __float_as_uint(nd.c));
}

// variable f for f < n_feat, else a constant (w >> 8) * 2^-23 - 1 from the
// next word (exact in float, uniform on [-1, 1))
__device__ gp_node new_terminal(Stream &s, int n_feat) {
    gp_node nd;
    nd.op = GP_CONST;
    nd.feat = 0;
    nd.c = 0.0f;
    const int f = pick(s, n_feat + 1);
    if (f < n_feat) {
        nd.op = GP_VAR;
        nd.feat = (int16_t)f;
    } else {
        const uint32_t w = next_word(s);
        nd.c = __fsub_rn(__fmul_rn((float)(w >> 8), 0x1p-23f), 1.0f);
    }
    return nd;
}

// a "grow" tree of depth <= limit (<= 6, so <= 127 nodes) in prefix order:
// below the limit a node is a terminal when a word picks one of the 2
// terminal kinds among 2 + n_funcs, else one of the allowed functions.  Every
// lane draws the same words; depths: scratch of 128 entries
__device__ int grow_tree(Stream &s, const MutArgs &a, List &out, volatile uint8_t *depths) {
    const int lane = threadIdx.x & 31;
    int top = 0, n = 0;
    depths[top++] = 0;
    while (top > 0 && n < 127) {
        __syncwarp();
        const int d = depths[--top];
        __syncwarp();
        const bool terminal = d >= a.subtree_depth || pick(s, a.n_funcs + 2) < 2;
        gp_node nd;
        if (terminal) {
            nd = new_terminal(s, a.n_feat);
        } else {
            nd.op = a.funcs[pick(s, a.n_funcs)];
            nd.feat = 0;
            nd.c = 0.0f;
            for (int k = 0; k < arity_of(nd.op); ++k) depths[top++] = (uint8_t)(d + 1);
        }
        if (lane == 0) out.node[n] = bits_of(nd);
        ++n;
    }
    __syncwarp();
    return n;
}

// Length of the parent with subtree [i, i+si) replaced by donor subtree
// [j, j+sj), or 0 when that child would exceed 255 nodes or 20 stack slots.
// The nodes outside the subtree keep their heights (any subtree adds 1), and
// the donor's stand on the height behind the replaced one.
__device__ int splice_len(const List &par, int lp, int i, int si, const List &don, int j, int sj) {
    const int len = i + sj + (lp - i - si);
    if (len > GP_MAX_LEN) return 0;
    const int hw = max(max(highest(par, 0, i), highest(par, i + si, lp)),
                       (int)par.hgt[i + si] + highest(don, j, j + sj) - (int)don.hgt[j + sj]);
    return hw <= GP_MAX_STACK ? len : 0;
}

__device__ void splice_write(const List &par, int i, int si, const List &don, int j, int sj, int len,
                             uint2 *out) {
    for (int n = threadIdx.x & 31; n < len; n += 32)
        out[n] = n < i ? par.node[n] : n < i + sj ? don.node[j + n - i] : par.node[n - sj + si];
}

// the hoisted crossover: while the child does not fit, the donor subtree
// moves to a node drawn among its proper descendants
__device__ int hoisted_splice(Stream &s, const List &par, int lp, int i, const List &don, int ld, int j,
                              uint2 *out) {
    const int si = subtree_size(par, lp, i);
    int sj = subtree_size(don, ld, j);
    for (int guard = 0; guard <= GP_MAX_LEN; ++guard) {
        const int len = splice_len(par, lp, i, si, don, j, sj);
        if (len > 0) {
            splice_write(par, i, si, don, j, sj, len, out);
            return len;
        }
        if (sj == 1) return 0;  // a terminal always fits a valid parent
        j = j + 1 + pick(s, sj - 1);
        sj = subtree_size(don, ld, j);
    }
    return 0;
}

// One warp per offspring: every lane draws the same words, and the lists are
// scanned, searched and copied 32 nodes at a time in shared memory.  Bound by
// latency; one thread per offspring walking the lists in global memory took
// 49 us for 4096 offspring of 19 nodes, this 12 us.
constexpr int kPlanWarps = 4;

__global__ void __launch_bounds__(kPlanWarps * 32) mutate_plan_kernel(const MutArgs a) {
    __shared__ List lists[kPlanWarps][2];
    __shared__ uint8_t depths[kPlanWarps][128];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t = blockIdx.x * kPlanWarps + warp;
    if (t >= a.n_out) return;  // the whole warp
    List &par = lists[warp][0], &don = lists[warp][1];
    uint2 *child = reinterpret_cast<uint2 *>(a.scratch + (size_t)t * kSlot);
    Stream s;
    s.key = make_uint2((uint32_t)a.seed, (uint32_t)(a.seed >> 32));
    s.t = (uint32_t)t;
    s.c2 = (uint32_t)a.offset;
    s.c3 = (uint32_t)(a.offset >> 32);
    s.k = 0;
    const uint32_t u = next_word(s);
    int kind = GP_MUT_REPRODUCTION;
    for (int q = 0; q < 4; ++q)
        if ((uint64_t)u < a.thr[q]) {
            kind = q + 1;
            break;
        }
    const int pi = a.parents[2 * t], di = a.parents[2 * t + 1];
    const bool found = pi >= 0 && pi < a.n_progs && di >= 0 && di < a.n_progs;
    const int op0 = found ? a.offsets[pi] : 0, od = found ? a.offsets[di] : 0;
    int lp = found ? a.offsets[pi + 1] - op0 : 0;
    const int ld = found ? a.offsets[di + 1] - od : 0;
    if (!found && lane == 0) atomicOr(a.dev_status, GP_DEV_BAD_PARENT);
    if (lp < 1 || lp > GP_MAX_LEN) {  // a one-node program 0
        if (lane == 0) {
            child[0] = make_uint2(GP_CONST, 0u);
            a.lens[t] = 1;
            if (a.kind) a.kind[t] = GP_MUT_REPRODUCTION;
        }
        return;
    }
    for (int m = lane; m < lp; m += 32) par.node[m] = load_node(a.progs + op0, m);
    const bool donor = kind == GP_MUT_CROSSOVER && ld >= 1 && ld <= GP_MAX_LEN;
    if (donor)
        for (int m = lane; m < ld; m += 32) don.node[m] = load_node(a.progs + od, m);
    __syncwarp();
    if (!scan_list(par, lp, a.n_feat)) kind = GP_MUT_REPRODUCTION;
    if (kind == GP_MUT_CROSSOVER && !(donor && scan_list(don, ld, a.n_feat))) kind = GP_MUT_REPRODUCTION;

    int len = 0;
    if (kind == GP_MUT_CROSSOVER) {
        const int i = pick(s, lp);
        const int j = pick(s, ld);
        len = hoisted_splice(s, par, lp, i, don, ld, j, child);
    } else if (kind == GP_MUT_SUBTREE) {
        const int lt = grow_tree(s, a, don, depths[warp]);
        scan_list(don, lt, a.n_feat);
        const int i = pick(s, lp);
        len = hoisted_splice(s, par, lp, i, don, lt, 0, child);
    } else if (kind == GP_MUT_HOIST) {
        const int i = pick(s, lp);
        const int si = subtree_size(par, lp, i);
        const int k = si > 1 ? i + 1 + pick(s, si - 1) : i;
        const int sk = subtree_size(par, lp, k);
        len = splice_len(par, lp, i, si, par, k, sk);
        if (len > 0) splice_write(par, i, si, par, k, sk, len, child);
    } else if (kind == GP_MUT_POINT) {
        len = lp;
        for (int m = 0; m < lp; ++m) {
            if ((uint64_t)next_word(s) >= a.thr_replace) continue;
            const int ar = arity_of(op_of(par, m));
            gp_node nd;
            nd.op = GP_CONST;
            nd.feat = 0;
            nd.c = 0.0f;
            if (ar == 0) {
                nd = new_terminal(s, a.n_feat);
            } else {
                const int ns = ar == 1 ? a.n_unary : a.n_binary;
                if (ns <= 0) continue;
                const int idx = pick(s, ns);
                nd.op = ar == 1 ? a.unary[idx] : a.binary[idx];
            }
            __syncwarp();  // every lane has read node m
            if (lane == 0) par.node[m] = bits_of(nd);
        }
        __syncwarp();
        for (int m = lane; m < lp; m += 32) child[m] = par.node[m];
    }
    if (len == 0) {  // reproduction, or a splice that could not fit
        for (int m = lane; m < lp; m += 32) child[m] = par.node[m];
        len = lp;
        kind = GP_MUT_REPRODUCTION;
    }
    if (lane == 0) {
        a.lens[t] = len;
        if (a.kind) a.kind[t] = kind;
    }
}

// exclusive scan of the lengths in one block, 1024 at a time with a carry
__global__ void __launch_bounds__(1024) mutate_scan_kernel(const MutArgs a) {
    __shared__ int32_t warp_sum[32];
    __shared__ int32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int base = 0; base < a.n_out; base += 1024) {
        const int t = base + (int)threadIdx.x;
        const int32_t v = t < a.n_out ? a.lens[t] : 0;
        int32_t x = v;  // inclusive scan within the warp
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_sum[warp] = x;
        __syncthreads();
        if (warp == 0) {
            int32_t w = warp_sum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += y;
            }
            warp_sum[lane] = w;  // inclusive over warps
        }
        __syncthreads();
        const int32_t before = carry + (warp > 0 ? warp_sum[warp - 1] : 0) + x - v;
        if (t < a.n_out) a.out_offsets[t] = before;
        __syncthreads();
        if (threadIdx.x == 1023) carry = before + v;
        __syncthreads();
    }
    if (threadIdx.x == 0) a.out_offsets[a.n_out] = carry;
}

// one warp per child: scratch slot -> packed output
__global__ void __launch_bounds__(256) mutate_copy_kernel(const MutArgs a) {
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (t >= a.n_out) return;
    const int len = a.lens[t];
    const gp_node *src = a.scratch + (size_t)t * kSlot;
    gp_node *dst = a.out + a.out_offsets[t];
    for (int m = lane; m < len; m += 32) dst[m] = src[m];
}

}  // namespace

cudaError_t launch_mutate(const MutArgs &a, cudaStream_t st) {
    if (a.n_out <= 0) return cudaSuccess;
    mutate_plan_kernel<<<(a.n_out + kPlanWarps - 1) / kPlanWarps, kPlanWarps * 32, 0, st>>>(a);
    mutate_scan_kernel<<<1, 1024, 0, st>>>(a);
    mutate_copy_kernel<<<(a.n_out * 32 + 255) / 256, 256, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace gpk
