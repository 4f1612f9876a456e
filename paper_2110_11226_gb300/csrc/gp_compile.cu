// gp_compile.cu -- device pre-pass: validate each prefix list, compile it
// to the register-stack form (gp_internal.cuh), and sort the programs into
// classes (stack depth, extended functions) and by length (length-bucketed
// work queue); plus the
// deterministic total-weight sum.
#include <algorithm>

#include "gp_internal.cuh"
#include "gp_interp.cuh"

namespace gpk {

static __host__ __device__ inline int op_arity(int op) {
    if (op == GP_CONST || op == GP_VAR) return 0;
    if ((op >= GP_ADD && op <= GP_DIV) || op == GP_MAX || op == GP_MIN) return 2;
    if (op >= GP_SQRT && op <= GP_COSH) return 1;
    return -1;
}

static inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

Layout make_layout(int n_progs, int n_chunks, bool grad, bool moments) {
    Layout L{};
    size_t o = 0;
    size_t P = (size_t)(n_progs > 0 ? n_progs : 1);
    size_t C = (size_t)(n_chunks > 0 ? n_chunks : 1);
    L.counters = o;    o = align256(o + 8 * sizeof(unsigned long long));
    L.sumw = o;        o = align256(o + sizeof(double));
    L.sumw_part = o;   o = align256(o + kSumwBlocks * sizeof(double));
    L.code = o;        o = align256(o + P * (grad ? kGradCodeStride : kCodeStride) * sizeof(uint2));
    L.meta = o;        o = align256(o + P * sizeof(ProgMeta));
    L.order = o;       o = align256(o + P * sizeof(int32_t));
    L.class_count = o; o = align256(o + (kOrderClasses + 2) * sizeof(int32_t));
    L.part = o;        o = align256(o + P * C * sizeof(float));
    if (moments) {
        L.ystat = o;      o = align256(o + 4 * sizeof(double));
        L.ystat_part = o; o = align256(o + 2 * kSumwBlocks * sizeof(double));
        L.shift = o;      o = align256(o + P * sizeof(float));
        L.mom = o;        o = align256(o + P * C * 3 * sizeof(double));
    }
    if (grad) {
        L.gpart = o;   o = align256(o + P * C * GP_MAX_CONSTS * sizeof(float));
    }
    L.total = o;
    return L;
}

Workspace carve(void *base, const Layout &L, bool grad) {
    char *b = static_cast<char *>(base);
    Workspace w{};
    w.counters = reinterpret_cast<unsigned long long *>(b + L.counters);
    w.sumw = reinterpret_cast<double *>(b + L.sumw);
    w.sumw_part = reinterpret_cast<double *>(b + L.sumw_part);
    w.code = reinterpret_cast<uint2 *>(b + L.code);
    w.meta = reinterpret_cast<ProgMeta *>(b + L.meta);
    w.order = reinterpret_cast<int32_t *>(b + L.order);
    w.class_count = reinterpret_cast<int32_t *>(b + L.class_count);
    w.part = reinterpret_cast<float *>(b + L.part);
    if (L.mom) {
        w.ystat = reinterpret_cast<double *>(b + L.ystat);
        w.ystat_part = reinterpret_cast<double *>(b + L.ystat_part);
        w.shift = reinterpret_cast<float *>(b + L.shift);
        w.mom = reinterpret_cast<double *>(b + L.mom);
    }
    if (grad) w.gpart = reinterpret_cast<float *>(b + L.gpart);
    w.bytes = L.total;
    return w;
}

// The value of a function node whose operands are all constants, computed
// with the evaluator's own FP32 operations, so the folded constant is the
// very number the evaluator would produce on every row.
__device__ float fold_unary(int op, float a) {
    switch (op) {
        case GP_SQRT: return f_sqrt(a);
        case GP_LOG: return f_log(a);
        case GP_EXP: return f_exp(a);
        case GP_SIN:
        case GP_COS:
        case GP_TAN: {
            float t[1] = {a};
            trig_rows<1>(t, op - GP_SIN);
            return t[0];
        }
        case GP_ABS: return f_abs(a);
        case GP_NEG: return f_neg(a);
        case GP_INV: return f_inv(a);
        case GP_SQ: return f_sq(a);
        case GP_CUBE: return f_cube(a);
        case GP_CBRT: return f_cbrt(a);
        case GP_TANH: return f_tanh(a);
        case GP_ATAN: return f_atan(a);
        case GP_SINH: return f_sinh(a);
        default: return f_cosh(a);
    }
}

__device__ float fold_binary(int op, float l, float r) {
    switch (op) {
        case GP_ADD: return f_add(l, r);
        case GP_SUB: return f_sub(l, r);
        case GP_MUL: return f_mul(l, r);
        case GP_DIV: return f_div(l, r);
        case GP_MAX: return f_max(l, r);
        default: return f_min(l, r);
    }
}

// One warp per program, lane = node of a 32-node chunk of the prefix list.
// What a reverse scan with a stack does node after node comes from counts
// over the list instead, each a popc of warp ballots plus a carry per chunk:
//   - the stack height after node j (validity, high-water mark, and the
//     number of the stack slot in the compiled form) is the number of
//     terminals minus the number of binary nodes among the nodes >= j;
//   - the subtree of j ends at the first m > j whose height is below j's;
//   - a subtree is constant-only when no VAR lies in its range;
//   - a word's place is the number of words that the nodes > j emit.
// Only the values of constant-only subtrees (and, with a.shift, of every
// node at row 0) depend on one another; they are computed in rounds, each
// node once its operands are there.  Folding constant-only subtrees leaves
// every row's result bit-identical: the same FP32 operations run on the
// same inputs, once per program instead of once per row.
//
// Bound by latency: a program is about 1 KB of traffic and a few hundred
// dependent instructions.  One thread per program over local-memory arrays
// took 115 us for 1024 programs of 12 nodes (12.5 us now) and 310 us for
// 4096 of 19 nodes (34 us now).
constexpr int kCompileWarps = 4;
constexpr int kNodeChunks = (GP_MAX_LEN + 31) / 32;

struct CompileScratch {    // of one warp
    uint2 node[256];       // op | feat << 16, constant
    float val[256];        // value of a constant-only subtree (or at row 0)
    uint32_t hgt[65];      // bytes: stack height after node j; 0 from len on
    uint8_t end[256];      // one past the subtree of j
    uint8_t par[256];      // parent
    uint8_t vpre[257];     // VAR nodes before j
    uint8_t cpre[257];     // CONST nodes before j, at most GP_MAX_CONSTS
    uint8_t rdy[256];      // val is there
    // terminal: 1 = folded into its parent; binary: 0 / 1 R / 2 L folded;
    // any node: 3 = inside a constant-only subtree (dropped)
    uint8_t mode[256];
};

__global__ void __launch_bounds__(kCompileWarps * 32) compile_kernel(CompileArgs a) {
    __shared__ CompileScratch scratch[kCompileWarps];
    griddep_wait();
    griddep_launch();
    const int lane = threadIdx.x & 31;
    const int p = blockIdx.x * kCompileWarps + (threadIdx.x >> 5);
    if (p >= a.n_progs) return;  // the whole warp
    CompileScratch &S = scratch[threadIdx.x >> 5];
    const unsigned full = 0xffffffffu;
    const unsigned ge = full << lane, gt = ge & ~(1u << lane), lt = ~ge;
    const int off = a.offsets[p];
    const int len = a.offsets[p + 1] - off;
    uint2 *out = a.code + (size_t)p * (a.grad ? kGradCodeStride : kCodeStride);
    // 32-bit words: a node is only 4-byte aligned
    const uint32_t *prog = reinterpret_cast<const uint32_t *>(a.progs + off);
    const bool row0 = a.shift != nullptr;
    uint8_t *hgt = reinterpret_cast<uint8_t *>(S.hgt);

    // validity, from the end of the list: the failure met first by the
    // reverse scan is the one at the largest node
    int status = GP_PROG_OK;
    if (len < 1 || len > GP_MAX_LEN) status = GP_PROG_BAD_LENGTH;
    const int chunks = status == GP_PROG_OK ? (len + 31) >> 5 : 0;
    int carry = 0, hw = 0, n_consts = 0;
    for (int c = chunks - 1; c >= 0; --c) {
        const int j = c * 32 + lane;
        const bool in = j < len;
        const uint2 nd = in ? make_uint2(prog[2 * j], prog[2 * j + 1]) : make_uint2(0u, 0u);
        const int op = (int16_t)(nd.x & 0xffffu), feat = (int16_t)(nd.x >> 16);
        const int ar = in ? op_arity(op) : 1;  // past the end: height unchanged
        const unsigned leaf = __ballot_sync(full, ar == 0), bin = __ballot_sync(full, ar == 2);
        const int h = carry + __popc(leaf & ge) - __popc(bin & ge);
        const int before = carry + __popc(leaf & gt) - __popc(bin & gt);
        int code = GP_PROG_OK;
        if (in) {
            if (ar < 0) code = GP_PROG_BAD_OP;
            else if (op == GP_VAR && (feat < 0 || feat >= a.n_feat)) code = GP_PROG_BAD_FEATURE;
            else if (before < ar) code = GP_PROG_UNDERFLOW;
            S.node[j] = nd;
            hgt[j] = (uint8_t)h;
            hw = max(hw, h);
        }
        const unsigned bad = __ballot_sync(full, code != GP_PROG_OK);
        if (bad) {
            status = __shfl_sync(full, code, 31 - __clz(bad));
            break;
        }
        n_consts += __popc(__ballot_sync(full, in && op == GP_CONST));
        carry += __popc(leaf) - __popc(bin);
    }
    hw = __reduce_max_sync(full, hw);
    if (status == GP_PROG_OK && carry != 1) status = GP_PROG_LEFTOVER;
    if (status == GP_PROG_OK && hw > GP_MAX_STACK) status = GP_PROG_TOO_DEEP;
    if (a.out_prog_status && lane == 0) a.out_prog_status[p] = status;
    if (status != GP_PROG_OK) {
        if (lane == 0) {
            if (row0) a.shift[p] = 0.0f;
            out[0] = make_uint2(make_ins(OP_END, 0, 0), 0u);
            a.meta[p] = ProgMeta{1, status, 0, 0, 0};
            atomicOr(a.dev_status, GP_DEV_BAD_PROGRAM);
        }
        return;
    }
    // heights of 0 past the end stop the search below (heights are 1..20)
    if (lane < 4) hgt[len + lane] = 0;
    __syncwarp();

    // subtree ends: the first byte after j below j's height, four at a time;
    // prefix counts of VAR and CONST; the terminals' values
    int vcar = 0, ccar = 0;
    for (int c = 0; c < chunks; ++c) {
        const int j = c * 32 + lane;
        const bool in = j < len;
        const uint2 nd = in ? S.node[j] : make_uint2(GP_NUM_OPS, 0u);
        const int op = (int16_t)(nd.x & 0xffffu);
        const unsigned vm = __ballot_sync(full, op == GP_VAR), cm = __ballot_sync(full, op == GP_CONST);
        if (in) {
            S.vpre[j] = (uint8_t)(vcar + __popc(vm & lt));
            S.cpre[j] = (uint8_t)min(ccar + __popc(cm & lt), GP_MAX_CONSTS);
            int q = (j + 1) >> 2;
            const uint32_t h4 = (uint32_t)hgt[j] * 0x01010101u;
            uint32_t m = __vcmpltu4(S.hgt[q], h4) & (0xffffffffu << (((j + 1) & 3) * 8));
            while (m == 0u) m = __vcmpltu4(S.hgt[++q], h4);
            S.end[j] = (uint8_t)(q * 4 + ((__ffs(m) - 1) >> 3));
            S.mode[j] = 0;
            S.rdy[j] = op <= GP_VAR;
            if (op == GP_CONST) S.val[j] = __uint_as_float(nd.y);
            if (op == GP_VAR) S.val[j] = row0 ? a.X[(int64_t)(int16_t)(nd.x >> 16) * a.ld] : 0.0f;
        }
        vcar += __popc(vm);
        ccar += __popc(cm);
    }
    if (lane == 0) {
        S.vpre[len] = (uint8_t)vcar;
        S.cpre[len] = (uint8_t)min(ccar, GP_MAX_CONSTS);
        S.par[0] = 0;
    }
    __syncwarp();

    // constant-only subtrees (k8, bit c: this lane's node of chunk c; the
    // gradient form folds no function), the parents, and the function
    // values still to compute
    uint32_t k8 = 0u, todo = 0u;
    for (int c = 0; c < chunks; ++c) {
        const int j = c * 32 + lane;
        if (j >= len) break;
        const int ar = op_arity((int16_t)(S.node[j].x & 0xffffu));
        const bool k = S.vpre[S.end[j]] == S.vpre[j] && (ar == 0 || !a.grad);
        k8 |= (uint32_t)k << c;
        if (ar > 0) {
            S.par[j + 1] = (uint8_t)j;
            if (ar == 2) S.par[S.end[j + 1]] = (uint8_t)j;
            todo |= (uint32_t)(k || row0) << c;
        }
    }
    __syncwarp();
    while (__any_sync(full, todo != 0u)) {
        // from the last chunk on: operands come after their node
        for (int c = chunks - 1; c >= 0; --c) {
            const int j = c * 32 + lane;
            bool go = (todo >> c) & 1u;
            int op = 0, rc = 0;
            if (go) {
                op = (int16_t)(S.node[j].x & 0xffffu);
                rc = op_arity(op) == 2 ? S.end[j + 1] : j + 1;
                go = S.rdy[j + 1] && S.rdy[rc];
            }
            if (!__any_sync(full, go)) continue;
            if (go) {
                S.val[j] = op_arity(op) == 1 ? fold_unary(op, S.val[j + 1])
                                             : fold_binary(op, S.val[j + 1], S.val[rc]);
                todo &= ~(1u << c);
            }
            __syncwarp();
            if (go) S.rdy[j] = 1;
            __syncwarp();
        }
    }
    if (row0 && lane == 0) {
        // a non-finite value would poison every shifted row; 0 is as good
        // as any other finite shift
        const float k0 = S.val[0];
        a.shift[p] = isfinite(k0) ? k0 : 0.0f;
    }
    // drop the inside of every maximal constant-only subtree: the nodes
    // whose parent is constant-only (its root becomes one constant, a
    // terminal); then fold terminal children of binary nodes (prefer the
    // right one).  kst: the constant-only flag per node, for the others' use
    // (rdy is free now)
    for (int c = 0; c < chunks; ++c) {
        const int j = c * 32 + lane;
        if (j < len) S.rdy[j] = (k8 >> c) & 1u;
    }
    uint8_t *kon = S.rdy;
    __syncwarp();
    for (int c = 0; c < chunks; ++c) {
        const int j = c * 32 + lane;
        if (j >= len) break;
        const int op = (int16_t)(S.node[j].x & 0xffffu);
        if (kon[j]) {
            if (j > 0 && kon[S.par[j]]) S.mode[j] = 3;
            continue;
        }
        // max and min take both operands from the stack
        if (op_arity(op) != 2 || op > GP_DIV) continue;
        const int lc = j + 1, rc = S.end[lc];
        const int opl = (int16_t)(S.node[lc].x & 0xffffu), opr = (int16_t)(S.node[rc].x & 0xffffu);
        if (opr <= GP_VAR || kon[rc]) {
            S.mode[rc] = 1;
            S.mode[j] = 1;
        } else if (opl <= GP_VAR || kon[lc]) {
            S.mode[lc] = 1;
            S.mode[j] = 2;
        }
    }
    __syncwarp();

    // emit, from the end of the list
    int n = 0, sp_car = 0, depth = 0;
    bool ext = false;  // an instruction of the extended classes was emitted
    // more than two columns: each column read names the next one; the chunk's
    // last is completed when a later chunk emits one (at: its place, -1 none)
    const bool linked = a.n_feat > 2;
    int link_at = -1;
    uint32_t first_feat = 0u;
    for (int c = chunks - 1; c >= 0; --c) {
        const int j = c * 32 + lane;
        const bool in = j < len;
        const uint2 nd = in ? S.node[j] : make_uint2(0u, 0u);
        const bool k = in && kon[j];
        const int op = k ? GP_CONST : (int16_t)(nd.x & 0xffffu);
        const int ar = op_arity(op);
        const int mode = in ? S.mode[j] : 3;
        const bool emit = mode != 3 && !(ar == 0 && mode);
        const unsigned up = __ballot_sync(full, emit && ar == 0);
        const unsigned down = __ballot_sync(full, emit && ar == 2 && mode == 0);
        const int sp = sp_car + __popc(up & gt) - __popc(down & gt);  // before the word
        depth = max(depth, sp_car + __popc(up & ge) - __popc(down & ge));
        uint2 word = make_uint2(0u, 0u);
        // gradient form: a marker word before the word when one of its
        // operands holds constants (j_top: the node whose value is the top
        // operand, j_other: the other operand's node; -1 where the partial
        // derivative is 1 and leaves the tangents as they are)
        int j_top = -1, j_other = -1;
        bool fresh = false, column = false;
        if (emit && ar == 0) {
            const bool x = op == GP_VAR;
            const uint32_t feat = x ? nd.x >> 16 : 0u;
            const bool spill = sp > 0;  // the old top goes to slot sp-1
            const uint32_t w = (spill ? (x ? OP_PUSH_X_SP : OP_PUSH_C_SP) : (x ? OP_PUSH_X : OP_PUSH_C)) |
                               (feat == 1u && !linked ? kOpCol1 : 0u);
            word = make_uint2(make_ins(w, spill ? sp - 1 : 0, feat), k ? __float_as_uint(S.val[j]) : nd.y);
            column = x;
            if (!x) {  // the constant's own tangent starts at 1
                j_other = j;
                fresh = true;
            }
        } else if (emit && ar == 1) {
            const bool e = op > GP_INV;  // extended function: its number in the feature field
            // the loop of class 0 does not run tan (the gradient's classes go by
            // the extended functions alone)
            ext |= e || (op == GP_TAN && !a.grad);
            word.x = e ? make_ins(OP_EXT1, 0, (uint32_t)(op - GP_SQ))
                       : make_ins(OP_SQRT + (op - GP_SQRT), 0, 0);
            j_top = j + 1;
        } else if (emit) {
            // add, sub, mul, div, max, min
            const int b = op <= GP_DIV ? op - GP_ADD : 4 + (op - GP_MAX);
            const int lc = j + 1, rc = S.end[lc];
            if (mode == 0) {
                // right operand in slot sp-2, left operand is t (add: both
                // partials 1; sub: 1 for t)
                ext |= b >= 4;
                word.x = b >= 4 ? make_ins(OP_EXT2, sp - 2, (uint32_t)(b - 4))
                                : make_ins(OP_ADD_S + (uint32_t)b, sp - 2, 0);
                if (b != 0) {
                    j_top = b == 1 ? -1 : lc;
                    j_other = rc;
                }
            } else {
                const int tj = (mode == 1) ? rc : lc;  // the inline terminal
                const uint2 t = S.node[tj];
                const bool x = !kon[tj];               // X or C variant
                const uint32_t feat = x ? t.x >> 16 : 0u;
                // right terminal: t = op(t, u); left terminal: t = op(u, t)
                // (add, and sub with the terminal on the right, leave the
                // top's tangents as they are)
                const uint32_t fwd = b == 0 ? OP_ADD_X : b == 1 ? OP_SUB_X : b == 2 ? OP_MUL_X : OP_DIV_X;
                const uint32_t rev = b == 0 ? OP_ADD_X : b == 1 ? OP_RSUB_X : b == 2 ? OP_MUL_X : OP_RDIV_X;
                const uint32_t w = (((mode == 1) ? fwd : rev) + (x ? 0u : 1u)) |
                                   (feat == 1u && !linked ? kOpCol1 : 0u);
                column = x;
                word = make_uint2(make_ins(w, 0, feat), x ? t.y : __float_as_uint(S.val[tj]));
                j_top = (b == 0 || (b == 1 && mode == 1)) ? -1 : (mode == 1) ? lc : rc;
                j_other = tj;
                fresh = !x;
            }
        }
        uint2 mark = make_uint2(0u, 0u);
        if (a.grad && emit) {
            const uint32_t tlo = j_top >= 0 ? S.cpre[j_top] : 0u;
            const uint32_t thi = j_top >= 0 ? S.cpre[S.end[j_top]] : 0u;
            const uint32_t olo = j_other >= 0 ? S.cpre[j_other] : 0u;
            const uint32_t ohi = j_other >= 0 ? S.cpre[S.end[j_other]] : 0u;
            if (tlo != thi || olo != ohi) {
                // the two common shapes get tails of their own in the fast loop
                const uint32_t shape = (thi == tlo + 1 && olo == ohi) ? 1u
                                     : (tlo == thi && ohi == olo + 1 && fresh) ? 2u : 0u;
                mark = make_uint2(kGradMark | (shape << 8),
                                  tlo | (thi << 5) | (olo << 10) | (ohi << 15) | ((fresh ? 1u : 0u) << 20));
            }
        }
        const unsigned words = __ballot_sync(full, emit), marks = __ballot_sync(full, mark.x != 0u);
        int at = n + __popc(words & gt) + __popc(marks & gt) + (mark.x != 0u);
        if (linked) {
            const unsigned cols = __ballot_sync(full, column);
            const uint32_t feat = word.x >> 16;
            const int succ = 31 - __clz(cols & lt);  // the lane emitted next; -1: a later chunk's
            const uint32_t next = __shfl_sync(full, feat, succ & 31);
            if (column && succ >= 0) word.y = next;
            if (cols) {
                const int head = 31 - __clz(cols), tail = __ffs(cols) - 1;
                const uint32_t f = __shfl_sync(full, feat, head);
                if (link_at < 0) first_feat = f;
                else if (lane == 0) out[link_at].y = f;
                link_at = __shfl_sync(full, at, tail);
            }
        }
        if (emit) {
            if (mark.x) out[at - 1] = mark;
            out[at] = word;
        }
        __syncwarp();  // (out[link_at] is completed by another lane)
        n += __popc(words) + __popc(marks);
        sp_car += __popc(up) - __popc(down);
    }
    depth = __reduce_max_sync(full, depth);
    ext = __any_sync(full, ext);
    if (lane == 0) {
        if (link_at >= 0) out[link_at].y = out[link_at].x >> 16;  // no next: its own
        out[n] = make_uint2(make_ins(OP_END, 0, 0), first_feat);
        a.meta[p] = ProgMeta{n + 1, GP_PROG_OK, (int16_t)depth, (int16_t)(ext ? 1 : 0), n_consts};
    }
}

cudaError_t launch_compile(const CompileArgs &a, cudaStream_t st) {
    if (a.n_progs <= 0) return cudaSuccess;
    const int grid = (a.n_progs + kCompileWarps - 1) / kCompileWarps;
    return launch_chained(compile_kernel, grid, kCompileWarps * 32, 0, st, a);
}

// Counting sort of program ids: key = class * 256 + (256 - n_ins), so the
// classes follow one another (0, 1, 2, 3) and, inside a class, longer programs
// come first (longest-processing-time order for the dynamic work queue).
// mode 0: the evaluator's classes (stack depth, extended functions); mode
// 1: the gradient's buckets (constants, stack depth), whose programs with
// their marker words may exceed 256 words (those share the first key).
// Invalid programs (n_ins = 1) land at the end of class 0.  Order inside
// one key is arbitrary; results do not depend on it.  One block: the counts
// and the scan of the 1280 keys stay in shared memory (a serial scan of the
// keys by one thread took 27 us; 4.7 us now for 1024 programs, 7.4 for 4096).  It also clears the work-queue
// counters of the launches that follow and, without weights, writes the
// total weight.
constexpr int kOrderBins = kOrderClasses * 256;
constexpr int kOrderThreads = 1024;
constexpr int kBinsPerThread = (kOrderBins + kOrderThreads - 1) / kOrderThreads;

__device__ __forceinline__ int order_key(const ProgMeta &m, int mode) {
    const int cls = mode == 0 ? prog_class(m.depth, m.ext) : grad_bucket(m.n_consts, m.depth, m.ext);
    return cls * 256 + (256 - min(m.n_ins, 256));
}

__global__ void __launch_bounds__(kOrderThreads) order_kernel(const ProgMeta *meta, int n_progs,
                                                              int32_t *order, int32_t *class_count,
                                                              int mode, int edge,
                                                              unsigned long long *counters,
                                                              double *sumw, int64_t n_rows) {
    __shared__ int cursor[kOrderThreads * kBinsPerThread + 1];  // counts, then first positions
    __shared__ int warp_sum[kOrderThreads / 32];
    griddep_wait();
    griddep_launch();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t < 8 && counters) counters[t] = 0ull;
    if (t == 0 && sumw) *sumw = (double)n_rows;
#pragma unroll
    for (int q = 0; q < kBinsPerThread; ++q) cursor[q * kOrderThreads + t] = 0;
    __syncthreads();
    for (int p = t; p < n_progs; p += kOrderThreads) atomicAdd(&cursor[order_key(meta[p], mode)], 1);
    __syncthreads();
    int v[kBinsPerThread], run = 0;
#pragma unroll
    for (int q = 0; q < kBinsPerThread; ++q) {
        v[q] = cursor[t * kBinsPerThread + q];
        run += v[q];
    }
    int x = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    int before = x - run;
    for (int w = 0; w < warp; ++w) before += warp_sum[w];
#pragma unroll
    for (int q = 0; q < kBinsPerThread; ++q) {
        cursor[t * kBinsPerThread + q] = before;
        before += v[q];
    }
    __syncthreads();
    if (t < kOrderClasses)
        class_count[t] = (t + 1 < kOrderClasses ? cursor[(t + 1) * 256] : n_progs) - cursor[t * 256];
    // class-0 programs longer than edge: keys 0 .. 255 - edge (n_ins > edge)
    if (t == 0) {
        class_count[kOrderClasses] = edge > 0 ? cursor[256 - edge] : 0;
        class_count[kOrderClasses + 1] = 0;
    }
    __syncthreads();
    for (int p = t; p < n_progs; p += kOrderThreads)
        order[atomicAdd(&cursor[order_key(meta[p], mode)], 1)] = p;
}

cudaError_t launch_order(const ProgMeta *meta, int n_progs, int32_t *order, int32_t *class_count,
                         cudaStream_t st, unsigned long long *counters, int mode, int edge,
                         double *sumw, int64_t n_rows) {
    return launch_chained(order_kernel, 1, kOrderThreads, 0, st, meta, n_progs, order, class_count, mode,
                          edge, counters, sumw, n_rows);
}

// FP64 sums over the rows with a fixed partition: block b sums rows
// [b*span, (b+1)*span) with a fixed per-thread stride and a fixed tree; the
// block that finishes last (a ticket, which it resets) adds the block sums
// with the same tree.  One launch per sum: as a second launch in which one
// thread added the 512 block sums one after another, the last step took 30
// us, 52 us for a pair of sums (the whole kernel now: 13 us and 23 us for 1M
// rows).
constexpr int kSumThreads = 256;

// 1024 rows a block at least (4 per thread), kSumwBlocks blocks at most
static inline int sum_blocks(int64_t n_rows) {
    return (int)std::min<int64_t>((n_rows + 1023) / 1024, kSumwBlocks);
}

// K sums per thread -> red[k][0]; every thread of the block calls it
template <int K>
__device__ __forceinline__ void block_tree(double (&v)[K], double (&red)[K][kSumThreads]) {
    const int t = threadIdx.x;
#pragma unroll
    for (int k = 0; k < K; ++k) red[k][t] = v[k];
    __syncthreads();
    for (int h = kSumThreads / 2; h > 0; h >>= 1) {
        if (t < h)
#pragma unroll
            for (int k = 0; k < K; ++k) red[k][t] += red[k][t + h];
        __syncthreads();
    }
}

// the block sums of the whole grid into red[k][0] of the block that comes
// last; false in every other block
template <int K>
__device__ bool grid_tree(double (&v)[K], double (&red)[K][kSumThreads], double *part,
                          unsigned long long *ticket) {
    __shared__ bool last;
    const int t = threadIdx.x;
    block_tree<K>(v, red);
    if (t == 0) {
#pragma unroll
        for (int k = 0; k < K; ++k) part[K * blockIdx.x + k] = red[k][0];
        __threadfence();
        last = atomicAdd(ticket, 1ull) + 1ull == (unsigned long long)gridDim.x;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    double s[K];
#pragma unroll
    for (int k = 0; k < K; ++k) s[k] = 0.0;
    for (int b = t; b < (int)gridDim.x; b += kSumThreads)
#pragma unroll
        for (int k = 0; k < K; ++k) s[k] += __ldcg(part + K * b + k);
    block_tree<K>(s, red);
    if (t == 0) *ticket = 0ull;
    return true;
}

__global__ void __launch_bounds__(kSumThreads) sumw_kernel(const float *__restrict__ w, int64_t n_rows,
                                                           double *part, double *sumw,
                                                           unsigned long long *ticket) {
    __shared__ double red[1][kSumThreads];
    griddep_wait();
    griddep_launch();
    const int64_t span = (n_rows + gridDim.x - 1) / gridDim.x;
    const int64_t r0 = (int64_t)blockIdx.x * span;
    const int64_t r1 = min(n_rows, r0 + span);
    double s[1] = {0.0};
#pragma unroll 4
    for (int64_t r = r0 + threadIdx.x; r < r1; r += kSumThreads) s[0] += (double)w[r];
    if (grid_tree<1>(s, red, part, ticket) && threadIdx.x == 0) *sumw = red[0][0];
}

cudaError_t launch_sumw(const float *w, int64_t n_rows, double *part, double *sumw,
                        unsigned long long *ticket, cudaStream_t st) {
    return launch_chained(sumw_kernel, sum_blocks(n_rows), kSumThreads, 0, st, w, n_rows, part, sumw,
                          ticket);
}

// Statistics of y for the correlation fitness: phase 0 sums w y and sets
// ybar = sum w y / sum w (FP64) and its float rounding; phase 1 sums
// w yc and w yc^2 with yc = fl(y - fl(ybar)), the very values the
// evaluator forms.
template <int PHASE>
__global__ void __launch_bounds__(kSumThreads) ystats_kernel(const float *__restrict__ y,
                                                             const float *__restrict__ w,
                                                             int64_t n_rows, const double *sumw,
                                                             double *ystat, double *part,
                                                             unsigned long long *ticket) {
    constexpr int K = PHASE + 1;
    __shared__ double red[K][kSumThreads];
    griddep_wait();
    griddep_launch();
    const int64_t span = (n_rows + gridDim.x - 1) / gridDim.x;
    const int64_t r0 = (int64_t)blockIdx.x * span;
    const int64_t r1 = min(n_rows, r0 + span);
    const float ybar = PHASE ? (float)ystat[3] : 0.0f;
    double s[K];
#pragma unroll
    for (int k = 0; k < K; ++k) s[k] = 0.0;
#pragma unroll 4
    for (int64_t r = r0 + threadIdx.x; r < r1; r += kSumThreads) {
        const double wr = w ? (double)w[r] : 1.0;
        if (PHASE == 0) {
            s[0] += wr * (double)y[r];
        } else {
            const double yc = (double)__fsub_rn(y[r], ybar);
            s[0] += wr * yc;
            s[K - 1] += wr * yc * yc;
        }
    }
    if (grid_tree<K>(s, red, part, ticket) && threadIdx.x == 0) {
        if (PHASE == 0) {
            const double yb = red[0][0] / *sumw;
            ystat[0] = yb;
            ystat[3] = (double)(float)yb;
        } else {
            ystat[1] = red[0][0];
            ystat[2] = red[K - 1][0];
        }
    }
}

cudaError_t launch_ystats(const float *y, const float *w, int64_t n_rows, const double *sumw,
                          double *part, double *ystat, unsigned long long *ticket, cudaStream_t st) {
    const int grid = sum_blocks(n_rows);
    const cudaError_t e =
        launch_chained(ystats_kernel<0>, grid, kSumThreads, 0, st, y, w, n_rows, sumw, ystat, part, ticket);
    if (e != cudaSuccess) return e;
    return launch_chained(ystats_kernel<1>, grid, kSumThreads, 0, st, y, w, n_rows, sumw, ystat, part,
                          ticket);
}

}  // namespace gpk
