// gp_grad.cu -- gradients of fitness with respect to the ephemeral
// constants (forward mode), and one Adam step on the constants.  Neither
// has a counterpart in the paper; they serve constant tuning between
// generations.
//
// Forward mode on the compiled stack form of the evaluator
// (gp_internal.cuh), in its gradient variant: no constant-only subtree is
// folded, and a marker word precedes every word whose operands hold
// constants, naming the constants under each operand (they form contiguous
// ranges of the prefix-order numbering).  Each row carries one tangent per
// constant, dt[k] = d(value holding c_k)/d(c_k): a pushed constant starts
// at 1, and a marked word multiplies the tangents under each operand by
// its partial derivative with respect to that operand, so after the root
// dt[k] is d(program)/d(c_k).  Every constant is a leaf used once, so a
// row costs the forward pass plus one multiply per (constant, ancestor)
// pair -- no tape and no reverse sweep: the values and tangents live in
// registers and a few shared-memory slots per row.
//
// A block takes one (program, row chunk) item; its warps run the program
// over their own sub-tiles of 128 rows (4 per lane) with the evaluator's
// fast loop (the same FP32 operations on every row, so the fitness is
// gp_evaluate's but for the order of its sums) in its gradient variant, which
// hands the words it does not run back to grad_word.  The loss derivative per
// row times the tangents gives each constant's share.  Programs are bucketed by what their stack and
// constants need of shared memory (grad_bucket), one launch per bucket.
// Per-lane sums are FP32 (the loss Kahan-compensated), warp sums
// fixed-order, chunk sums FP64 in a fixed order (gp_reduce.cu).
//
// Bound by instruction issue and by fetching 130 KB of code a word here and a
// word there (61% of the issue slots taken at 32 warps per SM, 1 cycle in 5
// of a warp waiting for instructions), hence as many warps per SM as 64
// registers allow: with all of a Pagie-1 population's programs at 16
// warps the gradient takes 10.9 ms, at 24 warps 9.3 and as it is 8.3 ms (2048
// programs, depth 4-10, 262144 rows).  What the packed shared memory, column
// reads in the loop (with more than two columns; the next column's rows are
// prefetched as in the evaluator) and launches that overlap at their
// edges gave: those 2048 programs 9.18 -> 8.27 ms; 1024 programs, depth 3-7, 28
// columns x 200000 rows 1.17 -> 1.10 ms; 512 programs x 1000 rows 94 -> 60 us.
// The rows of a lane, the order of its sums and which words run where are part
// of the results: a gradient that cancels out is rounding alone, and Adam's
// first steps divide it by its own size.
#include <atomic>

#include "gp_internal.cuh"
#include "gp_interp.cuh"

namespace gpk {

namespace {

__device__ __forceinline__ float sgnf(float x) {
    return x > 0.0f ? 1.0f : (x < 0.0f ? -1.0f : 0.0f);
}

// d loss / d p of one row (the metric readings of Sec. III-C3)
__device__ __forceinline__ float g_dloss(int metric, float p, float y) {
    if (metric == GP_MAE) return sgnf(__fsub_rn(p, y));
    if (metric == GP_LOGLOSS) {
        float s;
        if (p >= 0.0f) {
            s = __fdiv_rn(1.0f, __fadd_rn(1.0f, expf(-p)));
        } else {
            const float e = expf(p);
            s = __fdiv_rn(e, __fadd_rn(1.0f, e));
        }
        return __fsub_rn(s, y);
    }
    return __fmul_rn(2.0f, __fsub_rn(p, y));
}

// derivative of a unary word at input u with output v (the protected
// operators have derivative 0 on their protected branch)
__device__ __forceinline__ float d_unary(uint32_t op, uint32_t ext, float u, float v) {
    switch (op) {
    case OP_SQRT: return (u == 0.0f) ? 0.0f : __fdiv_rn(sgnf(u), __fmul_rn(2.0f, v));
    case OP_LOG: return fabsf(u) < kThr ? 0.0f : __frcp_rn(u);
    case OP_EXP: return v;
    case OP_SIN: return cosf(u);
    case OP_COS: return -sinf(u);
    case OP_TAN: return __fadd_rn(1.0f, __fmul_rn(v, v));
    case OP_ABS: return sgnf(u);
    case OP_NEG: return -1.0f;
    case OP_INV: return fabsf(u) < kThr ? 0.0f : -__fmul_rn(v, v);
    default:  // OP_EXT1
        switch (ext) {
        case EXT_SQ: return __fmul_rn(2.0f, u);
        case EXT_CUBE: return __fmul_rn(3.0f, __fmul_rn(u, u));
        case EXT_CBRT: return (u == 0.0f) ? 0.0f : __frcp_rn(__fmul_rn(3.0f, __fmul_rn(v, v)));
        case EXT_TANH: return __fsub_rn(1.0f, __fmul_rn(v, v));
        case EXT_ATAN: return __frcp_rn(__fadd_rn(1.0f, __fmul_rn(u, u)));
        case EXT_SINH: return coshf(u);
        default: return sinhf(u);  // EXT_COSH
        }
    }
}

// the extended unary functions of one row (the evaluator's, so the forward
// values are its values)
__device__ __forceinline__ float f_ext1(uint32_t fn, float x) {
    switch (fn) {
    case EXT_SQ: return f_sq(x);
    case EXT_CUBE: return f_cube(x);
    case EXT_CBRT: return f_cbrt(x);
    case EXT_TANH: return f_tanh(x);
    case EXT_ATAN: return f_atan(x);
    case EXT_SINH: return f_sinh(x);
    default: return f_cosh(x);
    }
}

}  // namespace

// The tangents of a lane's four rows: one float4 per constant k at the
// shared-memory address db + k * 512.  They are read and written only by
// volatile asm statements (here and in the fast loop, which declares no
// memory clobber), so their order is kept.
__device__ __forceinline__ float4 tan_load(uint32_t a) {
    float4 d;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(d.x), "=f"(d.y), "=f"(d.z), "=f"(d.w)
                 : "r"(a));
    return d;
}
__device__ __forceinline__ void tan_store(uint32_t a, float4 d) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(d.x), "f"(d.y),
                 "f"(d.z), "f"(d.w)
                 : "memory");
}

// One word of the gradient form that the fast loop handed back (a marked
// word it does not run or whose fast path gave up, or an unmarked word it
// does not run): its value with the evaluator's operations and, after a
// marker (mk != 0), its partial derivatives with respect to the top
// operand t (pt) and the other operand (po), applied to the tangents of
// the constants under each (kGradMark).  Four rows per lane; the stack
// slot of this lane's rows is one float4 (sb + slot * 512 bytes), the
// tangent of constant k one float4 at db + k * 512.
// The gradient's four rows of a lane as pairs: always consecutive, so that
// which rows a lane's sums hold does not depend on the alignment (the
// gradient of a constant that cancels out is rounding alone, and an Adam
// step divides it by its own size); with vec 16-byte loads, else 4-byte ones,
// rows past p[last] 0.
__device__ __forceinline__ void load_quad(uint64_t (&v)[2], const float *__restrict__ p, bool vec,
                                          int last) {
    if (vec) {
        const ulonglong2 f = __ldg(reinterpret_cast<const ulonglong2 *>(p));
        v[0] = f.x;
        v[1] = f.y;
    } else {
        float f[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) f[j] = (j <= last) ? __ldg(p + j) : 0.0f;
        v[0] = pack2(f[0], f[1]);
        v[1] = pack2(f[2], f[3]);
    }
}

template <bool XREG>
__device__ __forceinline__ void grad_word(uint32_t w, float c, uint32_t mk, uint64_t (&tp)[2],
                                          const uint64_t (&x0)[2], const uint64_t (&x1)[2],
                                          const float *__restrict__ xc, int64_t ld, bool packed,
                                          int last, uint32_t sb, uint32_t db) {
    constexpr int R = 4;
    float t[R];
    unpack2(tp[0], t[0], t[1]);
    unpack2(tp[1], t[2], t[3]);
    const uint32_t opc = w & 31u;
    const uint32_t fn = (w >> 16) & 7u;
    const uint32_t sa = sb + ((w >> 8) & 255u) * 512u;
    // the other operand: a stack slot (S forms, EXT2), a column (X forms,
    // PUSH_X), else the word's constant
    float o[R];
    const bool from_slot = (opc >= OP_ADD_S && opc <= OP_DIV_S) || opc == OP_EXT2;
    const bool from_col = opc == OP_PUSH_X || opc == OP_PUSH_X_SP ||
                          (opc >= OP_ADD_X && opc <= OP_RDIV_X && ((opc - OP_ADD_X) & 1u) == 0u);
    if (from_slot) {
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(o[0]), "=f"(o[1]), "=f"(o[2]), "=f"(o[3])
                     : "r"(sa));
    } else if (from_col) {
        const int feat = (int)(w >> 16);
        uint64_t op[2];
        if (XREG) {
            op[0] = feat ? x1[0] : x0[0];
            op[1] = feat ? x1[1] : x0[1];
        } else {
            load_quad(op, xc + (int64_t)feat * ld, packed, last);
        }
        unpack2(op[0], o[0], o[1]);
        unpack2(op[1], o[2], o[3]);
    } else {
#pragma unroll
        for (int j = 0; j < R; ++j) o[j] = c;
    }
    if (opc == OP_PUSH_X_SP || opc == OP_PUSH_C_SP)
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(sa), "f"(t[0]), "f"(t[1]),
                     "f"(t[2]), "f"(t[3])
                     : "memory");
    float v[R];
#define GP_ROWS(stmt) _Pragma("unroll") for (int j = 0; j < R; ++j) { stmt; }
    switch (opc) {
    case OP_ADD_S: case OP_ADD_X: case OP_ADD_C: GP_ROWS(v[j] = f_add(t[j], o[j])) break;
    case OP_SUB_S: case OP_SUB_X: case OP_SUB_C: GP_ROWS(v[j] = f_sub(t[j], o[j])) break;
    case OP_RSUB_X: case OP_RSUB_C: GP_ROWS(v[j] = f_sub(o[j], t[j])) break;
    case OP_MUL_S: case OP_MUL_X: case OP_MUL_C: GP_ROWS(v[j] = f_mul(t[j], o[j])) break;
    case OP_DIV_S: case OP_DIV_X: case OP_DIV_C: GP_ROWS(v[j] = f_div(t[j], o[j])) break;
    case OP_RDIV_X: case OP_RDIV_C: GP_ROWS(v[j] = f_div(o[j], t[j])) break;
    case OP_SQRT: GP_ROWS(v[j] = f_sqrt(t[j])) break;
    case OP_LOG: GP_ROWS(v[j] = f_log(t[j])) break;
    case OP_EXP: GP_ROWS(v[j] = f_exp(t[j])) break;
    case OP_SIN: case OP_COS: case OP_TAN:
        GP_ROWS(v[j] = t[j])
        trig_rows<R>(v, (int)(opc - OP_SIN));
        break;
    case OP_ABS: GP_ROWS(v[j] = f_abs(t[j])) break;
    case OP_NEG: GP_ROWS(v[j] = f_neg(t[j])) break;
    case OP_INV: GP_ROWS(v[j] = f_inv(t[j])) break;
    case OP_EXT1: GP_ROWS(v[j] = f_ext1(fn, t[j])) break;
    case OP_EXT2:
        if (fn == EXT_MAX) { GP_ROWS(v[j] = f_max(t[j], o[j])) }
        else { GP_ROWS(v[j] = f_min(t[j], o[j])) }
        break;
    default: GP_ROWS(v[j] = o[j]) break;  // the pushes (OP_END never gets here)
    }
    if (mk != 0u) {
        float pt[R], po[R];
        GP_ROWS(pt[j] = 1.0f; po[j] = 1.0f)
        switch (opc) {
        case OP_SUB_S: case OP_SUB_X: case OP_SUB_C: GP_ROWS(po[j] = -1.0f) break;
        case OP_RSUB_X: case OP_RSUB_C: GP_ROWS(pt[j] = -1.0f) break;
        case OP_MUL_S: case OP_MUL_X: case OP_MUL_C: GP_ROWS(pt[j] = o[j]; po[j] = t[j]) break;
        case OP_DIV_S: case OP_DIV_X: case OP_DIV_C:
            GP_ROWS(const bool p0 = fabsf(o[j]) < kThr;
                    pt[j] = p0 ? 0.0f : __frcp_rn(o[j]);
                    po[j] = p0 ? 0.0f : -__fdiv_rn(v[j], o[j]))
            break;
        case OP_RDIV_X: case OP_RDIV_C:
            GP_ROWS(const bool p0 = fabsf(t[j]) < kThr;
                    pt[j] = p0 ? 0.0f : -__fdiv_rn(v[j], t[j]);
                    po[j] = p0 ? 0.0f : __frcp_rn(t[j]))
            break;
        case OP_EXT2:
            GP_ROWS(const bool left = (fn == EXT_MAX) ? (t[j] > o[j] || t[j] != t[j])
                                                      : (t[j] < o[j] || t[j] != t[j]);
                    pt[j] = left ? 1.0f : 0.0f; po[j] = left ? 0.0f : 1.0f)
            break;
        case OP_SQRT: case OP_LOG: case OP_EXP: case OP_SIN: case OP_COS: case OP_TAN:
        case OP_ABS: case OP_NEG: case OP_INV: case OP_EXT1:
            GP_ROWS(pt[j] = d_unary(opc, fn, t[j], v[j]))
            break;
        default: break;  // add and the pushes: both partials 1
        }
        const int tlo = (int)(mk & 31u), thi = (int)((mk >> 5) & 31u);
        const int olo = (int)((mk >> 10) & 31u), ohi = (int)((mk >> 15) & 31u);
        const bool fresh = ((mk >> 20) & 1u) != 0u;
        for (int k = tlo; k < thi; ++k) {
            float4 d = tan_load(db + (uint32_t)k * 512u);
            d.x = __fmul_rn(d.x, pt[0]);
            d.y = __fmul_rn(d.y, pt[1]);
            d.z = __fmul_rn(d.z, pt[2]);
            d.w = __fmul_rn(d.w, pt[3]);
            tan_store(db + (uint32_t)k * 512u, d);
        }
        for (int k = olo; k < ohi; ++k) {
            float4 d = fresh ? make_float4(1.0f, 1.0f, 1.0f, 1.0f) : tan_load(db + (uint32_t)k * 512u);
            d.x = __fmul_rn(d.x, po[0]);
            d.y = __fmul_rn(d.y, po[1]);
            d.z = __fmul_rn(d.z, po[2]);
            d.w = __fmul_rn(d.w, po[3]);
            tan_store(db + (uint32_t)k * 512u, d);
        }
    }
    tp[0] = pack2(v[0], v[1]);
    tp[1] = pack2(v[2], v[3]);
#undef GP_ROWS
}

// Runs one program of the gradient form over the lane's four rows: the
// gradient variant of the fast loop runs the words it can, marked ones
// with their tangent updates, and each word it hands back -- a marker with
// the word after it, or a word it does not run -- runs in grad_word.
// Returns the prediction in tp and leaves each constant's tangent
// d(prediction)/d(c_k) at db + k * 512.  The columns as in interpret().
template <bool XREG>
__device__ __forceinline__ void grad_run(uint64_t (&tp)[2], const uint2 *cbuf, uint64_t (&x0)[2],
                                         const uint64_t (&x1)[2], const float *__restrict__ xc,
                                         int64_t ld, uint32_t unit, uint32_t mode, bool packed, int last,
                                         uint32_t sb, uint32_t db) {
    asm volatile("" : "=l"(tp[0]), "=l"(tp[1]));  // (the first word is a push)
    uint32_t pa = (uint32_t)__cvta_generic_to_shared(cbuf);
#pragma unroll 1
    for (;;) {
        uint32_t hw;
        float hc;
        if constexpr (XREG) fast_r4_divs_x_grad(pa, tp, x0, x1, sb, db, hw, hc);
        else fast_r4_divs_nox_grad(pa, tp, x0, xc, unit, mode, sb, db, hw, hc);
        uint32_t w = __shfl_sync(0xffffffffu, hw, 0);
        float c = hc;
        uint32_t mk = 0u;
        if ((w & 63u) == kGradMark) {
            mk = __shfl_sync(0xffffffffu, __float_as_uint(hc), 0);
            uint32_t w2, c2;
            asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(w2), "=r"(c2) : "r"(pa));
            pa += 8u;
            w = __shfl_sync(0xffffffffu, w2, 0);
            c = __uint_as_float(c2);
        }
        if ((w & 31u) == OP_END) break;
        grad_word<XREG>(w, c, mk, tp, x0, x1, xc, ld, packed, last, sb, db);
    }
}

// shared memory of one block: the program's words (through the buffer's
// end OP_END), then per warp UNITS x 128 bytes: the value stack [depth - 1][32
// lanes] and the tangents [constants][32 lanes], one float4 (four rows) per
// entry, and (without GREG) the constants' sums [constants][32 lanes]
template <int WARPS, int UNITS>
constexpr size_t grad_smem_bytes() {
    return (size_t)(kGradCodeStride + 2) * sizeof(uint2) + (size_t)WARPS * UNITS * 128;
}

// GREG: the constants' sums in registers (unrolled over GP_MAX_CONSTS), else in
// shared memory, so that a bucket's limit need not be a number of constants
template <int WARPS, int UNITS, int MINB, bool GREG, bool XREG>
__global__ void __launch_bounds__(WARPS * 32, MINB) grad_kernel(const GradArgs a) {
    constexpr int R = 4, KT = GREG ? GP_MAX_CONSTS : 1;
    static_assert(GP_MAX_CONSTS <= 32 && WARPS >= 2, "one thread per constant in warp 1");
    static_assert((kGradCodeStride + 2) * sizeof(uint2) % 16 == 0, "stack alignment");
    extern __shared__ float4 smem_grad[];
    uint2 *cbuf = reinterpret_cast<uint2 *>(smem_grad);
    float4 *const mine_all = smem_grad + (kGradCodeStride + 2) * sizeof(uint2) / 16;
    __shared__ float wsum[WARPS];
    __shared__ float wgrad[WARPS][GP_MAX_CONSTS];
    __shared__ int4 s_item[2];  // chunk (-1: the queue is empty), program, words, constants | stack slots << 8 (-1: none to run)
    __shared__ unsigned long long s_total;
    __shared__ int s_begin, s_n;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    float4 *const mine = mine_all + (size_t)warp * UNITS * 8;  // the warp's units
    const uint32_t sb = (uint32_t)__cvta_generic_to_shared(mine + lane);
    // thread 0 takes the next item while the block works on this one (as in
    // the evaluator)
    auto take = [&](unsigned long long item, int slot) {
        int4 it = make_int4(-1, 0, 0, 0);
        if (item < s_total) {
            const uint32_t n = (uint32_t)s_n;
            it.x = (int)((s_total >> 32) ? item / n : (uint32_t)item / n);
            it.y = a.order[s_begin + (int)(item - (unsigned long long)it.x * n)];
            const ProgMeta m = a.meta[it.y];
            it.z = m.n_ins;
            it.w = m.n_consts | (m.depth - 1) << 8;
            if (m.status != GP_PROG_OK || m.n_consts > GP_MAX_CONSTS || m.n_ins > kGradCodeStride) {
                it.w = -1;
                if (m.n_consts > GP_MAX_CONSTS) atomicOr(a.dev_status, GP_DEV_TOO_MANY_CONSTS);
            }
        }
        s_item[slot] = it;
    };
    griddep_wait();
    griddep_launch();
    if (threadIdx.x == 0) {
        int begin = 0;
        for (int b = 0; b < a.bucket; ++b) begin += a.class_count[b];
        s_begin = begin;
        s_n = a.class_count[a.bucket];
        s_total = (unsigned long long)s_n * (unsigned long long)a.n_chunks;
        take(blockIdx.x, 0);  // the counter hands out the items from gridDim.x on
    }
    __syncthreads();

    for (int cur = 0;; cur ^= 1) {
        // (read again where it is needed: held across the interpreter the
        // item's numbers would spill)
        const volatile int4 *it = &s_item[cur];
        if (it->x < 0) break;
        const bool ok = it->w >= 0;
        if (ok) {
            const uint2 *src = a.code + (size_t)it->y * kGradCodeStride;
            const int n_ins = it->z;
            for (int i = threadIdx.x; i < n_ins; i += WARPS * 32) {
                uint2 v = src[i];
                // a column read's constant: the next column read, as an offset
                if (!XREG && (kColumnOps >> (v.x & 31u) & 1u))
                    v.y = (uint32_t)((uint64_t)v.y * (uint64_t)(a.x_unit == 16 ? a.ld >> 2 : a.ld));
                cbuf[i] = v;
            }
        }
        __syncthreads();  // the words are there
        unsigned long long next = 0;
        if (threadIdx.x == 0) next = gridDim.x + atomicAdd(a.counter + a.bucket, 1ULL);

        const int n_in = (int)min(a.n_rows - (int64_t)it->x * a.chunk_rows, a.chunk_rows);
        // the tangents lie past the stack, the sums past the tangents
        const uint32_t db = sb + (uint32_t)(it->w >> 8) * 512u;
        float *const gm = reinterpret_cast<float *>(mine + ((it->w >> 8) + (it->w & 255)) * 32) + lane;
        float gs[KT];
#pragma unroll
        for (int k = 0; k < KT; ++k) gs[k] = 0.0f;
        if (!GREG && ok)
            for (int k = 0; k < (it->w & 255); ++k) gm[k * 32] = 0.0f;
        float ls = 0.0f, lc = 0.0f;
        uint64_t x0[2], x1[2];
        auto first_column = [&](int base) {
            const bool pk = __all_sync(0xffffffffu, base + 32 * R <= n_in) && a.vec_ok;
            const int o = base + lane * R;
            const int64_t feat = cbuf[it->z - 1].y;
            load_quad(x0, a.X + (feat * a.ld + (int64_t)it->x * a.chunk_rows + o), pk, n_in - 1 - o);
        };
        if (!XREG && ok && warp * 32 * R < n_in) first_column(warp * 32 * R);
        for (int base = warp * 32 * R; base < n_in && ok; base += WARPS * 32 * R) {
            const bool whole = __all_sync(0xffffffffu, base + 32 * R <= n_in);
            const bool packed = whole && a.vec_ok;
            const int o = base + lane * R;
            const int last = n_in - 1 - o;
            uint64_t t[2];
            {
                const float *xr = a.X + ((int64_t)it->x * a.chunk_rows + o);
                if (XREG) {
                    load_quad(x0, xr, packed, last);
                    load_quad(x1, xr + (a.n_feat == 2 ? a.ld : 0), packed, last);
                }
                const uint32_t mode = a.x_unit == 0 || !whole ? 2u : packed ? 0u : 1u;
                grad_run<XREG>(t, cbuf, x0, x1, xr, a.ld, (uint32_t)a.x_unit, mode, packed,
                                          last, sb, db);
            }
            const int64_t r = (int64_t)it->x * a.chunk_rows + o;
            const int nc = it->w & 255;
            if (!XREG && base + WARPS * 32 * R < n_in) first_column(base + WARPS * 32 * R);
            // the loss and its derivative per row
            const int nv = whole ? R : last + 1;  // rows of the lane that count
            uint64_t yv[2], wv[2];
            load_quad(yv, a.y + r, packed, last);
            if (a.w) load_quad(wv, a.w + r, packed, last);
            kahan_add(ls, lc, loss_sum<R>(a.metric, t, yv, wv, a.w != nullptr, whole, nv));
            float at[R];
            {
                float tv[R], yy[R], ww[R];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    unpack2(t[i], tv[2 * i], tv[2 * i + 1]);
                    unpack2(yv[i], yy[2 * i], yy[2 * i + 1]);
                    if (a.w) unpack2(wv[i], ww[2 * i], ww[2 * i + 1]);
                }
                if (a.metric == GP_MAE) {
#pragma unroll
                    for (int j = 0; j < R; ++j) at[j] = g_dloss(GP_MAE, tv[j], yy[j]);
                } else if (a.metric == GP_LOGLOSS) {
#pragma unroll
                    for (int j = 0; j < R; ++j) at[j] = g_dloss(GP_LOGLOSS, tv[j], yy[j]);
                } else {
#pragma unroll
                    for (int j = 0; j < R; ++j) at[j] = g_dloss(GP_MSE, tv[j], yy[j]);
                }
                if (a.w) {
#pragma unroll
                    for (int j = 0; j < R; ++j) at[j] = __fmul_rn(ww[j], at[j]);
                }
            }
            // each constant's share: the rows' loss derivatives times its
            // tangents (rows past the end do not count, whatever they hold)
            auto share = [&](const float4 d) {
                float q = __fmul_rn(at[0], d.x);
                if (whole) {
                    q = __fadd_rn(q, __fmul_rn(at[1], d.y));
                    q = __fadd_rn(q, __fmul_rn(at[2], d.z));
                    return __fadd_rn(q, __fmul_rn(at[3], d.w));
                }
                q = nv > 0 ? q : 0.0f;
                q = nv > 1 ? __fadd_rn(q, __fmul_rn(at[1], d.y)) : q;
                q = nv > 2 ? __fadd_rn(q, __fmul_rn(at[2], d.z)) : q;
                return nv > 3 ? __fadd_rn(q, __fmul_rn(at[3], d.w)) : q;
            };
            if (GREG) {
#pragma unroll
                for (int k = 0; k < KT; ++k)
                    if (k < nc) gs[k] = __fadd_rn(gs[k], share(tan_load(db + (uint32_t)k * 512u)));
            } else {
#pragma unroll 1
                for (int k = 0; k < nc; ++k)
                    gm[k * 32] = __fadd_rn(gm[k * 32], share(tan_load(db + (uint32_t)k * 512u)));
            }
        }
        if (threadIdx.x == 0) take(next, cur ^ 1);
        const int nc = ok ? it->w & 255 : 0;
        // fixed butterfly per warp, then the warps in order
        float lv = __fsub_rn(ls, lc);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) lv = __fadd_rn(lv, __shfl_xor_sync(0xffffffffu, lv, off));
        if (lane == 0) wsum[warp] = lv;
        auto total = [&](int k, float v) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, off));
            if (lane == 0) wgrad[warp][k] = v;
        };
        if (GREG) {
#pragma unroll
            for (int k = 0; k < KT; ++k)
                if (k < nc) total(k, gs[k]);
        } else {
            for (int k = 0; k < nc; ++k) total(k, gm[k * 32]);
        }
        __syncthreads();  // the sums and the next item complete; everyone is done with cbuf
        if (threadIdx.x == 0) {
            float v = 0.0f;
            for (int q = 0; q < WARPS; ++q) v = __fadd_rn(v, wsum[q]);
            a.part[(size_t)it->y * a.n_chunks + it->x] = ok ? v : __int_as_float(0x7fc00000);
        } else if (threadIdx.x >= 32 && threadIdx.x < 32 + GP_MAX_CONSTS) {
            const int k = threadIdx.x - 32;
            float v = 0.0f;
            if (k < nc)
                for (int q = 0; q < WARPS; ++q) v = __fadd_rn(v, wgrad[q][k]);
            a.gpart[((size_t)it->y * a.n_chunks + it->x) * GP_MAX_CONSTS + k] =
                ok ? v : __int_as_float(0x7fc00000);
        }
    }
}

template <int WARPS, int UNITS, int MINB, bool GREG, bool XREG>
cudaError_t launch_grad_t(const GradArgs &a, int sms, cudaStream_t st, int *occ_out) {
    static std::atomic<int> known[kMaxDevices];  // resident blocks, asked for once per device
    constexpr size_t smem = grad_smem_bytes<WARPS, UNITS>();
    auto k = grad_kernel<WARPS, UNITS, MINB, GREG, XREG>;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    int occ = known[dev].load(std::memory_order_acquire);
    if (occ == 0) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, WARPS * 32, smem);
        if (e != cudaSuccess) return e;
        occ = occ > 0 ? occ : 1;
        known[dev].store(occ, std::memory_order_release);
    }
    if (occ_out) {
        *occ_out = occ;
        return cudaSuccess;
    }
    return launch_chained(k, sms * occ, WARPS * 32, smem, st, a);
}

// Four rows per lane, 8 warps and 4, 3 or 2 blocks per SM by what the bucket's
// programs need of shared memory (grad_bucket); bucket 3: 4 warps, 3 blocks.
#define GP_GRAD_LAUNCH(W, U, M, G) \
    (xreg ? launch_grad_t<W, U, M, G, true>(a, sms, st, occ) \
          : launch_grad_t<W, U, M, G, false>(a, sms, st, occ))
cudaError_t launch_grad(const GradArgs &a, int sms, cudaStream_t st, int *occ) {
    const bool xreg = a.n_feat <= 2;
    switch (a.bucket) {
    case 0: return GP_GRAD_LAUNCH(8, kGradUnits0, 4, false);
    case 1: return GP_GRAD_LAUNCH(8, kGradUnits1, 3, false);
    case 2: return GP_GRAD_LAUNCH(8, grad_units(GP_MAX_CONSTS, kSmallDepth), 2, false);
    default: return GP_GRAD_LAUNCH(4, 4 * (kDeepSlots + GP_MAX_CONSTS), 3, true);
    }
}
#undef GP_GRAD_LAUNCH

// Adam: one thread per program walks its prefix list; the k-th CONST node
// takes slot k of grad / m / v.
__global__ void __launch_bounds__(128) adam_kernel(AdamArgs a) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.n_progs) return;
    const int off = a.offsets[p];
    const int len = a.offsets[p + 1] - off;
    if (len < 1 || len > GP_MAX_LEN) return;
    const float b1t = 1.0f - powf(a.beta1, (float)a.step);
    const float b2t = 1.0f - powf(a.beta2, (float)a.step);
    int k = 0;
    for (int j = 0; j < len && k < GP_MAX_CONSTS; ++j) {
        gp_node *nd = a.progs + off + j;
        if (nd->op != GP_CONST) continue;
        const size_t i = (size_t)p * GP_MAX_CONSTS + k;
        const float g = a.grad[i];
        if (isfinite(g)) {
            const float mi = __fadd_rn(__fmul_rn(a.beta1, a.m[i]), __fmul_rn(1.0f - a.beta1, g));
            const float vi = __fadd_rn(__fmul_rn(a.beta2, a.v[i]),
                                       __fmul_rn(1.0f - a.beta2, __fmul_rn(g, g)));
            a.m[i] = mi;
            a.v[i] = vi;
            const float mh = __fdiv_rn(mi, b1t);
            const float vh = __fdiv_rn(vi, b2t);
            const float stp = __fdiv_rn(__fmul_rn(a.lr, mh), __fadd_rn(__fsqrt_rn(vh), a.eps));
            nd->c = __fsub_rn(nd->c, stp);
        }
        ++k;
    }
}

cudaError_t launch_adam(const AdamArgs &a, cudaStream_t st) {
    if (a.n_progs <= 0) return cudaSuccess;
    adam_kernel<<<(a.n_progs + 127) / 128, 128, 0, st>>>(a);
    return cudaGetLastError();
}

// One thread per program: the k-th CONST node in prefix order is slot k.
__global__ void __launch_bounds__(128) consts_kernel(gp_node *progs, const int32_t *offsets,
                                                     int n_progs, float *consts, bool to_nodes) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n_progs) return;
    const int off = offsets[p];
    const int len = offsets[p + 1] - off;
    float *row = consts + (size_t)p * GP_MAX_CONSTS;
    int k = 0;
    if (len >= 1 && len <= GP_MAX_LEN) {
        for (int j = 0; j < len && k < GP_MAX_CONSTS; ++j) {
            gp_node *nd = progs + off + j;
            if (nd->op != GP_CONST) continue;
            if (to_nodes) nd->c = row[k];
            else row[k] = nd->c;
            ++k;
        }
    }
    if (!to_nodes)
        for (; k < GP_MAX_CONSTS; ++k) row[k] = 0.0f;
}

cudaError_t launch_consts(gp_node *progs, const int32_t *offsets, int n_progs, float *consts,
                          bool to_nodes, cudaStream_t st) {
    if (n_progs <= 0) return cudaSuccess;
    consts_kernel<<<(n_progs + 127) / 128, 128, 0, st>>>(progs, offsets, n_progs, consts, to_nodes);
    return cudaGetLastError();
}

}  // namespace gpk
