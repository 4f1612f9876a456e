// gp_interp.cuh -- the batched persistent evaluator (the hot loop).
//
// Work: every (program, row-chunk) pair of one program class is an item of a
// dynamic queue (one atomic counter); items are ordered chunk-major and,
// inside a chunk, longest program first, so the blocks that share the GPU
// at any moment work on the same few row chunks (X stays in L2) and the
// queue drains with the short items last.
//
// A block takes one item, the way the paper's execution kernel gives each
// block one program (Sec. III-C3, III-D1): the program's compiled
// instructions are copied once into shared memory and every warp of the
// block runs that same instruction stream over its own sub-tiles of 32*RPT
// rows (sub-tile w, w + warps, ...).  Within a warp the instruction stream
// is uniform, so the dispatch switch never diverges; across the block the
// warps walk the same few switch cases, which keeps the SM's instruction
// working set small.  In a whole sub-tile of 16-byte aligned columns lane l
// owns rows base + l*RPT .. +RPT-1 (16-byte loads); in a ragged one, or when
// the column length leaves columns unaligned, rows base + l + 32 j (coalesced
// 4-byte loads).  The top of the stack is the
// register array t[RPT]; deeper values sit in the warp's slice of a
// shared-memory stack, one float4 per (slot, group of 4 rows, lane), so a
// push or pop is one or two conflict-free 16-byte accesses per lane.  Each
// instruction costs one indexed branch (the inline-PTX fast loop, 4 or 8 rows
// per lane) or one switch, and nothing else that branches:
// measured on this GPU, an interpreter's dispatch latency grows with every
// dependent branch per instruction (about 20-40 cycles each) and with the
// number of distinct code locations it jumps between, so operand source and
// spill are part of the operation code rather than separate tests.
//
// After a sub-tile each lane turns its RPT predictions into weighted losses
// (the fused form of the paper's matrix-vector loss step) and adds them into
// a Kahan-compensated FP32 sum; at the end of the item each warp adds its 32
// lane sums with a fixed butterfly and thread 0 adds the warp sums in warp
// order, writing one partial per (program, chunk).  A separate pass adds the
// partials of a program in chunk order in FP64.  Every step has a fixed
// order, so results do not depend on which block ran which item.
//
// What surrounds the words -- loads, loss, loop -- costs 110 instructions per
// program and sub-tile at 8 rows per lane, of some 850 (220 before the rows
// were kept as pairs throughout, the ragged case put behind one vote, the next
// item taken by one thread and squares added with FMA: Pagie-1 16M x 4096
// 301 -> 260 ms with the shorter dispatch; with 28 unaligned columns, where a
// lane's consecutive rows took eight 4-byte loads of 32 sectors each, 22.2 ->
// 16.3 ms).
#pragma once

#include <atomic>

#include "gp_internal.cuh"
#include "gp_math.cuh"
#include "gp_fast.cuh"

namespace gpk {

// warps per block: 8, or 4 at 16 rows per thread (its shared-memory stack
// is twice as large per warp)
template <int RPT>
__host__ __device__ constexpr int eval_warps() { return RPT >= 16 ? 4 : 8; }

// ---- the function set (FP32, IEEE operators, no contraction) -----------
__device__ __forceinline__ float f_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float f_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float f_mul(float a, float b) { return __fmul_rn(a, b); }
// The protected operators compute the operation on every row and select
// afterwards: written as a branch around the operation, the compiler keeps
// a per-row branch, which costs more than the operation saved (measured).
__device__ __forceinline__ float f_div(float a, float b) {
    const float q = __fdiv_rn(a, b);
    return fabsf(b) < kThr ? 1.0f : q;
}
__device__ __forceinline__ float f_sqrt(float a) { return __fsqrt_rn(fabsf(a)); }
__device__ __forceinline__ float f_log(float a) {
    // the logarithm sees max(|a|, thr); inf and NaN, for which both tests
    // fail, are passed through
    const float b = fabsf(a);
    const float l = log_pos(fmaxf(b, kThr));
    return b < kThr ? 0.0f : (b <= 3.40282347e38f ? l : b);
}
__device__ __forceinline__ float f_exp(float a) {
    if (fabsf(a) < kExpFast) return exp_fast(a);
    if (a >= kExpInf) return __int_as_float(0x7f800000);
    return a <= kExpZero ? 0.0f : exp_wide(a);  // NaN: NaN
}
__device__ __forceinline__ float f_abs(float a) { return fabsf(a); }
__device__ __forceinline__ float f_neg(float a) { return -a; }
__device__ __forceinline__ float f_inv(float a) {
    const float r = __frcp_rn(a);
    return fabsf(a) < kThr ? 0.0f : r;
}

// per-row loss (metric readings of Sec. III-C3, FP32)
__device__ __forceinline__ float row_loss(int metric, float p, float y) {
    if (metric == GP_MAE) return fabsf(__fsub_rn(p, y));
    if (metric == GP_LOGLOSS) {
        const float ap = fabsf(p);
        const float c = (p >= 0.0f) ? __fsub_rn(1.0f, y) : y;
        const float lin = (c == 0.0f) ? 0.0f : __fmul_rn(c, ap);
        return __fadd_rn(lin, log1pf(expf(-ap)));
    }
    const float d = __fsub_rn(p, y);
    return __fmul_rn(d, d);
}

// two rows in one 64-bit register pair
__device__ __forceinline__ uint64_t pack2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t r, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}

// A lane's rows as pairs.  packed: RPT consecutive rows
// from p, 16-byte loads; else rows p[0], p[32], p[64], ..., the last of them
// at most p[last] (a ragged sub-tile reads its last row again; those rows
// do not count).
template <int RPT, int FMODE>
__device__ __forceinline__ void load_pairs(uint64_t (&v)[RPT / 2], const float *__restrict__ p,
                                           bool packed, int last) {
    if (packed) {
#pragma unroll
        for (int q = 0; q < RPT / 4; ++q) {
            const ulonglong2 f = __ldg(reinterpret_cast<const ulonglong2 *>(p) + q);
            v[2 * q] = f.x;
            v[2 * q + 1] = f.y;
        }
    } else {
        // keeps the minima in this branch: hoisted above it they cost feature
        // mode 0 registers and 8 instructions a sub-tile (4M x 50: 21.2 ->
        // 19.7 ms); mode 2 is better off without (16M x 4096: 259 against 263)
        if (FMODE == 0) asm volatile("" : "+r"(last));
#pragma unroll
        for (int i = 0; i < RPT / 2; ++i)
            v[i] = pack2(__ldg(p + min(64 * i, last)), __ldg(p + min(64 * i + 32, last)));
    }
}

__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// the weighted losses of a lane's rows added up (the first nv rows count);
// the metric and the weights are tested once, not per row.  The squares of
// whole sub-tiles (their products with the weights) are added as they are
// formed, without a rounding of their own, even and odd rows apart (9
// instructions for 8 rows instead of 24).  A weight multiplies the square, as
// in the other branch: w d first would stay finite for some errors whose
// square does not, in whole sub-tiles alone
template <int RPT>
__device__ __forceinline__ float loss_sum(int metric, const uint64_t (&tp)[RPT / 2],
                                          const uint64_t (&yp)[RPT / 2],
                                          const uint64_t (&wp)[RPT / 2], bool has_w, bool full,
                                          int nv) {
    if (full && (metric == GP_MSE || metric == GP_RMSE)) {
        uint64_t e2 = 0ull;
#pragma unroll
        for (int i = 0; i < RPT / 2; ++i) {
            const uint64_t d = sub2(tp[i], yp[i]);
            e2 = has_w ? fma2(wp[i], mul2(d, d), e2) : fma2(d, d, e2);
        }
        float lo, hi;
        unpack2(e2, lo, hi);
        return __fadd_rn(lo, hi);
    }
    float l[RPT], t[RPT], yv[RPT];
#pragma unroll
    for (int i = 0; i < RPT / 2; ++i) {
        unpack2(tp[i], t[2 * i], t[2 * i + 1]);
        unpack2(yp[i], yv[2 * i], yv[2 * i + 1]);
    }
    if (metric == GP_MAE) {
#pragma unroll
        for (int j = 0; j < RPT; ++j) l[j] = row_loss(GP_MAE, t[j], yv[j]);
    } else if (metric == GP_LOGLOSS) {
#pragma unroll
        for (int j = 0; j < RPT; ++j) l[j] = row_loss(GP_LOGLOSS, t[j], yv[j]);
    } else {
#pragma unroll
        for (int j = 0; j < RPT; ++j) l[j] = row_loss(GP_MSE, t[j], yv[j]);
    }
    if (has_w) {
        float wv[RPT];
#pragma unroll
        for (int i = 0; i < RPT / 2; ++i) unpack2(wp[i], wv[2 * i], wv[2 * i + 1]);
#pragma unroll
        for (int j = 0; j < RPT; ++j) l[j] = __fmul_rn(wv[j], l[j]);
    }
    float e = 0.0f;
    if (full) {
#pragma unroll
        for (int j = 0; j < RPT; ++j) e = __fadd_rn(e, l[j]);
    } else {
#pragma unroll
        for (int j = 0; j < RPT; ++j) e = (j < nv) ? __fadd_rn(e, l[j]) : e;
    }
    return e;
}

__device__ __forceinline__ void kahan_add(float &s, float &c, float x) {
    const float yv = __fsub_rn(x, c);
    const float tv = __fadd_rn(s, yv);
    // once the sum is infinite or NaN the compensation is meaningless
    c = isfinite(tv) ? __fsub_rn(__fsub_rn(tv, s), yv) : 0.0f;
    s = tv;
}

// The extended unary functions of four rows, out of line: with a case of
// their own each in the dispatch switch (a 6-bit switch), their code made
// the loop 4-5% slower on programs that never use them (measured on
// Pagie-1 x 4096 programs).
static __device__ __noinline__ float4 ext_rows4(float4 v, uint32_t f) {
    switch (f) {
        case EXT_SQ: return make_float4(f_sq(v.x), f_sq(v.y), f_sq(v.z), f_sq(v.w));
        case EXT_CUBE: return make_float4(f_cube(v.x), f_cube(v.y), f_cube(v.z), f_cube(v.w));
        case EXT_CBRT: return make_float4(f_cbrt(v.x), f_cbrt(v.y), f_cbrt(v.z), f_cbrt(v.w));
        case EXT_TANH: return make_float4(f_tanh(v.x), f_tanh(v.y), f_tanh(v.z), f_tanh(v.w));
        case EXT_ATAN: return make_float4(f_atan(v.x), f_atan(v.y), f_atan(v.z), f_atan(v.w));
        case EXT_SINH: return make_float4(f_sinh(v.x), f_sinh(v.y), f_sinh(v.z), f_sinh(v.w));
        default: return make_float4(f_cosh(v.x), f_cosh(v.y), f_cosh(v.z), f_cosh(v.w));
    }
}

// ---- the fast loop: indexed-branch dispatch in inline PTX ------------
// The compiler lowers the dispatch switch to a tree of compares and
// branches (about 12 instructions per dispatch, measured with ncu's
// per-opcode counts); PTX's brx.idx jumps through a table instead (about
// 3).  gp_fast.cuh (written by gen_fast.py) holds the loop for 4 and 8 rows
// per lane: a lane's rows sit in RPT/2 64-bit pairs and add, sub, mul and
// fma run as one packed f32x2 instruction per pair (per-element round to
// nearest, no flush to zero: the bits of the scalar operations).  It runs
// pushes and stack moves, add/sub/mul with every operand form, abs, neg, the
// protected divisions, square root, reciprocal, sin, cos, log and exp (the
// steps and constants of gp_math.cuh, so results are the same bits), column
// reads from registers (XREG) or one ahead from memory, and, with EXT, sq,
// cube, max and min.  It stops at the first word it does not run (END, tan,
// the other extended functions, arguments outside a fast path in any row of
// the warp, column reads of a ragged sub-tile), hands that word and its
// constant back to the switch below and leaves pa just past it.
template <int RPT, bool EXT, bool XREG, bool LEAN>
__device__ __forceinline__ void run_fast(uint32_t &pa, uint64_t (&t)[RPT / 2],
                                         uint64_t (&x0)[RPT / 2], const uint64_t (&x1)[RPT / 2],
                                         const float *xc, uint32_t unit, uint32_t mode, uint32_t &sp,
                                         uint32_t &hw, float &hc) {
    if constexpr (RPT == 4) {
        if constexpr (!EXT && XREG) fast_r4_divs_x(pa, t, x0, x1, sp, hw, hc);
        else if constexpr (!EXT) fast_r4_divs_nox(pa, t, x0, xc, unit, mode, sp, hw, hc);
        else if constexpr (XREG) fast_r4_ext_x(pa, t, x0, x1, sp, hw, hc);
        else fast_r4_ext_nox(pa, t, x0, xc, unit, mode, sp, hw, hc);
    } else {
        if constexpr (LEAN && XREG) fast_r8_divs_x_lean(pa, t, x0, x1, sp, hw, hc);
        else if constexpr (LEAN) fast_r8_divs_nox_lean(pa, t, x0, xc, unit, mode, sp, hw, hc);
        else if constexpr (!EXT && XREG) fast_r8_divs_x(pa, t, x0, x1, sp, hw, hc);
        else if constexpr (!EXT) fast_r8_divs_nox(pa, t, x0, xc, unit, mode, sp, hw, hc);
        else if constexpr (XREG) fast_r8_ext_x(pa, t, x0, x1, sp, hw, hc);
        else fast_r8_ext_nox(pa, t, x0, xc, unit, mode, sp, hw, hc);
    }
}

// Runs one compiled program over RPT rows per lane; returns the top of the
// stack in tp, rows as pairs.  stk = this warp's stack slice, already offset
// by the lane; xc, packed and last: column 0 at the lane's first row, and how
// the lane's rows follow it (load_pairs).  x0p and x1p: columns 0 and 1
// (FMODE 2), else the first column that the program reads in x0p (unit and
// mode: how the loop reads the next ones, see gp_fast.cuh).
// The instruction buffer holds the pre-pass's words, the last of them OP_END,
// as a dispatch index and a constant each, and their upper halves (the column
// or the extended function, read by the switch alone) in aux.  Its pushes and
// pops balance within the class's stack, so a pointer serves for the slots.
//
// Dispatch cost is what this loop is tuned for (per-opcode instruction
// counts measured with ncu on chains of one operation).  At 4 and 8 rows
// per lane the fast loop runs most words and hands the others, one at a
// time, to the switch below.  The instruction word and the stack are addressed
// through 32-bit shared-memory addresses computed once; the opcode is
// broadcast from lane 0, which lets the compiler treat the switch as
// warp-uniform (no reconvergence barrier per instruction); the switch
// covers every value of its 5-bit operand that occurs, so it needs no range test;
// and the word is loaded when it is needed rather than one ahead, which
// saves the register copies of a prefetch.
template <int RPT, int NSLOT, int FMODE, bool EXT, bool LEAN>
__device__ __forceinline__ void interpret(uint64_t (&tp)[RPT / 2], const uint2 *__restrict__ cbuf,
                                          uint64_t (&x0p)[RPT / 2],
                                          const uint64_t (&x1p)[RPT / 2],
                                          const float *__restrict__ xc, int64_t ld, uint32_t unit,
                                          uint32_t mode, bool packed, int last, float4 *stk,
                                          const uint16_t *aux) {
    // EXT: the extended functions are compiled in (classes 1 and 2).  In
    // class 0, where nearly all programs of the usual function set run,
    // their cases cost 2-3% (measured on Pagie-1 x 4096 programs, which
    // never use them)
    constexpr bool kExt = EXT;
    // the first word is a push: the rows need no value before it
#pragma unroll
    for (int i = 0; i < RPT / 2; ++i) asm volatile("" : "=l"(tp[i]));
    // pa: shared-memory address of the next instruction word
    uint32_t pa = (uint32_t)__cvta_generic_to_shared(cbuf);
    uint32_t sp = (uint32_t)__cvta_generic_to_shared(stk);  // this lane's next free slot
    constexpr uint32_t kSlotBytes = RPT / 4 * 32u * 16u;
    // 4 or 8 rows per lane: the fast loop runs what it can and hands back
    // the rest, one word at a time, to the switch below
    constexpr bool kFast = RPT == 4 || RPT == 8;
#pragma unroll 1
    for (;;) {
        uint2 ins;
        if constexpr (kFast) {
            float hc;
            run_fast<RPT, EXT, FMODE == 2, LEAN>(pa, tp, x0p, x1p, xc, unit, mode, sp, ins.x, hc);
            ins.y = __float_as_uint(hc);
        } else {
            asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];"
                         : "=r"(ins.x), "=r"(ins.y)
                         : "r"(pa));
            pa += 8u;
        }
        const uint32_t w = __shfl_sync(0xffffffffu, ins.x, 0);
        // the end of the program, once per sub-tile: out before the switch
        if ((w & 31u) == OP_END) break;
        float t[RPT];
#pragma unroll
        for (int i = 0; i < RPT / 2; ++i) unpack2(tp[i], t[2 * i], t[2 * i + 1]);
        const float c = __uint_as_float(ins.y);
// the word's upper half
#define GP_HI ((uint32_t)aux[(pa - (uint32_t)__cvta_generic_to_shared(cbuf)) / 8u - 1u])
// operand helpers: stack slot, X column, constant
// (the stack is laid out [slot][q][lane] in float4)
#define GP_SLOT_LOAD(u)                                                         \
    {                                                                           \
        _Pragma("unroll") for (int q = 0; q < RPT / 4; ++q) {                   \
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"             \
                         : "=f"(u[4 * q]), "=f"(u[4 * q + 1]),                  \
                           "=f"(u[4 * q + 2]), "=f"(u[4 * q + 3])               \
                         : "r"(sp + q * 512u));                                 \
        }                                                                       \
    }
#define GP_POP(u) { sp -= kSlotBytes; GP_SLOT_LOAD(u) }
#define GP_SPILL()                                                              \
    {                                                                           \
        _Pragma("unroll") for (int q = 0; q < RPT / 4; ++q)                     \
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};"             \
                         ::"r"(sp + q * 512u),                                  \
                           "f"(t[4 * q]), "f"(t[4 * q + 1]), "f"(t[4 * q + 2]),  \
                           "f"(t[4 * q + 3])                                    \
                         : "memory");                                           \
        sp += kSlotBytes;                                                       \
    }
#define GP_X_LOAD(u)                                                            \
    {                                                                           \
        const int feat = FMODE == 2 ? (int)(w >> 5) : (int)GP_HI;               \
        uint64_t up[RPT / 2];                                                   \
        if (FMODE == 2) {                                                       \
            _Pragma("unroll") for (int i = 0; i < RPT / 2; ++i) up[i] = feat ? x1p[i] : x0p[i]; \
        } else {                                                                \
            load_pairs<RPT, FMODE>(up, xc + (int64_t)feat * ld, packed, last);         \
        }                                                                       \
        _Pragma("unroll") for (int i = 0; i < RPT / 2; ++i)                     \
            unpack2(up[i], u[2 * i], u[2 * i + 1]);                             \
    }
#define GP_T(expr) _Pragma("unroll") for (int j = 0; j < RPT; ++j) t[j] = expr;
#define GP_U_C(u) _Pragma("unroll") for (int j = 0; j < RPT; ++j) u[j] = c;
        float u[RPT];
        switch (w & 31u) {
            case OP_PUSH_X: GP_X_LOAD(u) GP_T(u[j]) break;
            case OP_PUSH_C: GP_T(c) break;
            case OP_PUSH_X_SP: GP_SPILL() GP_X_LOAD(u) GP_T(u[j]) break;
            case OP_PUSH_C_SP: GP_SPILL() GP_T(c) break;
            case OP_ADD_S: GP_POP(u) GP_T(f_add(t[j], u[j])) break;
            case OP_SUB_S: GP_POP(u) GP_T(f_sub(t[j], u[j])) break;
            case OP_MUL_S: GP_POP(u) GP_T(f_mul(t[j], u[j])) break;
            case OP_DIV_S:  // (the loop has moved sp for a division that it hands back)
                if (kFast) GP_SLOT_LOAD(u) else GP_POP(u)
                goto div_tu;
            case OP_ADD_X: GP_X_LOAD(u) GP_T(f_add(t[j], u[j])) break;
            case OP_ADD_C: GP_T(f_add(t[j], c)) break;
            case OP_SUB_X: GP_X_LOAD(u) GP_T(f_sub(t[j], u[j])) break;
            case OP_SUB_C: GP_T(f_sub(t[j], c)) break;
            case OP_RSUB_X: GP_X_LOAD(u) GP_T(f_sub(u[j], t[j])) break;
            case OP_RSUB_C: GP_T(f_sub(c, t[j])) break;
            case OP_MUL_X: GP_X_LOAD(u) GP_T(f_mul(t[j], u[j])) break;
            case OP_MUL_C: GP_T(f_mul(t[j], c)) break;
            case OP_DIV_X: GP_X_LOAD(u) goto div_tu;
            case OP_DIV_C: GP_U_C(u) goto div_tu;
            case OP_RDIV_X: GP_X_LOAD(u) goto div_ut;
            case OP_RDIV_C: GP_U_C(u) goto div_ut;
            case OP_SQRT: GP_T(f_sqrt(t[j])) break;
            case OP_LOG: GP_T(f_log(t[j])) break;
            case OP_EXP: GP_T(f_exp(t[j])) break;
            case OP_SIN:
            case OP_COS:
            case OP_TAN: trig_rows<RPT>(t, (int)(w & 31u) - OP_SIN); break;
            case OP_ABS: GP_T(f_abs(t[j])) break;
            case OP_NEG: GP_T(f_neg(t[j])) break;
            case OP_INV: GP_T(f_inv(t[j])) break;
            case OP_EXT1:  // out of line, four rows per call
                if constexpr (kExt) {
                    const uint32_t fn = GP_HI;
                    _Pragma("unroll") for (int g = 0; g < RPT / 4; ++g) {
                        const float4 r = ext_rows4(
                            make_float4(t[4 * g], t[4 * g + 1], t[4 * g + 2], t[4 * g + 3]),
                            fn);
                        t[4 * g] = r.x; t[4 * g + 1] = r.y; t[4 * g + 2] = r.z; t[4 * g + 3] = r.w;
                    }
                    break;
                } else {
                    goto done;
                }
            case OP_END:
                goto done;
            default:  // every other value has a case above, but OP_EXT2, which the loop runs
                __builtin_unreachable();
        }
        goto next;
        // division has one body per operand order, shared by its operand cases
    div_tu:
        GP_T(f_div(t[j], u[j]))
        goto next;
    div_ut:
        GP_T(f_div(u[j], t[j]))
    next:
#pragma unroll
        for (int i = 0; i < RPT / 2; ++i) tp[i] = pack2(t[2 * i], t[2 * i + 1]);
#undef GP_T
#undef GP_U_C
#undef GP_X_LOAD
#undef GP_SPILL
#undef GP_HI
#undef GP_POP
#undef GP_SLOT_LOAD
    }
done:;
}

// shared memory of one block: the program's instructions, then the stack
template <int RPT, int NSLOT>
constexpr size_t eval_smem_bytes() {
    return (size_t)(kCodeStride + 2) * sizeof(uint2) +
           (size_t)eval_warps<RPT>() * NSLOT * (RPT / 4) * 32 * sizeof(float4);
}

// epilogues: the weighted loss sum, the predictions, or the moment sums
// of the correlation fitness.  At 8 rows per thread the loss and store
// epilogues ask for 4 resident blocks (at most 64 registers, with the
// 6-slot stack of class 0: 295 against 312 ms at 3 blocks on Pagie-1 16M
// x 4096), the moment epilogue for 3 (at most 85 registers).  At 4 rows the moment epilogue asks for 5 (at most 48
// registers, a few spilled words: 4% faster than 4 blocks at 59 registers
// on Pagie-1 16M x 4096); the others are left alone (46 registers: 5 fit),
// because asking for 5 blocks there changed their schedule and cost 7%.
constexpr int kEpiLoss = 0, kEpiPred = 1, kEpiMom = 2;

template <int RPT, int NSLOT, int FMODE, int EPI, bool EXT>
__global__ void __launch_bounds__(eval_warps<RPT>() * 32,
                                  RPT == 8 ? (EPI == kEpiMom || EXT ? 3 : 4)
                                           : (EPI == kEpiMom && RPT == 4 ? 5 : 0))
    eval_kernel(const EvalArgs a) {
    constexpr bool PRED = EPI == kEpiPred;
    constexpr bool MOM = EPI == kEpiMom;
    // Special values (NaN, infinities, zero) run in the loop, except for the
    // fitness of class 0 at 8 rows, where the paths' code cost 2.3% (Pagie-1 16M
    // x 4096) and a program that meets many has no fitness.  Handed back,
    // they took most words of a table with 1% of NaN out of the loop:
    // predictions of 512 programs, 200000 rows x 5 columns, 1.14 -> 0.46 ms, over
    // the paper's set 2.23 -> 0.66; without NaN no difference
    constexpr bool kLean = RPT == 8 && !EXT && !PRED;
    constexpr int kEvalWarps = eval_warps<RPT>();
    constexpr int kEvalBlock = kEvalWarps * 32;
    extern __shared__ float4 smem_eval[];
    uint2 *cbuf = reinterpret_cast<uint2 *>(smem_eval);
    float4 *stack_all = smem_eval + ((kCodeStride + 2) * sizeof(uint2) + 15) / 16;
    __shared__ float wsum[kEvalWarps];
    __shared__ double wmom[MOM ? kEvalWarps : 1][3];
    __shared__ int4 s_item[2];  // chunk (-1: the queue is empty), program, words, status
    __shared__ unsigned long long s_total;
    __shared__ int s_begin, s_n;
    __shared__ uint16_t aux[kCodeStride + 2];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    float4 *stk = stack_all + (size_t)warp * NSLOT * (RPT / 4) * 32 + lane;

    // Thread 0 takes the next item while the block works on this one: it
    // alone waits for the counter and splits the number into (chunk, rank).
    // What it needs for that, and the item itself, sit in shared memory: in
    // registers they would stay live across the interpreter
    auto take = [&](unsigned long long item, int slot) {
        int4 it = make_int4(-1, 0, 0, 0);
        if (item < s_total) {
            const uint32_t n = (uint32_t)s_n;
            it.x = (int)((s_total >> 32) ? item / n : (uint32_t)item / n);
            it.y = a.order[s_begin + (int)(item - (unsigned long long)it.x * n)];
            const ProgMeta m = a.meta[it.y];
            it.z = m.n_ins;
            it.w = m.status;
        }
        s_item[slot] = it;
    };
    griddep_wait();
    griddep_launch();
    const float ybar = MOM ? (float)a.ystat[3] : 0.0f;
    if (threadIdx.x == 0) {
        const int qc = a.qcls ? a.qcls - 1 : a.cls;  // the span of the program order
        int begin = 0, n = a.class_count[qc];
        for (int b = 0; b < qc; ++b) begin += a.class_count[b];
        if (a.sub == 1) {  // the long programs of class 0 (first in its order)
            n = a.class_count[kOrderClasses];
        } else if (a.sub == 2) {  // the rest of class 0
            begin = a.class_count[kOrderClasses];
            n -= begin;
        }
        s_begin = begin;
        s_n = n;
        s_total = (unsigned long long)n * (unsigned long long)a.n_chunks;
        take(blockIdx.x, 0);  // the counter hands out the items from gridDim.x on
    }
    __syncthreads();

    // one item per pass: every number comes up once, so a block makes at most
    // s_total passes
    for (int cur = 0;; cur ^= 1) {
        const int4 it = s_item[cur];
        const int chunk = it.x, p = it.y;
        if (chunk < 0) break;
        const int64_t rb = (int64_t)chunk * a.chunk_rows;
        const int n_in = (int)(min(a.n_rows, rb + a.chunk_rows) - rb);
        const bool ok = it.w == GP_PROG_OK;
        // the program's words (OP_END the last of them)
        if (ok) {
            const uint2 *src = a.code + (size_t)p * (a.code_stride ? a.code_stride : kCodeStride);
            for (int i = threadIdx.x; i < it.z && i <= kCodeStride; i += kEvalBlock) {
                uint2 v = src[i];
                aux[i] = (uint16_t)(v.x >> 16);
                // a column read's constant: the next column read, as an offset
                if (FMODE == 0 && (kColumnOps >> (v.x & 31u) & 1u))
                    v.y = (uint32_t)((uint64_t)v.y * (uint64_t)(a.x_unit == 16 ? a.ld >> 2 : a.ld));
                const uint32_t op = v.x & 31u, fn = v.x >> 16;
                uint32_t index = v.x & 63u;
                if (EXT && op == OP_EXT2) index = fn == EXT_MAX ? kIndexMax : kIndexMin;
                if (EXT && op == OP_EXT1 && fn <= EXT_CUBE) index = fn == EXT_SQ ? kIndexSq : kIndexCube;
                cbuf[i] = make_uint2(index, v.y);
            }
        }
        __syncthreads();  // the words are there
        unsigned long long next = 0;
        if (threadIdx.x == 0) next = gridDim.x + atomicAdd(a.counter, 1ULL);

        float ks = 0.0f, kc = 0.0f;
        float ms[3] = {0.0f, 0.0f, 0.0f}, mc[3] = {0.0f, 0.0f, 0.0f};
        const float shift = MOM ? a.shift[p] : 0.0f;
        // FMODE 0: x0 holds the first column that the program reads (END's
        // constant); its loads for the next sub-tile are issued before the
        // loss of this one
        uint64_t x0[RPT / 2], x1[RPT / 2];
        auto first_column = [&](int base) {
            const bool pk = __all_sync(0xffffffffu, base + 32 * RPT <= n_in) && a.vec_ok;
            const int o = base + (pk ? lane * RPT : lane);
            const volatile int4 *it = &s_item[cur];
            const int64_t feat = cbuf[it->z - 1].y;
            load_pairs<RPT, FMODE>(x0, a.X + (feat * a.ld + (int64_t)it->x * a.chunk_rows + o), pk,
                            n_in - 1 - o);
        };
        constexpr bool kAhead = FMODE == 0;  // the loop reads columns ahead
        if (kAhead && ok && warp * 32 * RPT < n_in) first_column(warp * 32 * RPT);
        for (int base = warp * 32 * RPT; base < n_in && ok; base += kEvalWarps * 32 * RPT) {
            // whole: every row of the sub-tile is in the chunk; packed: and
            // the lane's rows are consecutive.  One test for the warp (a vote:
            // the compiler then knows that the warp agrees, and needs no
            // reconvergence around the loads and the loss)
            const bool whole = __all_sync(0xffffffffu, base + 32 * RPT <= n_in);
            const bool packed = whole && a.vec_ok;
            const int o = base + (packed ? lane * RPT : lane);  // the lane's first row
            const int last = n_in - 1 - o;   // its furthest row (negative: none; see load_pairs)
            uint64_t t[RPT / 2];
            {
                const float *xr = a.X + (rb + o);
                if (FMODE == 2) {
                    load_pairs<RPT, FMODE>(x0, xr, packed, last);
                    load_pairs<RPT, FMODE>(x1, xr + a.ld, packed, last);
                }
                const uint32_t mode = a.x_unit == 0 || !whole ? 2u : packed ? 0u : 1u;
                interpret<RPT, NSLOT, FMODE, EXT, kLean>(t, cbuf, x0, x1, xr, a.ld, (uint32_t)a.x_unit, mode,
                                                  packed, last, stk, aux);
            }
            // the lane's first row again; in feature mode 0 from the item, as held
            // across the interpreter it would cost two registers that spill
            // (4M x 50: 21.5 -> 20.4 ms; with two columns, where nothing
            // spills, 16M x 4096 260 -> 268 ms)
            const int64_t r =
                (FMODE == 2 ? rb : (int64_t)*const_cast<volatile int *>(&s_item[cur].x) * a.chunk_rows) + o;
            const int nv = whole ? RPT : (last + 32) >> 5;  // rows of the lane that count
            if (kAhead && base + kEvalWarps * 32 * RPT < n_in)
                first_column(base + kEvalWarps * 32 * RPT);
            if (PRED) {
                float *dst = a.pred + (size_t)p * a.n_rows + r;
                if (packed) {
#pragma unroll
                    for (int q = 0; q < RPT / 4; ++q)
                        reinterpret_cast<ulonglong2 *>(dst)[q] = make_ulonglong2(t[2 * q], t[2 * q + 1]);
                } else {
#pragma unroll
                    for (int i = 0; i < RPT / 2; ++i) {
                        float lo, hi;
                        unpack2(t[i], lo, hi);
                        if (2 * i < nv) dst[64 * i] = lo;
                        if (2 * i + 1 < nv) dst[64 * i + 32] = hi;
                    }
                }
                continue;
            }
            uint64_t yv[RPT / 2], wv[RPT / 2];
            load_pairs<RPT, FMODE>(yv, a.y + r, packed, last);
            if (a.w) load_pairs<RPT, FMODE>(wv, a.w + r, packed, last);
            if (MOM) {
                // d = p - shift keeps the sums of squares free of the
                // cancellation a large mean would cause
                float e1 = 0.0f, e2 = 0.0f, e3 = 0.0f;
#pragma unroll
                for (int j = 0; j < RPT; ++j) {
                    float tv[2], yy[2], ww[2] = {1.0f, 1.0f};
                    unpack2(t[j / 2], tv[0], tv[1]);
                    unpack2(yv[j / 2], yy[0], yy[1]);
                    if (a.w) unpack2(wv[j / 2], ww[0], ww[1]);
                    const float d = __fsub_rn(tv[j & 1], shift);
                    const float yc_ = __fsub_rn(yy[j & 1], ybar);
                    const float wd = a.w ? __fmul_rn(ww[j & 1], d) : d;
                    const bool in = j < nv;
                    e1 = in ? __fadd_rn(e1, wd) : e1;
                    e2 = in ? __fadd_rn(e2, __fmul_rn(wd, d)) : e2;
                    e3 = in ? __fadd_rn(e3, __fmul_rn(wd, yc_)) : e3;
                }
                kahan_add(ms[0], mc[0], e1);
                kahan_add(ms[1], mc[1], e2);
                kahan_add(ms[2], mc[2], e3);
            } else {
                kahan_add(ks, kc, loss_sum<RPT>(a.metric, t, yv, wv, a.w != nullptr, whole, nv));
            }
        }
        if (threadIdx.x == 0) take(next, cur ^ 1);
        if (MOM) {
            // the lane's compensated sums in FP64, then a fixed butterfly
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                double v = (double)ms[k] - (double)mc[k];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == 0) wmom[warp][k] = v;
            }
        } else if (!PRED) {
            float v = __fsub_rn(ks, kc);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
            if (lane == 0) wsum[warp] = v;
        }
        __syncthreads();  // wsum and the next item complete; everyone is done with cbuf
        if (PRED) {
            if (!ok)
                for (int i = threadIdx.x; i < n_in; i += kEvalBlock)
                    a.pred[(size_t)p * a.n_rows + rb + i] = __int_as_float(0x7fc00000);
        } else if (MOM && threadIdx.x < 3) {
            double v = 0.0;
            for (int w = 0; w < kEvalWarps; ++w) v += wmom[w][threadIdx.x];
            a.mom[((size_t)p * a.n_chunks + chunk) * 3 + threadIdx.x] =
                ok ? v : __longlong_as_double(0x7ff8000000000000LL);
        } else if (!MOM && threadIdx.x == 0) {
            float v = 0.0f;
            for (int w = 0; w < kEvalWarps; ++w) v = __fadd_rn(v, wsum[w]);
            a.part[(size_t)p * a.n_chunks + chunk] = ok ? v : __int_as_float(0x7fc00000);
        }
    }
}

// Resident blocks per SM, after making the instance's shared memory
// available; asked for once per device (the two runtime calls took 3 us of
// each of an evaluation's four launches)
template <int RPT, int NSLOT, int FMODE, int EPI, bool EXT>
int info_t(int block, int *regs) {
    (void)block;
    static std::atomic<int> known[kMaxDevices];  // blocks + 1
    constexpr size_t smem = eval_smem_bytes<RPT, NSLOT>();
    auto k = eval_kernel<RPT, NSLOT, FMODE, EPI, EXT>;
    if (regs) {
        cudaFuncAttributes fa{};
        if (cudaFuncGetAttributes(&fa, k) != cudaSuccess) return 0;
        *regs = fa.numRegs;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
    int n = known[dev].load(std::memory_order_acquire) - 1;
    if (n >= 0) return n;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, eval_warps<RPT>() * 32, smem) != cudaSuccess)
        return 0;
    known[dev].store(n + 1, std::memory_order_release);
    return n;
}

template <int RPT, int NSLOT, int FMODE, int EPI, bool EXT>
cudaError_t launch_eval_t(const EvalArgs &a, int grid, int block, cudaStream_t st) {
    constexpr size_t smem = eval_smem_bytes<RPT, NSLOT>();
    if (info_t<RPT, NSLOT, FMODE, EPI, EXT>(block, nullptr) < 1) {
        const cudaError_t e = cudaGetLastError();
        return e != cudaSuccess ? e : cudaErrorInvalidConfiguration;
    }
    return launch_chained(eval_kernel<RPT, NSLOT, FMODE, EPI, EXT>, grid, eval_warps<RPT>() * 32, smem, st,
                          a);
}

}  // namespace gpk
