// Step decisions from exact fixed-point totals with little FP64 work.  An
// FP64 instruction holds a GB300 scheduler for 64 cycles and a division takes
// 1,300, so one decision in plain FP64 takes 5,000 cycles (2.4 us), longer
// than the rest of an iteration of a small problem.
#pragma once
#include "fw_device.cuh"

namespace fw {

// A positive value as (h + l) 2^e with h in [1, 2) and l in [0, 2^-23): 46
// bits, cut off below.
struct Pair {
    float h, l;
    int e;
};
__device__ __forceinline__ Pair pair_of_bits(unsigned long long m, int e) {   // msb of m set
    Pair p;
    p.h = __uint_as_float(0x3f800000u | (uint32_t(m >> 40) & 0x7fffffu));
    p.l = __uint_as_float(0x34000000u | (uint32_t(m >> 17) & 0x7fffffu)) - 0x1p-23f;
    p.e = e;
    return p;
}
__device__ __forceinline__ int msb128(unsigned long long lo, unsigned long long hi) {
    return hi ? 63 - __clzll(static_cast<long long>(hi)) : -1 - __clzll(static_cast<long long>(lo));
}
// of a positive Q64.64 number
__device__ __forceinline__ Pair pair_of_fx(unsigned long long lo, unsigned long long hi) {
    const int e = msb128(lo, hi);
    const int c = 63 - e;   // left shift that brings the msb to bit 127
    unsigned long long m;
    if (c >= 64) m = lo << (c - 64);
    else m = c ? (hi << c) | (lo >> (64 - c)) : hi;
    return pair_of_bits(m, e);
}
// of a positive normal double
__device__ __forceinline__ Pair pair_of_double(double v) {
    const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(v));
    return pair_of_bits((b << 11) | 0x8000000000000000ull, int(b >> 52) - 1023);
}
// 2^d for d in [-126, 127]
__device__ __forceinline__ float exp2_int(int d) { return __uint_as_float(uint32_t(d + 127) << 23); }

// What the quick decision needs besides the totals, prepared once per launch
// (or decision): 2/eps, and the gap threshold once g_0 is known.
struct QuickCfg {
    Pair c2;          // 2/eps
    Pair tol;         // gap_tol, or gap_tol * g_0
    int has_c2;       // 0: eps = inf
    int tol_mode;     // 0: no threshold (gap_tol = 0), 1: tol holds it, 2: not representable here
    int armijo, max_iters;
};
__device__ __forceinline__ bool pair_range(double v) {   // positive, well inside the float exponents
    const int ex = int(static_cast<unsigned long long>(__double_as_longlong(v)) >> 52);   // sign included
    return ex > 1023 - 100 && ex < 1023 + 100;
}
__device__ __forceinline__ QuickCfg quick_cfg(const StepCfg& cfg, double g0) {
    QuickCfg q;
    q.has_c2 = !positive_bits(cfg.inv_eps) ? 0 : pair_range(cfg.inv_eps) ? 1 : 2;
    q.c2 = pair_of_double(cfg.inv_eps);
    ++q.c2.e;
    q.tol_mode = 0;
    q.tol = q.c2;
    if (positive_bits(cfg.gap_tol)) {
        const double tol = cfg.tol_mode ? cfg.gap_tol * g0 : cfg.gap_tol;
        q.tol_mode = pair_range(tol) ? 1 : 2;
        q.tol = pair_of_double(tol);
    }
    q.armijo = cfg.step_rule;
    q.max_iters = cfg.max_iters;
    return q;
}

// The step of decide() as the FP32 update uses it, from the totals as 128-bit
// numbers, without FP64; called by one warp with total q = (lo, hi) in lane q
// and X = <D,LD> + sum w||D||^2 (S5 - S3 + S2, exact) in lane 6.  g, X and
// (2/eps)||D||^2 are taken to 46 bits, so g/q is known to 2^-36 (q may lose 6
// bits to cancellation); its float rounding is returned only when no value
// that close to it rounds differently, which also covers decide()'s own FP64
// roundings.  False when that fails, when the decision might stop the solve,
// or when a value is out of the range handled: the caller then takes decide().
__device__ __forceinline__ bool quick_step(unsigned long long lo, unsigned long long hi, bool flag,
                                           int iter, const QuickCfg& cfg, float& alpha) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool neg = static_cast<long long>(hi) < 0;
    const bool zero = (hi | lo) == 0ull;
    if (neg) {   // |v| - 2^-64: close enough for its leading bit
        hi = ~hi;
        lo = ~lo;
    }
    const Pair v = pair_of_fx(lo, zero ? 1ull : hi);   // positive lanes only
    // no stop: finite totals, active rows, g > 0 and above the threshold, iterations left
    const unsigned need = 1u | (1u << 4) | (1u << 6) | (cfg.has_c2 ? 2u : 0u);
    const unsigned pos = __ballot_sync(full, !neg && !zero);
    if (flag || cfg.has_c2 == 2 || cfg.tol_mode == 2 || iter >= cfg.max_iters ||
        (pos & need) != need)
        return false;
    // the terms of X must not cancel by more than 6 bits
    const int em = __reduce_max_sync(full, (lane == 2 || lane == 3 || lane == 5) && !zero ? v.e : -128);
    Pair g, x, n;
    g.h = __shfl_sync(full, v.h, 0);
    g.l = __shfl_sync(full, v.l, 0);
    g.e = __shfl_sync(full, v.e, 0);
    x.h = __shfl_sync(full, v.h, 6);
    x.l = __shfl_sync(full, v.l, 6);
    x.e = __shfl_sync(full, v.e, 6);
    n.h = __shfl_sync(full, v.h, 1);
    n.l = __shfl_sync(full, v.l, 1);
    n.e = __shfl_sync(full, v.e, 1);
    if (em - x.e > 5) return false;
    if (cfg.tol_mode) {
        const int d = g.e - cfg.tol.e;
        if (d < 0) return false;
        if (d < 2 && !(g.h * exp2_int(d) > cfg.tol.h * (1.0f + 0x1p-20f))) return false;
    }
    float qh = x.h, ql = x.l;
    if (cfg.has_c2) {
        const int d = n.e + cfg.c2.e - x.e;
        if (d >= 2) {   // the penalty term is at least twice X: q < 0
            alpha = 1.0f;
            return true;
        }
        if (d > -60) {
            const float sc = exp2_int(d);
            float th = n.h * cfg.c2.h;
            float tl = __fmaf_rn(n.h, cfg.c2.h, -th);
            tl = __fmaf_rn(n.h, cfg.c2.l, __fmaf_rn(n.l, cfg.c2.h, tl));
            th *= sc;
            tl *= sc;
            qh = __fsub_rn(x.h, th);
            const float bb = __fsub_rn(qh, x.h);
            const float er =
                __fadd_rn(__fsub_rn(x.h, __fsub_rn(qh, bb)), __fsub_rn(-th, bb));
            ql = __fadd_rn(er, __fsub_rn(x.l, tl));
            const float s = __fadd_rn(qh, ql);
            ql = __fsub_rn(ql, __fsub_rn(s, qh));
            qh = s;
            if (qh < -0x1p-6f) {
                alpha = 1.0f;
                return true;
            }
            if (qh < 0x1p-6f) return false;
        }
    }
    // r = g / q 2^(x.e): one Newton correction of the quotient
    float rc;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rc) : "f"(qh));
    const float r1 = __fmul_rn(g.h, rc);
    float rem = __fmaf_rn(-r1, qh, g.h);
    rem = __fadd_rn(rem, __fmaf_rn(-r1, ql, g.l));
    const float r2 = __fmul_rn(rem, rc);
    const float rh = __fadd_rn(r1, r2);
    const float rl = __fsub_rn(r2, __fsub_rn(rh, r1));
    const uint32_t rb = __float_as_uint(rh);
    const int er = int(rb >> 23) - 127;          // rh > 0
    const int e = g.e - x.e;
    if (e + er < -100) return false;
    if (cfg.armijo) {
        // largest 0.5^j <= amax = 2 (1 - 1e-6) r
        const float am = __fmul_rn(rh, 2.0f * (1.0f - 1e-6f));
        const uint32_t ab = __float_as_uint(am);
        const float mant = __uint_as_float((ab & 0x7fffffu) | 0x3f800000u);
        if (mant < 1.0f + 0x1p-20f || mant > 2.0f - 0x1p-20f) return false;
        const int ea = int(ab >> 23) - 127 + e;
        alpha = ea >= 0 ? 1.0f : exp2_int(max(ea, -126));
        return ea > -100;
    }
    if ((rb & 0x7fffffu) == 0u) return false;    // spacing changes at a power of two
    const float half = exp2_int(er - 24);        // half the spacing at rh
    if (!(fabsf(rl) < half * (1.0f - 0x1p-10f))) return false;
    alpha = e + er >= 0 ? 1.0f : rh * exp2_int(e);
    return true;
}

}  // namespace fw
