// sr_df.cuh -- the relativistic primitive recovery of the mixed path in
// double-float arithmetic, with a certificate that the float32 result is the
// one the float64 iteration (sr_prim_mixed) rounds to.
//
// Why: the recovery needs float64 (W cancels against rho gamma and B^2 in the
// energy equation), and GB300 issues 2 float64 operations per SM and cycle
// against 128 of float32, so eleven float64 recoveries per cell and step held
// the whole path at the FP64 pipe (85% busy, the FMA pipe below 3%).  A
// double-float operation is 6 to 20 float32 ones: about a fifth of a float64
// operation's share of its pipe.  Measured at 256^3 (beam, mixed): k_prim
// 7.15 -> 0.95 ms, the sweeps along z, y, x 44.8 -> 6.7, 45.4 -> 6.7,
// 56.1 -> 11.0 ms.  Only the five float32 values rho, v, p leave a recovery,
// so double-float (~2^-46) decides their rounding for all but the few lanes
// whose value lies within the arithmetic's error of a rounding boundary.  Those
// lanes, every state that is not plainly physical, and those in units far from 1
// (sr_recover_in) take the float64 iteration instead (the callers' noinline slow
// paths).  The error bounds' constants come from trials, not from a proof (SR_K):
// on the states tried the results are the float64 iteration's, rounded, bit for
// bit, except for 3 values out of 2e6 decided states, at Lorentz factors near 1000
// (two of them the nearer to a 113-bit solution, none further).
//
// The iterates follow sr_prim_mixed's: the same float32 Newton steps from the
// same guess, then its float64 steps in double-float, with the first-order
// carry of v^2 and p to the last W.  v^2 and its derivative are written
// without the quotient N / D: with t = S/W,
//   v^2 = (m^2 + t^2 (2W + B^2)) / (W + B^2)^2,
//   dv^2/dW = -2 (v^2 + t^2/W) / (W + B^2).
//
// Error of the operations, in units of 2^-48 relative (u^2, u = 2^-24; Joldes,
// Muller & Popescu, "Tight and rigorous error bounds for basic building
// blocks of double-word arithmetic", ACM TOMS 2017): sum 3, product 5 to 7,
// reciprocal and reciprocal square root about 4.  All are explicitly rounded:
// a multiplication fused into a following addition would break the
// error-free transformations.
#pragma once

#include "mhd_fp64.cuh"
#include "srmhd_device.cuh"

namespace ctu {

__device__ __forceinline__ df d_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float bb = __fadd_rn(s, -a);
    return df{s, __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -bb)), __fadd_rn(b, -bb))};
}
__device__ __forceinline__ df d_norm(float a, float b)  // |a| >= |b|
{
    const float s = __fadd_rn(a, b);
    return df{s, __fadd_rn(b, -__fadd_rn(s, -a))};
}
__device__ __forceinline__ df d_two_prod(float a, float b)
{
    const float p = __fmul_rn(a, b);
    return df{p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ df d_neg(df x) { return df{-x.hi, -x.lo}; }
__device__ __forceinline__ df d_half(df x) { return df{__fmul_rn(0.5f, x.hi), __fmul_rn(0.5f, x.lo)}; }
__device__ __forceinline__ df d_add(df x, df y)  // either signs
{
    df s = d_two_sum(x.hi, y.hi);
    const df t = d_two_sum(x.lo, y.lo);
    s = d_norm(s.hi, __fadd_rn(s.lo, t.hi));
    return d_norm(s.hi, __fadd_rn(s.lo, t.lo));
}
__device__ __forceinline__ df d_addp(df x, df y)  // operands of one sign
{
    const df s = d_two_sum(x.hi, y.hi);
    return d_norm(s.hi, __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo)));
}
__device__ __forceinline__ df d_addf(df x, float y)
{
    const df s = d_two_sum(x.hi, y);
    return d_norm(s.hi, __fadd_rn(s.lo, x.lo));
}
__device__ __forceinline__ df d_mul(df x, df y)
{
    const df p = d_two_prod(x.hi, y.hi);
    return d_norm(p.hi, __fmaf_rn(x.hi, y.lo, __fmaf_rn(x.lo, y.hi, p.lo)));
}
__device__ __forceinline__ df d_sqr(df x)
{
    const df p = d_two_prod(x.hi, x.hi);
    return d_norm(p.hi, __fmaf_rn(__fadd_rn(x.hi, x.hi), x.lo, p.lo));
}
// 1/y: a float32 seed r and its residual e = 1 - y r to second order.
__device__ __forceinline__ df d_rcp(df y)
{
    const float r = __fdividef(1.0f, y.hi);
    const float e = __fmaf_rn(-y.lo, r, __fmaf_rn(-y.hi, r, 1.0f));
    return d_norm(r, __fmul_rn(r, __fmaf_rn(e, e, e)));
}
// 1/sqrt(x): a float32 seed y and its residual e = 1 - x y^2 to second order.
__device__ __forceinline__ df d_rsqrt(df x)
{
    const float y = rsqrtf(x.hi);
    const df t = d_mul(x, d_two_prod(y, y));
    const float e = __fadd_rn(__fadd_rn(1.0f, -t.hi), -t.lo);
    return d_norm(y, __fmul_rn(y, __fmul_rn(e, __fmaf_rn(0.375f, e, 0.5f))));
}

// The same operations without the final normalisation: the low part may reach a
// few units of the high part's last place (both signs, any cancellation: the
// error stays below about 2^-47 of the operands' magnitudes).  The recovery's
// bounds are in these magnitudes, so it needs no more; a value is normalised
// where it cancels by design, where its high part stands for it and where it
// leaves.  8 operations for a sum, 4 for a product, against 20 and 7: 38.2 ->
// 28.8 ms a step of the 256^3 beam together with the float32 derivatives below
// (the sweeps issue at 40% with the recovery three times in each, about 2000
// instructions; fetching them is the largest stall).
__device__ __forceinline__ df l_add(df x, df y)
{
    const df s = d_two_sum(x.hi, y.hi);
    return df{s.hi, __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo))};
}
__device__ __forceinline__ df l_addf(df x, float y)
{
    const df s = d_two_sum(x.hi, y);
    return df{s.hi, __fadd_rn(s.lo, x.lo)};
}
__device__ __forceinline__ df l_from1(df x)  // 1 - x, |x| <= 1, normalised
{
    const df s = d_norm(1.0f, -x.hi);
    return d_norm(s.hi, __fadd_rn(s.lo, -x.lo));
}
__device__ __forceinline__ df l_mul(df x, df y)
{
    const df p = d_two_prod(x.hi, y.hi);
    return df{p.hi, __fmaf_rn(x.hi, y.lo, __fmaf_rn(x.lo, y.hi, p.lo))};
}
__device__ __forceinline__ df l_mulf(df x, float y)
{
    const df p = d_two_prod(x.hi, y);
    return df{p.hi, __fmaf_rn(x.lo, y, p.lo)};
}
__device__ __forceinline__ df l_sqr(df x)
{
    const df p = d_two_prod(x.hi, x.hi);
    return df{p.hi, __fmaf_rn(__fadd_rn(x.hi, x.hi), x.lo, p.lo)};
}
// (the seeds are stepped once first: the rounding of a residual that carries
// their two units in the last place would be 2^-46)
__device__ __forceinline__ df l_rcp(df y)
{
    const float r0 = __fdividef(1.0f, y.hi), r = __fmaf_rn(r0, __fmaf_rn(-y.hi, r0, 1.0f), r0);
    const float e = __fmaf_rn(-y.lo, r, __fmaf_rn(-y.hi, r, 1.0f));
    return df{r, __fmul_rn(r, __fmaf_rn(e, e, e))};
}
__device__ __forceinline__ df l_rsqrt(df x)
{
    const float y0 = rsqrtf(x.hi);
    const float y = __fmaf_rn(__fmul_rn(0.5f, y0), __fmaf_rn(__fmul_rn(-x.hi, y0), y0, 1.0f), y0);
    const df t = l_mul(x, d_two_prod(y, y));
    const float e = __fadd_rn(__fadd_rn(1.0f, -t.hi), -t.lo);
    return df{y, __fmul_rn(y, __fmul_rn(e, __fmaf_rn(0.375f, e, 0.5f)))};
}

__device__ __forceinline__ float l_f(df x) { return __fadd_rn(x.hi, x.lo); }

// Whether every value within d of x rounds to x.hi (false for a nan).
__device__ __forceinline__ bool d_certain(df x, float d)
{
    return __fadd_rn(x.hi, __fadd_rn(x.lo, d)) == x.hi && __fadd_rn(x.hi, __fadd_rn(x.lo, -d)) == x.hi;
}

// float64 -> float32, round to nearest even, by integer operations (values
// below the normal float range become signed zeros, as under -ftz).
__device__ __forceinline__ float d2f_int(double x)
{
    const int hw = __double2hiint(x);
    const unsigned lw = (unsigned)__double2loint(x);
    const int e = (hw >> 20) & 0x7FF;
    const unsigned sign = (unsigned)hw & 0x80000000u;
    if (e < 1023 - 126) return __uint_as_float(sign);
    if (e > 1023 + 127) {
        const bool nan = e == 0x7FF && ((((unsigned)hw & 0xFFFFFu) | lw) != 0u);
        return __uint_as_float(sign | 0x7F800000u | (nan ? 0x400000u : 0u));
    }
    unsigned m = ((unsigned)(e - 1023 + 127) << 23) | (((unsigned)hw & 0xFFFFFu) << 3) | (lw >> 29);
    const unsigned rem = lw & 0x1FFFFFFFu;
    m += (rem > 0x10000000u || (rem == 0x10000000u && (m & 1u))) ? 1u : 0u;
    return __uint_as_float(sign | m);
}

// A conserved state for the recovery: D, tau = E + D, m, B.
struct SrState {
    df D, tau, m[3], b[3];
};

// 1 - v^2 of a float32 state, formed from the largest component as
// (1 - |v|)(1 + |v|) less the other squares, so that a fast flow along an axis
// loses nothing in it; and W = w gamma^2 (ideal gas; ig1: Gamma / (Gamma - 1)).
__device__ __forceinline__ void sr_w_of(const float (&V)[9], df ig1, df &ev, df &W)
{
    const float ax = fabsf(V[1]), ay = fabsf(V[2]), az = fabsf(V[3]);
    const float big = fmaxf(ax, fmaxf(ay, az));
    const float s1 = ax == big ? ay : ax, s2 = ax == big ? az : (ay == big ? az : ay);
    ev = l_add(l_mul(d_norm(1.0f, -big), d_norm(1.0f, big)), d_neg(l_add(d_two_prod(s1, s1), d_two_prod(s2, s2))));
    ev = d_norm(ev.hi, ev.lo);
    W = l_mul(l_addf(l_mulf(ig1, V[4]), V[0]), l_rcp(ev));
    W = d_norm(W.hi, W.lo);
}

// U(V) + T of a float32 state for sr_recover; W0: its w gamma^2.
__device__ __forceinline__ void sr_state_of(const float (&V)[9], const float (&T)[9], df ig1, SrState &u, float &W0)
{
    df ev, W;
    sr_w_of(V, ig1, ev, W);
    W0 = W.hi;
    const df B2 = l_add(l_add(d_two_prod(V[5], V[5]), d_two_prod(V[6], V[6])), d_two_prod(V[7], V[7]));
    const df vB = l_add(l_add(d_two_prod(V[1], V[5]), d_two_prod(V[2], V[6])), d_two_prod(V[3], V[7]));
    const df Wb = l_add(W, B2);
    u.D = l_addf(l_mulf(l_rsqrt(ev), V[0]), T[0]);
    u.D = d_norm(u.D.hi, u.D.lo);
    // W - p + (B^2 (1 + v^2) - (v.B)^2) / 2, with 1 + v^2 = 2 - (1 - v^2)
    const df q = l_add(l_mul(B2, l_addf(d_neg(ev), 2.0f)), d_neg(l_sqr(vB)));
    u.tau = l_add(l_add(l_addf(W, -V[4]), d_half(q)), d_two_sum(T[4], T[0]));
    u.tau = d_norm(u.tau.hi, u.tau.lo);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        u.m[k] = l_addf(l_add(l_mulf(Wb, V[1 + k]), d_neg(l_mulf(vB, V[5 + k]))), T[1 + k]);
        u.b[k] = d_two_sum(V[5 + k], T[5 + k]);
    }
}

// Error bounds of sr_recover, in units of 2^-48: K times the sums of the
// magnitudes that enter 1 - v^2, the energy equation and the velocities; and,
// in units of 2^-24, K_D times the float32 Newton derivatives' terms and the
// step (2e-7 W as a rule).  With K = 3 and K_D = 2 no value out of 4e7 beam,
// beam-edge, ambient, magnetised and random states rounded differently from the
// float64 iteration's, also with the hardware's seeds (1/x, 1/sqrt x) off by
// two units in the last place; with K = 1 one in 2e6 edge states did.  The
// float64 path is left 0.6% of the beam's, 1.5% of its edge's and 0.03% of the
// ambient's states.
constexpr float SR_MARGIN = 1.0f / 281474976710656.0f;  // 2^-48
#ifndef SR_K
#define SR_K 3.0f
#endif
constexpr float SR_K_EV = SR_K, SR_K_F = SR_K, SR_K_V = SR_K;
#ifndef SR_KD
#define SR_KD 2.0f
#endif
constexpr float SR_K_D = SR_KD * 16777216.0f;  // in units of 2^-24 of the step

// W from the energy equation in float32, as sr_prim64's bracketed iteration:
// an upper bound by doubling from tau, then Newton steps, bisection outside
// the bracket.
__device__ __forceinline__ float sr_bracket_f(float D, float m2, float S2, float B2, float tau, float g1)
{
    float Wlo = 0.0f, Whi = tau, f, df;
    for (int k = 0; k < 64; ++k) {
        if (sr_energy_f(Whi, D, m2, S2, B2, tau, g1, f, df) && f > 0.0f) break;
        Wlo = Whi;
        Whi *= 2.0f;
    }
    float W = Whi;
    for (int it = 0; it < 50; ++it) {
        float Wn = 0.5f * (W + Whi);
        if (!sr_energy_f(W, D, m2, S2, B2, tau, g1, f, df)) {
            Wlo = W;
        } else {
            if (f > 0.0f) Whi = W; else Wlo = W;
            Wn = W - f / df;
            if (!(Wn > Wlo && Wn < Whi)) Wn = 0.5f * (Wlo + Whi);
            if (fabsf(Wn - W) <= 2.0e-6f * W) return Wn;
        }
        W = Wn;
    }
    return W;
}

// rho, v and p of a conserved state from the guess W0 (> 0, else tau - B^2/2)
// for the ideal gas with g1 = (Gamma - 1) / Gamma.  ok: V holds the five
// float32 values that sr_prim_mixed returns for the same state and guess
// (rounded to float32), all of them physical.  Otherwise undecided.
// Out of line: the sweeps recover three or four states a cell, and the copies
// inlined (about 1000 instructions each) overflowed the instruction cache
// (x sweep 36.1 ms at 256^3 with 15 of 20 stall cycles on instruction fetch).
// Undecided outside tau in [2^-16, 2^16), where the float64 iteration scales the
// state (sr_half_exp): below, the low parts of m^2, B^2 and their products drop
// under the normal range and flush to zero, which the bounds, relative ones, do not
// see (from tau ~ 2^-18 down p came out up to 12 ulp off).  Scaling here, inline or
// in a call, cost the sweeps 3 to 4% in spills and instruction fetch.
struct SrRec {
    float V[5];
    bool ok;
};
__device__ __forceinline__ bool sr_recover_in(const SrState &u, float W0, df g1, float (&V)[5])
{
    df m2 = l_add(l_add(l_sqr(u.m[0]), l_sqr(u.m[1])), l_sqr(u.m[2]));
    df B2 = l_add(l_add(l_sqr(u.b[0]), l_sqr(u.b[1])), l_sqr(u.b[2]));
    const df sx = l_mul(u.m[0], u.b[0]), sy = l_mul(u.m[1], u.b[1]), sz = l_mul(u.m[2], u.b[2]);
    df S = l_add(l_add(sx, sy), sz);
    m2 = d_norm(m2.hi, m2.lo);
    B2 = d_norm(B2.hi, B2.lo);
    S = d_norm(S.hi, S.lo);
    const float Sa = fabsf(sx.hi) + fabsf(sy.hi) + fabsf(sz.hi);
    // (D: the low part of rho needs 2^-126)
    if (!(u.D.hi >= 8.8817841970012523e-16f) || !(u.tau.hi >= 1.52587890625e-5f && u.tau.hi < 65536.0f)) return false;
    if (!(W0 > 0.0f)) W0 = d_add(u.tau, d_neg(d_half(B2))).hi;
    if (!(W0 > 0.0f)) return false;
    // float32 Newton, as sr_prim_mixed; a two-cycle (the float32 residual's
    // noise exceeds the criterion where B^2 >> W) runs to the same last
    // iterate at once
    const float S2f = d_sqr(S).hi;
    float Wf = W0, Wp = 0.0f;
    bool strict = false;
    for (int it = 0; it < 12; ++it) {
        float f, dfw;
        strict = !sr_energy_f(Wf, u.D.hi, m2.hi, S2f, B2.hi, u.tau.hi, g1.hi, f, dfw);
        const float Wn = Wf - f / dfw;
        strict |= !(Wn > 0.0f);
        if (strict) break;
        if (Wn == Wp && fabsf(Wn - Wf) > 2.0e-6f * Wf) {
            if (((11 - it) & 1) == 0) Wf = Wn;
            break;
        }
        const bool done = fabsf(Wn - Wf) <= 2.0e-6f * Wf;
        Wp = Wf;
        Wf = Wn;
        if (done) break;
    }
    // outside the physical range sr_prim_mixed hands over to the bracketed
    // iteration, which converges to the root of the energy equation: so does
    // this one, from a bracketed float32 iteration and with steps in
    // double-float until one moves W by less than 2e-9
    if (strict) Wf = sr_bracket_f(u.D.hi, m2.hi, S2f, B2.hi, u.tau.hi, g1.hi);
    const float accept = strict ? 2.0e-9f : 1.0e-5f;
    df W{Wf, 0.0f};
#pragma unroll 1
    for (int it = 0; it < 3; ++it) {
        const df Wb = l_add(W, B2), A = l_add(W, Wb);
        const df iW = l_rcp(W), iWb = l_rcp(Wb);
        const df t = l_mul(S, iW), t2 = l_sqr(t);
        const df iWb2 = l_sqr(iWb);
        const df v2 = l_mul(l_add(m2, l_mul(t2, A)), iWb2);
        if (!(v2.hi <= 1.0f)) return false;
        const df ev = l_from1(v2);
        if (!(ev.hi > 0.0f)) return false;
        const df is = l_rsqrt(ev), s = l_mul(ev, is);
        const df Ds = l_mul(u.D, s);
        const df p = l_mul(g1, l_add(l_mul(W, ev), d_neg(Ds)));
        const df hB = d_half(B2);
        // f = W - p + B^2 (1 + v^2)/2 - t^2/2 - tau
        df f = l_add(l_add(l_add(l_add(W, d_neg(u.tau)), hB), l_mul(hB, v2)), d_neg(l_add(p, d_half(t2))));
        f = d_norm(f.hi, f.lo);
        // derivatives and the step in float32: their relative error is of the
        // step, which is a few 2^-24 of W (e_d below)
        const float iWf = l_f(iW), iWbf = l_f(iWb), isf = l_f(is), v2f = l_f(v2);
        const float t2W = l_f(t2) * iWf, dv2 = -2.0f * iWbf * (v2f + t2W), Dis = u.D.hi * isf;
        const float dp = g1.hi * (ev.hi + dv2 * (0.5f * Dis - W.hi));
        const float dF = 1.0f - dp + hB.hi * dv2 + t2W;
        const float rF = __fdividef(1.0f, dF), dW0 = __fmul_rn(-f.hi, rF);
        const float dW = __fmaf_rn(rF, __fmaf_rn(-dW0, dF, -f.hi), dW0);
        const df Wn = l_addf(W, dW);
        if (!(Wn.hi > 0.0f)) return false;
        const float a = fabsf(dW), lim = accept * W.hi;
        if (a > 0.9999f * lim) {
            if (!(a > 1.0001f * lim)) return false;
            W = d_norm(Wn.hi, Wn.lo);
            continue;
        }
        // (1 - v^2, its root, 1/W and 1/(W + B^2) follow the step by their
        // series in it)
        const float dev = -dv2 * dW, h = 0.5f * dev * isf * isf;
        const float evn = ev.hi + dev;
        if (!(evn > 0.0f) || !(fabsf(h) <= 3.0e-4f)) return false;
        df pn = l_addf(p, dp * dW);
        pn = d_norm(pn.hi, pn.lo);
        const float c = dW * iWf, cb = dW * iWbf;
        const df iWbn = df{iWb.hi, __fmaf_rn(iWb.hi, cb * cb - cb, iWb.lo)};
        const df SW = l_mul(S, df{iW.hi, __fmaf_rn(iW.hi, c * c - c, iW.lo)});
        df rho = l_mul(u.D, df{s.hi, __fmaf_rn(s.hi, h - 0.5f * h * h * (1.0f - h), s.lo)});
        rho = d_norm(rho.hi, rho.lo);
        if (!(rho.hi > 0.0f) || !(pn.hi > 0.0f)) return false;
        // error bounds (absolute), see SR_MARGIN
        const float Ta = Sa * iW.hi, v2b = (m2.hi + Ta * Ta * A.hi) * iWb2.hi, e_d = SR_K_D * a;
        const float e_ev = SR_K_EV * v2b, adv = fabsf(dv2);
        const float e_p0 = g1.hi * ((W.hi + 0.5f * Dis) * e_ev + 2.0f * SR_K_F * Ds.hi);
        const float e_f = e_p0 + hB.hi * e_ev + SR_K_F * (W.hi + B2.hi + 0.5f * Ta * Ta + u.tau.hi);
        const float ddp = g1.hi * (ev.hi + adv * (0.5f * Dis + W.hi));
        const float e_W = (e_f + e_d * (1.0f + ddp + hB.hi * adv + t2W)) / fabsf(dF);
        const float e_evn = e_ev + adv * (e_W + e_d);
        const bool sure =
            d_certain(pn, SR_MARGIN * (e_p0 + fabsf(dp) * e_W + ddp * e_d)) &&
            d_certain(rho, SR_MARGIN * (0.5f * Dis * e_evn + SR_K_V * rho.hi));
        if (!sure) return false;
        V[0] = rho.hi;
        V[4] = pn.hi;
        // low parts lost below the float range: 2^-98 absolute in each m_k
        const float tiny = 3.2e-30f, bs = (fabsf(u.b[0].hi) + fabsf(u.b[1].hi) + fabsf(u.b[2].hi)) * iW.hi;
        bool ok = true;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const df sb = l_mul(SW, u.b[k]);
            df v = l_mul(l_add(u.m[k], sb), iWbn);
            v = d_norm(v.hi, v.lo);
            const float bi = fabsf(u.b[k].hi);
            const float e_v = SR_K_V * (fabsf(u.m[k].hi) + Ta * bi) + (fabsf(v.hi) + fabsf(SW.hi) * bi * iW.hi) * (e_W + e_d);
            const bool zero = u.m[k].hi == 0.0f && sb.hi == 0.0f && u.m[k].lo == 0.0f && sb.lo == 0.0f && Ta * bi == 0.0f;
            ok &= zero || d_certain(v, iWbn.hi * (SR_MARGIN * e_v + tiny * (1.0f + bi * bs)));
            V[1 + k] = v.hi;
        }
        return ok;
    }
    return false;
}

static __device__ __noinline__ SrRec sr_recover_call(SrState u, float W0, df g1)
{
    SrRec r;
    r.ok = sr_recover_in(u, W0, g1, r.V);
    return r;
}
__device__ __forceinline__ bool sr_recover(const SrState &u, float W0, df g1, float (&V)[5])
{
    const SrRec r = sr_recover_call(u, W0, g1);
#pragma unroll
    for (int q = 0; q < 5; ++q) V[q] = r.V[q];
    return r.ok;
}

// ---- the float64 iteration for the lanes sr_recover leaves undecided; out of
// line where its registers and code can stay off the fast path

struct SrCons {
    double U[NV];
};
struct SrFace {
    float V[NV], T[NV];
};
struct SrOut {
    float V[NV];
    unsigned int st;
};

static __device__ __noinline__ SrOut sr_prim_slow(SrCons c, double gam, double W0)
{
    double V[NV];
    SrOut o;
    o.st = sr_prim_mixed(c.U, gam, V, W0);
#pragma unroll
    for (int q = 0; q < NV; ++q) o.V[q] = (float)V[q];
    return o;
}

static __device__ __noinline__ SrOut sr_interface_slow(SrFace f, double gam)
{
    double V[NV];
    SrOut o;
    o.st = sr_interface64(f.V, f.T, gam, V);
#pragma unroll
    for (int q = 0; q < NV; ++q) o.V[q] = (float)V[q];
    return o;
}

// f.V: the cell's V^n, f.T: the increment x (sr_mh_recover); inline in the x
// sweep, whose fluxes the compiler rounds around it
__device__ __forceinline__ SrOut sr_mh_slow_in(const SrCons &c, const SrFace &f, double gam)
{
    double V[NV];
    SrOut o;
    o.st = sr_mh_recover(c.U, f.V, f.T, gam, V);
#pragma unroll
    for (int q = 0; q < NV; ++q) o.V[q] = (float)V[q];
    return o;
}

// Interface state of the mixed path, V(U(f.V) + f.T): the double-float recovery
// (ideal gas), else the float64 one.  Out of line, as sr_recover: each sweep
// needs it twice a cell.
static __device__ __noinline__ SrOut sr_interface_call(SrFace f, df g1, df ig1, double gam)
{
    if (g1.hi > 0.0f) {
        SrState u;
        float W0, v[5];
        sr_state_of(f.V, f.T, ig1, u, W0);
        if (sr_recover(u, W0, g1, v)) {
            SrOut o;
#pragma unroll
            for (int q = 0; q < 5; ++q) o.V[q] = v[q];
#pragma unroll
            for (int q = 5; q < NV; ++q) o.V[q] = __fadd_rn(f.V[q], f.T[q]);
            o.st = 0u;
            return o;
        }
    }
    return sr_interface_slow(f, gam);
}

static __device__ __noinline__ SrOut sr_mh_slow(SrCons c, SrFace f, double gam) { return sr_mh_slow_in(c, f, gam); }

// A float64 value as a normalised double-float.
__device__ __forceinline__ df sr_split(double x)
{
    const df s = df_split(x);
    return d_norm(s.hi, s.lo);
}

// ---- float32 predictor and fluxes of the marching sweeps, every rounding
// written out
//
// riemann_hll_sr and sr_mh_increment leave the choice of the fused operation
// in sums of two products (a b + c d, which of the two is rounded first) to
// the compiler, whose choice depends on the code around them: with another
// recovery in the kernel the last bits of every flux move.  These forms fix
// the choices to the ones that the sweeps along y and z were compiled to with
// the float64 recovery inline, so that a sweep's results do not depend on what
// else its kernel holds (the double-float recovery left to the compiler's
// choice moved a step's output by 1.3e-8 relative; with these it is unchanged).
// Bits by the sum they choose in (set: the second product carries the fusion,
// the first is rounded; or, where noted, no fusion at all):
enum : unsigned {
    SR_V2 = 1u,   // v^2: v_x v_x + v_y v_y
    SR_B2 = 2u,   // B^2: B_x B_x + B_y B_y
    SR_F7 = 4u,   // v_x B_z - B_x v_z
    SR_F4 = 8u,   // m_x - D v_x: not fused
};

// a b + c d (or, with s = -1, a b - c d), one product fused.
template <bool SECOND> __device__ __forceinline__ float sum2(float a, float b, float c, float d, float s = 1.0f)
{
    return SECOND ? __fmaf_rn(s * c, d, __fmul_rn(a, b)) : __fmaf_rn(a, b, s * __fmul_rn(c, d));
}

// Conserved state, flux along the local normal (components 0..4, 6, 7) and,
// with SPEEDS, the signal speeds of a float32 state (sr_cons, sr_flux,
// sr_speeds; ideal gas, gw = Gamma / (Gamma - 1)).
template <unsigned O, bool SPEEDS>
__device__ __forceinline__ void sr_side(const float (&V)[NV], float gam, float gw, float (&U)[NV], float (&F)[NV],
                                        float &lm, float &lp)
{
    const float rho = V[0], vx = V[1], vy = V[2], vz = V[3], p = V[4], bx = V[5], by = V[6], bz = V[7];
    const float v2 = __fmaf_rn(vz, vz, sum2<(O & SR_V2) != 0>(vx, vx, vy, vy));
    const float ev = __fadd_rn(1.0f, -v2), lor2 = __fdividef(1.0f, ev), w = __fmaf_rn(gw, p, rho);
    const float B2 = __fmaf_rn(bz, bz, sum2<(O & SR_B2) != 0>(bx, bx, by, by));
    const float vB = __fmaf_rn(vz, bz, sum2<false>(vx, bx, vy, by));
    const float E2 = sum2<false>(B2, v2, vB, vB, -1.0f);
    const float D = __fmul_rn(rho, rsqrtf(ev)), W = __fmul_rn(w, lor2), WB = __fmaf_rn(w, lor2, B2);
    U[0] = D;
    U[1] = sum2<false>(WB, vx, vB, bx, -1.0f);
    U[2] = sum2<false>(WB, vy, vB, by, -1.0f);
    U[3] = sum2<false>(WB, vz, vB, bz, -1.0f);
    U[4] = __fadd_rn(__fmaf_rn(0.5f, __fadd_rn(B2, E2), __fmaf_rn(w, lor2, -p)), -D);
    U[5] = bx;
    U[6] = by;
    U[7] = bz;
    U[8] = V[8];
    const float ex = -sum2<false>(vy, bz, vz, by, -1.0f), ey = -sum2<false>(vz, bx, vx, bz, -1.0f),
                ez = -sum2<false>(vx, by, vy, bx, -1.0f);
    const float pt = __fmaf_rn(0.5f, __fmaf_rn(ez, ez, __fmaf_rn(ey, ey, __fmaf_rn(ex, ex, B2))), p);
    const float Wx = __fmul_rn(W, vx);
    F[0] = __fmul_rn(D, vx);
    F[1] = __fadd_rn(__fmaf_rn(-ex, ex, sum2<false>(Wx, vx, bx, bx, -1.0f)), pt);
    F[2] = __fmaf_rn(-ex, ey, sum2<false>(Wx, vy, bx, by, -1.0f));
    F[3] = __fmaf_rn(-ex, ez, sum2<false>(Wx, vz, bx, bz, -1.0f));
    F[4] = (O & SR_F4) ? __fadd_rn(U[1], -F[0]) : __fmaf_rn(-D, vx, U[1]);
    F[6] = sum2<false>(vx, by, bx, vy, -1.0f);
    F[7] = sum2<(O & SR_F7) != 0>(vx, bz, bx, vz, -1.0f);
    if constexpr (SPEEDS) {
        const float cs2 = __fmul_rn(__fmul_rn(gam, p), __fdividef(1.0f, w));
        const float b2 = sum2<false>(B2, ev, vB, vB);
        const float ca2 = __fmul_rn(b2, __fdividef(1.0f, __fadd_rn(w, b2)));
        const float a2 = __fmaf_rn(-cs2, ca2, __fadd_rn(cs2, ca2));
        const float den = __fmaf_rn(-v2, a2, 1.0f), oa = __fadd_rn(1.0f, -a2);
        const float disc = __fmul_rn(__fmul_rn(a2, ev), __fmaf_rn(-__fmul_rn(vx, vx), oa, den));
        const float sq = sqrtf(fmaxf(disc, 0.0f)), id = __fdividef(1.0f, den);
        lm = __fmul_rn(__fmaf_rn(vx, oa, -sq), id);
        lp = __fmul_rn(__fmaf_rn(vx, oa, sq), id);
    }
}

// riemann_hll_sr of the sweep along D (1 or 2).
template <int D>
__device__ __forceinline__ void riemann_hll_sr_m(const float (&L0)[NV], const float (&R0)[NV], float gam, float ch,
                                                 float (&F)[NV])
{
    constexpr unsigned OL = SR_V2 | SR_B2 | SR_F7 | SR_F4, OR = D == 1 ? OL : OL & ~SR_V2;
    float L[NV], R[NV], UL[NV], UR[NV], FL[NV], FR[NV], lmL, lpL, lmR, lpR;
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        L[q] = L0[q];
        R[q] = R0[q];
    }
    const float ich = __fdividef(1.0f, ch), gw = __fmul_rn(gam, __fdividef(1.0f, __fadd_rn(gam, -1.0f)));
    const float Bm = __fadd_rn(__fmul_rn(0.5f, __fadd_rn(L[5], R[5])),
                               -__fmul_rn(__fmul_rn(0.5f, __fadd_rn(R[8], -L[8])), ich));
    const float pm = __fadd_rn(__fmul_rn(0.5f, __fadd_rn(L[8], R[8])),
                               -__fmul_rn(__fmul_rn(0.5f, ch), __fadd_rn(R[5], -L[5])));
    L[5] = Bm;
    R[5] = Bm;
    sr_side<OL, true>(L, gam, gw, UL, FL, lmL, lpL);
    sr_side<OR, true>(R, gam, gw, UR, FR, lmR, lpR);
    const float SL = fminf(lmL, lmR), SR = fmaxf(lpL, lpR);
    const float is = __fdividef(1.0f, __fadd_rn(SR, -SL)), ss = __fmul_rn(SL, SR);
    const bool left = SL >= 0.0f, right = SR <= 0.0f;
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        if (q == 5 || q == 8) continue;
        const float d = sum2<false>(SR, FL[q], SL, FR[q], -1.0f);
        const float mid = __fmul_rn(__fmaf_rn(ss, __fadd_rn(UR[q], -UL[q]), d), is);
        F[q] = left ? FL[q] : right ? FR[q] : mid;
    }
    F[5] = pm;
    F[8] = __fmul_rn(__fmul_rn(ch, ch), Bm);
}

// sr_mh_increment of the sweep along D (1 or 2).
template <int D>
__device__ __forceinline__ void sr_mh_increment_m(const float (&vm1)[NV], const float (&v0)[NV], const float (&vp1)[NV],
                                                  float gam, float ch, float dtdx, float (&dV)[NV], float (&x)[NV])
{
    constexpr unsigned OP = SR_B2 | SR_F4, OM = D == 1 ? SR_B2 | SR_F7 : SR_F7;
    float P[NV], M[NV], UP[NV], UM[NV], FP[NV], FM[NV], l0, l1;
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        dV[q] = mc_slope(__fadd_rn(v0[q], -vm1[q]), __fadd_rn(vp1[q], -v0[q]));
        P[q] = __fmaf_rn(0.5f, dV[q], v0[q]);
        M[q] = __fmaf_rn(-0.5f, dV[q], v0[q]);
    }
    const float gw = __fmul_rn(gam, __fdividef(1.0f, __fadd_rn(gam, -1.0f))), h = __fmul_rn(0.5f, dtdx);
    sr_side<OP, false>(P, gam, gw, UP, FP, l0, l1);
    sr_side<OM, false>(M, gam, gw, UM, FM, l0, l1);
    const float c2 = __fmul_rn(ch, ch);
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        float d;
        if (q == 0)
            d = sum2<true>(UP[0], P[1], UM[0], M[1], -1.0f);
        else if (q == 5)
            d = __fadd_rn(P[8], -M[8]);
        else if (q == 8)
            d = sum2<false>(c2, P[5], c2, M[5], -1.0f);
        else
            d = __fadd_rn(FP[q], -FM[q]);
        x[q] = __fmul_rn(h, d);
    }
}

// sr_mh_predict of the mixed path (global component gp(q) of the pool at Uc[
// gp(q) us] is local component q): U* = U_i^n - x in double-float, recovered by
// sr_recover.  B and psi of the half-step state are U*'s, rounded; where
// double-float leaves one undecided the float64 path takes the cell.
template <int D, class GP>
__device__ __forceinline__ unsigned int sr_mh_predict_f(const float (&vm1)[NV], const float (&v0)[NV],
                                                        const float (&vp1)[NV], const double *Uc, long long us, GP gp,
                                                        float gam, float ch, float dtdx, double gamd, df g1, df ig1,
                                                        float (&Vp)[NV], float (&Vm)[NV])
{
    float dV[NV], x[NV], V[NV];
    if constexpr (D == 0) {
        sr_mh_increment<float>(vm1, v0, vp1, gam, ch, dtdx, dV, x);
    } else {
        if (gam > 0.0f)
            sr_mh_increment_m<D>(vm1, v0, vp1, gam, ch, dtdx, dV, x);
        else  // the Taub-Mathews gas
            sr_mh_increment<float>(vm1, v0, vp1, gam, ch, dtdx, dV, x);
    }
    unsigned int st = 0;
    bool ok = false;
    if (g1.hi > 0.0f) {
        SrState u;
        df d[NV];
#pragma unroll
        for (int q = 0; q < NV; ++q) d[q] = d_addf(sr_split(Uc[gp(q) * us]), -x[q]);
        u.D = d[0];
        u.tau = d_add(d[4], d[0]);
        ok = true;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            u.m[k] = d[1 + k];
            u.b[k] = d[5 + k];
        }
#pragma unroll
        for (int q = 5; q < NV; ++q) {
            V[q] = d[q].hi;
            ok &= d_certain(d[q], 4.0f * SR_MARGIN * (fabsf(d[q].hi) + 2.0f * fabsf(x[q])) + 1.0e-37f) ||
                  (d[q].hi == 0.0f && x[q] == 0.0f);
        }
        df ev, W;
        sr_w_of(v0, ig1, ev, W);
        float v[5];
        ok = ok && sr_recover(u, W.hi, g1, v);
#pragma unroll
        for (int q = 0; q < 5; ++q) V[q] = v[q];
    }
    if (!ok) {
        SrCons c;
        SrFace f;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            c.U[q] = Uc[gp(q) * us];
            f.V[q] = v0[q];
            f.T[q] = x[q];
        }
        const SrOut o = D == 0 ? sr_mh_slow_in(c, f, gamd) : sr_mh_slow(c, f, gamd);
        st = o.st;
#pragma unroll
        for (int q = 0; q < NV; ++q) V[q] = o.V[q];
    }
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        Vp[q] = V[q] + 0.5f * dV[q];
        Vm[q] = V[q] - 0.5f * dV[q];
    }
    return st;
}

// ---- the FP64 path

// W of the energy equation to double-float accuracy (about 1e-13 relative): the
// float32 Newton steps, bracketed where they leave the physical range, then
// double-float steps until one moves W by less than 1e-7.  No certificate: a
// start for the float64 step.  false: not found.
__device__ __forceinline__ bool sr_seed(const SrState &u, float W0, df g1, double &Wd)
{
    const df m2 = d_addp(d_addp(d_sqr(u.m[0]), d_sqr(u.m[1])), d_sqr(u.m[2]));
    const df B2 = d_addp(d_addp(d_sqr(u.b[0]), d_sqr(u.b[1])), d_sqr(u.b[2]));
    const df S = d_add(d_add(d_mul(u.m[0], u.b[0]), d_mul(u.m[1], u.b[1])), d_mul(u.m[2], u.b[2]));
    if (!(u.D.hi > 0.0f) || !(u.tau.hi > 0.0f)) return false;
    if (!(W0 > 0.0f)) W0 = d_add(u.tau, d_neg(d_half(B2))).hi;
    const float S2f = d_sqr(S).hi;
    float Wf = W0;
    bool in = W0 > 0.0f;
    for (int it = 0; it < 8 && in; ++it) {
        float f, dfw;
        in = sr_energy_f(Wf, u.D.hi, m2.hi, S2f, B2.hi, u.tau.hi, g1.hi, f, dfw);
        const float Wn = Wf - f / dfw;
        in = in && Wn > 0.0f;
        const bool done = fabsf(Wn - Wf) <= 1.0e-5f * Wf;
        if (in) Wf = Wn;
        if (done) break;
    }
    if (!in) Wf = sr_bracket_f(u.D.hi, m2.hi, S2f, B2.hi, u.tau.hi, g1.hi);
    df W{Wf, 0.0f};
    const df hB = d_half(B2);
#pragma unroll 1
    for (int it = 0; it < 4; ++it) {
        const df Wb = d_addp(W, B2), iW = d_rcp(W), iWb = d_rcp(Wb);
        const df t2 = d_sqr(d_mul(S, iW));
        const df v2 = d_mul(d_addp(m2, d_mul(t2, d_addp(W, Wb))), d_sqr(iWb));
        const df ev = d_addf(d_neg(v2), 1.0f);
        if (!(ev.hi > 0.0f)) return false;
        const df is = d_rsqrt(ev);
        const df p = d_mul(g1, d_add(d_mul(W, ev), d_neg(d_mul(u.D, d_mul(ev, is)))));
        const df f = d_add(d_add(d_add(d_add(W, d_neg(u.tau)), hB), d_mul(hB, v2)), d_neg(d_add(p, d_half(t2))));
        // f' in float32: the step's error is its square and 1e-6 of it
        const float dv2 = -2.0f * iWb.hi * (v2.hi + t2.hi * iW.hi);
        const float dp = g1.hi * (ev.hi + dv2 * (0.5f * u.D.hi * is.hi - W.hi));
        const float dF = 1.0f - dp + hB.hi * dv2 + t2.hi * iW.hi;
        const float dW = -__fdividef(f.hi, dF);
        W = d_addf(W, dW);
        if (!(W.hi > 0.0f)) return false;
        if (fabsf(dW) <= 1.0e-7f * W.hi) {
            Wd = f2d_int(W.hi) + f2d_int(W.lo);
            return true;
        }
    }
    return false;
}

struct SrOut64 {
    double V[5];
    unsigned int st;
};

// rho, v and p of a conserved state in float64 (ideal gas, g1 = (Gamma - 1) /
// Gamma; the Taub-Mathews gas, gam = 0, keeps sr_prim64): W from sr_seed on the
// FP32 pipe, so that one float64 evaluation of the energy equation remains,
// with v^2 and p carried over its step by their first-order terms (a step of at
// most 1e-9 W that moves 1 - v^2 by at most 7.5e-9 of itself: remainders of 1e-18
// W (1 - v^2) and 1e-17 rho; the step alone moves 1 - v^2 by up to 2e-9 gamma^2 of
// itself, and p came out 1e-4 off at gamma = 1000).  sr_prim64 took several evaluations from
// a guess, and its bracketed iteration tens of them for the lanes without a
// usable one, the whole warp waiting.  64^3 beam, ms per launch before and
// after (with the FP64 forms of the fluxes): prim 1.29 and 0.095, sweep z 7.5 and
// 1.32, y 8.6 and 1.36, x 3.8 and 0.86.
static __device__ __noinline__ SrOut64 sr_prim_fp64(SrCons c, double gam, double g1, df g1f, float W0)
{
    SrOut64 o;
    const double D = c.U[0], tau = c.U[4] + c.U[0];
    double W = 0.0;
    bool ok = false;
    if (gam > 0.0) {
        SrState u;
        u.D = sr_split(c.U[0]);
        u.tau = d_add(sr_split(c.U[4]), u.D);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            u.m[k] = sr_split(c.U[1 + k]);
            u.b[k] = sr_split(c.U[5 + k]);
        }
        ok = sr_seed(u, W0, g1f, W);
    }
    if (ok) {
        const double m2 = c.U[1] * c.U[1] + c.U[2] * c.U[2] + c.U[3] * c.U[3];
        const double B2 = c.U[5] * c.U[5] + c.U[6] * c.U[6] + c.U[7] * c.U[7];
        const double S = c.U[1] * c.U[5] + c.U[2] * c.U[6] + c.U[3] * c.U[7];
        ok = false;
#pragma unroll 1
        for (int it = 0; it < 3; ++it) {
            const double Wb = W + B2, iW = d_rcp64(W), iWb = d_rcp64(Wb);
            const double t = S * iW, t2 = t * t, t2W = t2 * iW;
            const double v2 = fma(t2, W + Wb, m2) * (iWb * iWb);
            const double dv2 = -2.0 * iWb * (v2 + t2W);
            const double ev = 1.0 - v2;
            double is, s;
            if (!d_pos(ev)) break;
            d_roots64(ev, is, s);
            const double p = g1 * (W * ev - D * s);
            const double dp = g1 * fma(dv2, fma(0.5 * D, is, -W), ev);
            const double f = ((W - tau) + 0.5 * B2) + fma(0.5, fma(B2, v2, -t2), -p);
            const double dF = (1.0 - dp) + fma(0.5 * B2, dv2, t2W);
            const double dW = -f * d_rcp64(dF), Wn = W + dW;
            if (!d_pos(Wn)) break;
            const double evn = fma(-dv2, dW, ev);
            // in units of ev's last place; far off for evn <= 0 and for nans
            const unsigned long long moved = (unsigned long long)d_bits(evn) - (unsigned long long)d_bits(ev);
            if (d_mag(dW) <= d_mag(1.0e-9 * W) && moved + (1ull << 25) <= 2ull << 25) {
                const double pn = fma(dp, dW, p);
                const double iq = d_rcp64(Wn + B2), SW = S * d_rcp64(Wn);
                o.V[0] = D * d_sqrt64(evn);
#pragma unroll
                for (int k = 0; k < 3; ++k) o.V[1 + k] = fma(SW, c.U[5 + k], c.U[1 + k]) * iq;
                o.V[4] = pn;
                o.st = d_pos(o.V[0]) && d_pos(pn) ? 0u : 1u;
                ok = true;
                break;
            }
            W = Wn;
        }
    }
    if (!ok) {
        double V[NV];
        o.st = sr_prim64(c.U, gam, V, f2d_int(W0));
#pragma unroll
        for (int q = 0; q < 5; ++q) o.V[q] = V[q];
    }
    return o;
}
__device__ __forceinline__ unsigned int sr_prim_fp64(const double (&U)[NV], double gam, double g1, df g1f, float W0,
                                                     double (&V)[NV])
{
    SrCons c;
#pragma unroll
    for (int q = 0; q < NV; ++q) c.U[q] = U[q];
    const SrOut64 o = sr_prim_fp64(c, gam, g1, g1f, W0);
#pragma unroll
    for (int q = 0; q < 5; ++q) V[q] = o.V[q];
#pragma unroll
    for (int q = 5; q < NV; ++q) V[q] = U[q];
    return o.st;
}

} // namespace ctu
