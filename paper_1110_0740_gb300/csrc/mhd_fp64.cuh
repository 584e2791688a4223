// mhd_fp64.cuh -- the float64 forms of the ideal-MHD arithmetic (predictor,
// HLLD, conversions) of the FP64 path.
//
// What bounds it: the FP64 pipe.  GB300 issues 2 float64 operations per SM and
// cycle, 1/64 of its float32 rate, and not only additions and products run
// there but every comparison, minimum and conversion, and an IEEE division or
// square root is about ten of them.  Integer operations on the same bits are
// all but free beside it.  So these forms
//   - take reciprocals and reciprocal square roots from the hardware's float64
//     seeds and one cubic (Halley) step, 3 and 5 operations, and share them: a
//     reciprocal square root gives the root, the reciprocal root and the
//     reciprocal;
//   - decide signs, minima and limiters on the bit patterns;
//   - reconstruct from the differences of the characteristic variables (four
//     projections instead of five, and no subtractions per field), and add the
//     result to the cell's own state;
//   - form one side's fluxes in the Riemann solver, the side the contact
//     picks, instead of both.
// Measured (96^3 blast, PPM, FP64, ms per launch, IEEE forms and these):
// first-order stage (three launches) 3.33 and 1.69, sweep z 3.14 and 1.77, y
// 3.13 and 1.77, x 3.47 and 2.07, the pipe 81 to 86% busy; a Riemann problem
// takes about 265 of its slots, a traced cell 650.
//
// Accuracy, in units of 2^-53 relative, measured on the device: 1/x 1.00,
// 1/sqrt(x) 1.25, sqrt(x) 1.49.  Against long double on random states, mean
// relative error of the IEEE forms and of these (on the host, seeds 2^-23 and 2^-22
// off): predicted states 2.0e-16 and 0.45e-16 (MC), 2.1e-16 and 0.45e-16 (PPM), HLLD
// fluxes 1.5e-16 and 1.1e-16: states are formed as the cell's or the side's own
// plus a small increment, which loses less than recombining them whole.  (Against a
// float64 evaluation in the IEEE forms' order, whose roundings those share, one
// step reads 1.3e-16 and 1.4e-16 in 2-D, 1.5e-16 and 1.7e-16 at 96^3.)  Zeros and values below the normal range are roots
// of 0, as they are to the float32 path.
#pragma once

#include "mhd_device.cuh"

namespace ctu {

__device__ __forceinline__ long long d_bits(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ double d_from(long long b) { return __longlong_as_double(b); }
constexpr long long D_SIGN = (long long)0x8000000000000000ull, D_ONE_EXP = 1ll << 52, D_INF = 0x7FFll << 52;

// x > 0 (also +inf) and x >= 0, false for nans, whose sign bit says nothing
__device__ __forceinline__ bool d_pos(double x)
{
    return (unsigned long long)(d_bits(x) - 1) < 0x7FF0000000000000ull;
}
__device__ __forceinline__ bool d_nonneg(double x)
{
    return (unsigned long long)d_bits(x) <= (unsigned long long)D_INF || d_bits(x) == D_SIGN;
}
// |x| as an ordered integer, twice a magnitude, half of it
__device__ __forceinline__ long long d_mag(double x) { return d_bits(x) & ~D_SIGN; }
__device__ __forceinline__ long long d_twice(long long m) { return m >= D_ONE_EXP ? m + D_ONE_EXP : m << 1; }
__device__ __forceinline__ long long d_halve(long long m) { return m >= 2 * D_ONE_EXP ? m - D_ONE_EXP : m >> 1; }

#ifdef __CUDACC__  // the hardware's seeds (a host build brings its own)
__device__ __forceinline__ double d_rcp_seed(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    return r;
}
__device__ __forceinline__ double d_rsqrt_seed(double x)
{
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    return r;
}
#endif

// 1/x: seed r and residual e = 1 - x r, r (1 + e + e^2).
__device__ __forceinline__ double d_rcp64(double x)
{
    const double r = d_rcp_seed(x);
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}
// 1/sqrt(x) in y and sqrt(x) in s: seed y and residual e = 1 - x y^2,
// y (1 + e/2 + 3 e^2/8).  x below the normal range: y = 0, s = 0.
__device__ __forceinline__ void d_roots64(double x, double &y, double &s)
{
    const double y0 = d_rsqrt_seed(x);
    const double p = x * y0;
    const double e = fma(-p, y0, 1.0);
    const double t = fma(e, 0.375, 0.5) * e;
    const bool z = d_mag(x) < D_ONE_EXP;
    y = z ? 0.0 : fma(y0, t, y0);
    s = z ? 0.0 : fma(p, t, p);
}
__device__ __forceinline__ double d_sqrt64(double x)
{
    double y, s;
    d_roots64(x, y, s);
    return s;
}

// Monotonised-central slope of dm, dp (mc_slope) as a bit pattern: sign times
// min(|dm + dp|/2, 2|dm|, 2|dp|), 0 unless both have one sign and neither is a nan.
__device__ __forceinline__ double d_mc64(double dm, double dp)
{
    const long long am = d_mag(dm), ap = d_mag(dp);
    const long long a = am < ap ? am : ap, b = d_mag(dm + dp), t = d_twice(a), h = d_halve(b);
    const bool same = (d_bits(dm) ^ d_bits(dp)) >= 0 && a != 0 && b <= D_INF;
    return same ? d_from((h < t ? h : t) | (d_bits(dm) & D_SIGN)) : 0.0;
}

// Deviations (wp, wm) from the cell's value of the interface values of one
// field, from its four differences d[m] = w_(m+1) - w_m (reconstruct()):
// PPM, MC-linear, or MinMod where the hybrid integration asks for it.
template <int RK>
__device__ __forceinline__ void d_reconstruct64(const double (&d)[4], int lim, double &wp, double &wm)
{
    if (recon_hybrid(RK) && lim == 2) {
        const long long am = d_mag(d[1]), ap = d_mag(d[2]);
        const bool same = (d_bits(d[1]) ^ d_bits(d[2])) >= 0 && am != 0 && ap != 0 && am <= D_INF && ap <= D_INF;
        const double s = same ? d_from(d_halve(am < ap ? am : ap) | (d_bits(d[1]) & D_SIGN)) : 0.0;
        wp = s;
        wm = -s;
        return;
    }
    const double s0 = d_mc64(d[1], d[2]);
    if (recon_base(RK) == RECON_MC) {
        wp = 0.5 * s0;
        wm = -wp;
        return;
    }
    const double sm = d_mc64(d[0], d[1]), sp = d_mc64(d[2], d[3]);
    const double p = fma(0.5, d[2], (s0 - sp) * (1.0 / 6.0));
    const double m = fma(-0.5, d[1], (sm - s0) * (1.0 / 6.0));
    const long long ap = d_mag(p), am = d_mag(m);
    const bool num = ap < D_INF && am < D_INF;  // a nan or an infinity stays one
    const bool extremum = num && (d_bits(p) ^ d_bits(m)) >= 0 && ap != 0 && am != 0;
    const long long tp = d_twice(ap), tm = d_twice(am);
    const double np = num && ap >= tm ? d_from(tm | (~d_bits(m) & D_SIGN)) : p;
    const double nm = num && am >= tp ? d_from(tp | (~d_bits(p) & D_SIGN)) : m;
    wp = extremum ? 0.0 : np;
    wm = extremum ? 0.0 : nm;
}

// trace() on the deviations (tracing modes ALL and UPWIND).
__device__ __forceinline__ void d_trace64(double wp, double wm, double nu, int mode, double &tp, double &tm)
{
    const double dw = wp - wm, d2w = wp + wm, h = -0.5 * nu;
    const double up = fma(h, fma(d2w, fma(-2.0, nu, 3.0), dw), wp);
    const double um = fma(h, fma(-d2w, fma(2.0, nu, 3.0), dw), wm);
    tp = (mode == 0) | d_pos(nu) ? up : wp;
    tm = (mode == 0) | d_pos(-nu) ? um : wm;
}

// char_predict() for the kinds without reference states.
template <int PPM>
__device__ __forceinline__ void char_predict64(const double (&vs)[5][NV], double gam, double ch, double dtdx, int upwind,
                                               int lim, double (&Vp)[NV], double (&Vm)[NV])
{
    const double rho = vs[2][0], u = vs[2][1], v1c = vs[2][2], v2c = vs[2][3], pc = vs[2][4];
    const double Bn = vs[2][5], B1c = vs[2][6], B2c = vs[2][7];
    double isr, srho, ia, a, idisc, disc, icf, cf;
    d_roots64(rho, isr, srho);
    const double irho = d_rcp64(rho);
    const double a2 = gam * pc * irho;
    d_roots64(a2, ia, a);
    const double ia2 = ia * ia;
    const double ca = fabs(Bn) * isr;
    const double B2 = B1c * B1c + B2c * B2c;
    const double bn2 = Bn * Bn * irho, bt2 = B2 * irho, b2 = bn2 + bt2;
    const double ab = a2 - b2;
    d_roots64(fma(ab, ab, 4.0 * a2 * bt2), idisc, disc);
    const double cf2 = 0.5 * (a2 + b2 + disc);
    d_roots64(cf2, icf, cf);
    const double cs = a * ca * icf;
    // the fast and slow weights: the larger is (|a^2 - b^2| + disc)/2, the
    // product of the two a^2 bt^2, both over disc
    const double big = 0.5 * (fabs(ab) + disc);
    const double small = a2 * bt2 * d_rcp64(big);
    const bool hot = d_nonneg(ab);
    double af = 1.0, as = 0.0;
    if (d_pos(disc)) {
        const double rb = d_sqrt64(big * idisc), rs = d_sqrt64(small * idisc);
        af = hot ? rb : rs;
        as = hot ? rs : rb;
    }
    double be1 = 0.70710678118654752440, be2 = 0.70710678118654752440;
    if (d_mag(bt2) > d_mag(Tol<double>::bt() * a2)) {
        double ibt, bt;
        d_roots64(B2, ibt, bt);
        be1 = B1c * ibt;
        be2 = B2c * ibt;
    }
    const double S = copysign(1.0, Bn);
    const double ich = d_rcp64(ch);

    // differences of the characteristic variables across the stencil
    const double fcf = af * cf, scs = as * cs, fcfS = fcf * S, scsS = scs * S;
    const double fr = af * irho, sr = as * irho, sb = as * a * isr, fb = af * a * isr;
    const double q1 = S * be2 * isr, q2 = S * be1 * isr;
    double wf_p[4], wf_m[4], wa_p[4], wa_m[4], ws_p[4], ws_m[4], we[4], wg_m[4], wg_p[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const double du = vs[m + 1][1] - vs[m][1], d1 = vs[m + 1][2] - vs[m][2], d2 = vs[m + 1][3] - vs[m][3];
        const double dp = vs[m + 1][4] - vs[m][4], dn = vs[m + 1][5] - vs[m][5];
        const double b1 = vs[m + 1][6] - vs[m][6], b2m = vs[m + 1][7] - vs[m][7], ds = vs[m + 1][8] - vs[m][8];
        const double PV = be1 * d1 + be2 * d2;
        const double PB = be1 * b1 + be2 * b2m;
        const double P = be1 * d2 - be2 * d1;
        const double Q = q1 * b1 - q2 * b2m;
        const double Xf = fcf * du - scsS * PV, Yf = fr * dp + sb * PB;
        const double Xs = scs * du + fcfS * PV, Ys = sr * dp - fb * PB;
        wf_p[m] = Yf + Xf;
        wf_m[m] = Yf - Xf;
        ws_p[m] = Ys + Xs;
        ws_m[m] = Ys - Xs;
        wa_p[m] = P + Q;
        wa_m[m] = P - Q;
        we[m] = fma(-dp, ia2, vs[m + 1][0] - vs[m][0]);
        wg_p[m] = fma(ds, ich, dn);
        wg_m[m] = fma(-ds, ich, dn);
    }
    double rp, rm, tpf_p, tmf_p, tpf_m, tmf_m, tpa_p, tma_p, tpa_m, tma_m;
    double tps_p, tms_p, tps_m, tms_m, tpe, tme, tpg_p, tmg_p, tpg_m, tmg_m;
    d_reconstruct64<PPM>(wf_m, lim, rp, rm);
    d_trace64(rp, rm, (u - cf) * dtdx, upwind, tpf_m, tmf_m);
    d_reconstruct64<PPM>(wa_m, lim, rp, rm);
    d_trace64(rp, rm, (u - ca) * dtdx, upwind, tpa_m, tma_m);
    d_reconstruct64<PPM>(ws_m, lim, rp, rm);
    d_trace64(rp, rm, (u - cs) * dtdx, upwind, tps_m, tms_m);
    d_reconstruct64<PPM>(we, lim, rp, rm);
    d_trace64(rp, rm, u * dtdx, upwind, tpe, tme);
    d_reconstruct64<PPM>(ws_p, lim, rp, rm);
    d_trace64(rp, rm, (u + cs) * dtdx, upwind, tps_p, tms_p);
    d_reconstruct64<PPM>(wa_p, lim, rp, rm);
    d_trace64(rp, rm, (u + ca) * dtdx, upwind, tpa_p, tma_p);
    d_reconstruct64<PPM>(wf_p, lim, rp, rm);
    d_trace64(rp, rm, (u + cf) * dtdx, upwind, tpf_p, tmf_p);
    double gpr, gmr, gpl, gml;
    d_reconstruct64<PPM>(wg_m, lim, gpl, gml);
    d_trace64(gpl, gml, -ch * dtdx, upwind, tpg_m, tmg_m);
    d_reconstruct64<PPM>(wg_p, lim, gpr, gmr);
    d_trace64(gpr, gmr, ch * dtdx, upwind, tpg_p, tmg_p);

    // S_Bx dB_n/dx + S_psi dpsi/dx, common to both interfaces
    const double dgp = gpr - gmr, dgm = gpl - gml;
    const double h = 0.5 * dtdx;
    const double hB = 0.5 * h * (dgp + dgm);  // h dB_n
    const double hps = 0.5 * h * ch * (dgp - dgm);
    const double vB = u * Bn + v1c * B1c + v2c * B2c;
    const double hr = hB * irho;
    double s[NV] = {vs[2][0], fma(Bn, hr, u), fma(B1c, hr, v1c), fma(B2c, hr, v2c),
                    fma(gam - 1.0, Bn * hps - vB * hB, pc), Bn, fma(v1c, hB, B1c), fma(v2c, hB, B2c), vs[2][8]};
    // A nan or infinity in the cell itself makes both states nans whole, as it would
    // as a term of every characteristic variable: the limiters drop its differences.
    int top = 0;
#pragma unroll
    for (int q = 0; q < NV; ++q) top = max(top, __double2hiint(vs[2][q]) & 0x7FFFFFFF);
    const long long lost = top >= 0x7FF00000 ? 0x7FF8ll << 48 : 0ll;
#pragma unroll
    for (int q = 0; q < NV; ++q) s[q] = d_from(d_bits(s[q]) | lost);

    // recombination with the right eigenvectors, added to the cell's state
    const double i2a2 = 0.5 * ia2, hrho = 0.5 * rho;
    const double kf = fcf * i2a2, ks = scs * i2a2, kfS = fcfS * i2a2, ksS = scsS * i2a2;
    const double sq = 0.5 * srho * ia;  // sqrt(rho) a / (2 a^2)
    const double k1 = 0.5 * S * srho * be2, k2 = 0.5 * S * srho * be1, hb1 = 0.5 * be1, hb2 = 0.5 * be2, hch = 0.5 * ch;
    auto combine = [&](double fp, double fm, double ap, double am, double sp_, double sm_, double e, double gp, double gm,
                       double (&V)[NV]) {
        const double fs = fp + fm, fd = fp - fm, ss = sp_ + sm_, sd = sp_ - sm_;
        const double as_ = ap + am, ad = ap - am;
        const double P = hrho * (af * fs + as * ss);
        V[0] = s[0] + fma(P, ia2, e);
        V[1] = s[1] + (kf * fd + ks * sd);
        const double tv = kfS * sd - ksS * fd;
        V[2] = s[2] + (tv * be1 - hb2 * as_);
        V[3] = s[3] + (tv * be2 + hb1 * as_);
        V[4] = s[4] + P;
        V[5] = fma(0.5, gp + gm, s[5]);
        const double tb = (as * fs - af * ss) * sq;
        V[6] = s[6] + (tb * be1 + k1 * ad);
        V[7] = s[7] + (tb * be2 - k2 * ad);
        V[8] = fma(hch, gp - gm, s[8]);
    };
    combine(tpf_p, tpf_m, tpa_p, tpa_m, tps_p, tps_m, tpe, tpg_p, tpg_m, Vp);
    combine(tmf_p, tmf_m, tma_p, tma_m, tms_p, tms_m, tme, tmg_p, tmg_m, Vm);
}

// Square of the fast speed from 1/rho.
__device__ __forceinline__ double d_fast2(double irho, double p, double Bn2, double Bt2, double gam)
{
    const double a2 = gam * p * irho, bt2 = Bt2 * irho, b2 = fma(Bn2, irho, bt2);
    const double ab = a2 - b2;
    return 0.5 * (a2 + b2 + d_sqrt64(fma(ab, ab, 4.0 * a2 * bt2)));
}

// riemann_hlld() in float64: the same solver; fluxes, conserved states and the
// star energy of the side the contact picks only.
__device__ __forceinline__ bool riemann_hlld(const double (&L)[NV], const double (&Rt)[NV], double gam, double ch,
                                             double (&F)[NV])
{
    const bool bad = !(d_pos(L[0]) && d_pos(L[4]) && d_pos(Rt[0]) && d_pos(Rt[4]));
    const double ich = d_rcp64(ch), igm = d_rcp64(gam - 1.0);
    const double Bn = 0.5 * ((L[5] + Rt[5]) - (Rt[8] - L[8]) * ich);
    const double pm = 0.5 * ((L[8] + Rt[8]) - ch * (Rt[5] - L[5]));
    const double Bn2 = Bn * Bn;
    const double rL = L[0], uL = L[1], vL = L[2], wL = L[3], pL = L[4], yL = L[6], zL = L[7];
    const double rR = Rt[0], uR = Rt[1], vR = Rt[2], wR = Rt[3], pR = Rt[4], yR = Rt[6], zR = Rt[7];
    const double tL = yL * yL + zL * zL, tR = yR * yR + zR * zR;
    const double hL = 0.5 * (Bn2 + tL), hR = 0.5 * (Bn2 + tR);
    const double ptL = pL + hL, ptR = pR + hR;
    const double cL = d_fast2(d_rcp64(rL), pL, Bn2, tL, gam), cR = d_fast2(d_rcp64(rR), pR, Bn2, tR, gam);
    const double cmax = d_sqrt64(d_mag(cL) > d_mag(cR) ? cL : cR);
    const bool lt = uL < uR;
    const double SL = (lt ? uL : uR) - cmax, SR = (lt ? uR : uL) + cmax;
    const double sdL = SL - uL, sdR = SR - uR;
    const double mL = sdL * rL, mR = sdR * rR;
    const double iden = d_rcp64(mR - mL);
    const double SM = ((mR * uR - mL * uL) + (ptL - ptR)) * iden;
    const bool outL = d_nonneg(SL), outR = !outL && d_nonneg(-SR);
    const bool right = outR || (!outL && !d_nonneg(SM));

    // the picked side
    const double r = right ? rR : rL, u = right ? uR : uL, v = right ? vR : vL, w = right ? wR : wL;
    const double p = right ? pR : pL, y = right ? yR : yL, z = right ? zR : zL, pt = right ? ptR : ptL;
    const double E = fma(p, igm, fma(0.5 * r, u * u + v * v + w * w, right ? hR : hL));
    const double vB = u * Bn + v * y + w * z;
    const double m0 = r * u;
    double G0 = m0, G1 = fma(m0, u, pt) - Bn2, G2 = m0 * v - Bn * y, G3 = m0 * w - Bn * z;
    double G4 = (E + pt) * u - Bn * vB, G6 = u * y - Bn * v, G7 = u * z - Bn * w;
    if (!(outL || outR)) {
        // every star state as its difference from the side's state, all of
        // them multiples of S_M - u: rho* - rho = rho (S_M - u)/(S - S_M),
        // v* - v = -B_t B_n k, B_t* - B_t = B_t m k, with m = rho (S - u) and
        // k = (S_M - u)/(m (S - S_M) - B_n^2)
        const double pts = fma(mR * mL, uR - uL, mR * ptL - mL * ptR) * iden;
        const double qL = SL - SM, qR = SR - SM;
        const double iqL = d_rcp64(qL), iqR = d_rcp64(qR);
        const double nL = SM - uL, nR = SM - uR;
        const double dL = fma(mL, qL, -Bn2), dR = fma(mR, qR, -Bn2);
        double kL = 0.0, kR = 0.0;
        if (d_mag(dL) > d_mag(Tol<double>::hlld() * fma(mL, sdL, Bn2))) kL = nL * d_rcp64(dL);
        if (d_mag(dR) > d_mag(Tol<double>::hlld() * fma(mR, sdR, Bn2))) kR = nR * d_rcp64(dR);
        const double gL = -Bn * kL, gR = -Bn * kR, fL = mL * kL, fR = mR * kR;
        const double vsL = fma(yL, gL, vL), wsL = fma(zL, gL, wL), ysL = fma(yL, fL, yL), zsL = fma(zL, fL, zL);
        const double vsR = fma(yR, gR, vR), wsR = fma(zR, gR, wR), ysR = fma(yR, fR, yR), zsR = fma(zR, fR, zR);
        const double S = right ? SR : SL, iq = right ? iqR : iqL, n = right ? nR : nL;
        const double g = right ? gR : gL, f = right ? fR : fL;
        const double ys = right ? ysR : ysL, zs = right ? zsR : zsL;
        const double dv = y * g, dw = z * g, dy = y * f, dz = z * f;
        const double dr = r * n * iq, rs = r + dr;
        // v.B - v*.B*
        const double dvB = -(n * Bn + dv * ys + v * dy + dw * zs + w * dz);
        G0 = fma(S, dr, G0);
        G1 = fma(S, rs * n + dr * u, G1);
        G2 = fma(S, rs * dv + dr * v, G2);
        G3 = fma(S, rs * dw + dr * w, G3);
        G4 = fma(S * iq, (E + pts) * n + (pts - pt) * u + Bn * dvB, G4);
        G6 = fma(S, dy, G6);
        G7 = fma(S, dz, G7);
        double iL, sqL, iR, sqR;
        d_roots64(mL * iqL, iL, sqL);
        d_roots64(mR * iqR, iR, sqR);
        const double aB = fabs(Bn);
        const double SLs = fma(-aB, iL, SM), SRs = fma(aB, iR, SM);
        if (!d_nonneg(SLs) && !d_nonneg(-SRs)) {
            // the double star state, from the picked side's star state
            const double sB = copysign(1.0, Bn);
            const double isq = d_rcp64(sqL + sqR), sLR = sqL * sqR * sB;
            const double cv = (right ? -sqL : sqR) * isq, cy = (right ? -sqR : sqL) * isq, cs = sB * isq, cx = sLR * isq;
            const double Dv = vsR - vsL, Dw = wsR - wsL, Dy = ysR - ysL, Dz = zsR - zsL;
            const double ev = cv * Dv + cs * Dy, ew = cv * Dw + cs * Dz, ey = cy * Dy + cx * Dv, ez = cy * Dz + cx * Dw;
            const double vs = v + dv, ws = w + dw;
            // v**.B** - v*.B*
            const double evB = ev * (ys + ey) + vs * ey + ew * (zs + ez) + ws * ez;
            const double Ss = right ? SRs : SLs, sq = right ? -sqR * sB : sqL * sB;
            const double rSs = rs * Ss;
            G2 = fma(rSs, ev, G2);
            G3 = fma(rSs, ew, G3);
            G4 = fma(Ss * sq, evB, G4);
            G6 = fma(Ss, ey, G6);
            G7 = fma(Ss, ez, G7);
        }
    }
    F[0] = G0; F[1] = G1; F[2] = G2; F[3] = G3; F[4] = G4;
    F[5] = pm;
    F[6] = G6; F[7] = G7;
    F[8] = ch * ch * Bn;
    return bad;
}

} // namespace ctu
