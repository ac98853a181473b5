// The pair terms of the FP64 path (particles fixed in pseudo-time).
//
// Its kernels are bound by the FP64 pipe (1.25 TFLOP/s measured, 1/62 of FP32),
// so what counts is the number of FP64 instructions per pair, an addition as much
// as an fma. Constants common to every pair are factored out of the sums: with
// dW/dr = (sigma / h) w(q), g = w r_ij / r and F = w r / (r^2 + eta h^2),
//   dp/dtau = sigma/h (c_div sum V_ij . g + c_edac sum p_ij F)
//   F_i     = sigma/h (-c_p sum (p_i + p_j) g + c_visc sum F V_ij)
// which takes 4 d + 3 instructions a pair (11 in 2D, 15 in 3D; with the constants
// inside the sums 18 and 23), every one of them on a difference or sum formed
// first as before. The geometry takes comparisons of high words instead of FP64
// comparisons, and a reciprocal square root and a division without the steps for special
// operands: with CUDA's, whose branches for those keep the pairs of a particle from
// overlapping, two steps of 200 x 200 moving particles with one launch an iteration take
// 7.4 ms instead of 4.9, of 30^3 without the cache 30.9 instead of 26.8.
#pragma once

#include "geometry.cuh"

namespace dtsph {

// 1/sqrt(x) for a normal positive x. The hardware's approximation y (PTX
// rsqrt.approx.ftz.f64: from the upper word of x, its lower word zero) takes one step of
// third order (Householder 1970; the binomial series of (1 - e)^(-1/2), e = 1 - x y^2): y
// (1 + e/2 + 3 e^2/8), truncated at 5/16 e^3. y has 21 bits, so y^2 is exact (x y would
// lose as much as the step's last bit). With e < 2^-18 the result is within (1 + 2^-2.6)
// 2^-53 of the value; CUDA's rsqrt is within 2^-52 (the tests bound the error and e).
__device__ __forceinline__ double rsqrt_step(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = __fma_rn(-x, __dmul_rn(y, y), 1.0);
    return __fma_rn(__dmul_rn(y, e), __fma_rn(0.375, e, 0.5), y);
}

// a / b where b and the quotient lie well inside the normal range. The hardware's
// approximation of 1/b (PTX rcp.approx.ftz.f64: from the upper word of b, its lower word
// zero) takes one third-order step of the geometric series, y (1 + e + e^2) with e = 1 -
// b y, truncated at e^3 < 2^-57; then Markstein's final step (IBM J. Res. Dev. 34, 1990):
// the residual a - b q of q = a y is exact, and q + y (a - b q) rounds the quotient but for
// about one operand pair in 2^50: the bits of the IEEE division (the tests compare them).
__device__ __forceinline__ double quotient(double a, double b)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
    const double e = __fma_rn(-b, y, 1.0);
    y = __fma_rn(y, __fma_rn(e, e, e), y);
    const double q = __dmul_rn(a, y);
    return __fma_rn(__fma_rn(-b, q, a), y, q);
}

// r_ij of a listed neighbour with the minimum image, and |r_ij|^2: sep64's
// operations, the image chosen by comparing high words (a listed pair lies within
// the list cutoff of one image, far from half a box length).
template <int D>
__device__ __forceinline__ double listed_sep64(const Geom &G, const double *xi, const double *__restrict__ x, int n,
                                               int j, double *d)
{
#pragma unroll
    for (int a = 0; a < D; ++a) {
        double v = __dsub_rn(xi[a], x[(size_t)a * n + j]);
        if (G.periodic[a] && (__double2hiint(v) & 0x7fffffff) > __double2hiint(G.halfL[a]))
            v = __double2hiint(v) < 0 ? __dadd_rn(v, G.L[a]) : __dsub_rn(v, G.L[a]);
        d[a] = v;
    }
    double r2 = __dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1]));
    if (D == 3) r2 = __dadd_rn(r2, __dmul_rn(d[2], d[2]));
    return r2;
}

// g and F of a pair, zeros from q = 3 on and at r = 0.
template <int D>
__device__ __forceinline__ void grad64(const Phys &P, const double *d, double r2, double *g, double &F)
{
#pragma unroll
    for (int a = 0; a < D; ++a) g[a] = 0.0;
    F = 0.0;
    if (__double2hiint(r2) < 0x00100000) return;        // r = 0 (or r^2 subnormal)
    const double rinv = rsqrt_step(r2);
    const double r = __dmul_rn(r2, rinv);
    const double q = __dmul_rn(r, P.inv_h);
    const int qh = __double2hiint(q);                   // 1, 2 and 3 have zero low words
    if (qh >= 0x40080000) return;
    const double a = __dsub_rn(3.0, q), a2 = __dmul_rn(a, a);
    double w = __dmul_rn(__dmul_rn(-5.0, a2), a2);
    if (qh < 0x40000000) {
        const double b = __dsub_rn(2.0, q), b2 = __dmul_rn(b, b);
        w = __fma_rn(__dmul_rn(30.0, b2), b2, w);
    }
    if (qh < 0x3ff00000) {
        const double c = __dsub_rn(1.0, q), c2 = __dmul_rn(c, c);
        w = __fma_rn(__dmul_rn(-75.0, c2), c2, w);
    }
    const double wr = __dmul_rn(w, rinv);
#pragma unroll
    for (int e = 0; e < D; ++e) g[e] = __dmul_rn(wr, d[e]);
    F = quotient(__dmul_rn(w, r), __dadd_rn(r2, P.eta_h2));
}

template <int D>
struct Sums64 {
    double vg, pF, pg[D], Fv[D];    // sum V_ij . g, p_ij F, (p_i + p_j) g, F V_ij
    __device__ __forceinline__ Sums64() : vg(0.0), pF(0.0)
    {
#pragma unroll
        for (int a = 0; a < D; ++a) pg[a] = Fv[a] = 0.0;
    }
};

// One pair's contribution; vv: the neighbour's velocity in the viscous terms, vd
// in the divergence term (WALLS; vv otherwise).
template <int D, bool WALLS>
__device__ __forceinline__ void pair64_accumulate(const PairConst<double> &k, const double *g, double F,
                                                  const double *vi, double pi, const double *vd, const double *vv,
                                                  double pj, Sums64<D> &A)
{
    double dv[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        dv[a] = __dsub_rn(vi[a], vv[a]);
        A.vg = __fma_rn(WALLS ? __dsub_rn(vi[a], vd[a]) : dv[a], g[a], A.vg);
        A.Fv[a] = __fma_rn(F, dv[a], A.Fv[a]);
    }
    A.pF = __fma_rn(__dsub_rn(pi, pj), F, A.pF);
    double pp = __dadd_rn(pi, pj);
    // the terms that most runs do without (artificial viscosity, the steady-mode
    // convection) sit behind one uniform test; they join sum (p_i + p_j) g in
    // units of c_p
    if (k.rare) {
        if (k.use_av) {
            // v_ij . r_ij < 0  <=>  v_ij . g > 0 (w < 0)
            double vvg = 0.0, g2 = 0.0;
#pragma unroll
            for (int a = 0; a < D; ++a) {
                vvg = __fma_rn(dv[a], g[a], vvg);
                g2 = __fma_rn(g[a], g[a], g2);
            }
            if (vvg > 0.0 && g2 > 0.0)
                pp = __dsub_rn(pp, __dmul_rn(k.c_av_m / k.c_p, __dmul_rn(vvg, F)) / g2);    // -m Pi_ij
        }
        if (k.steady) {
            // convection of Eq. (mom-steady): -(V_i + V_j) m/rho0 (V_i . g)
            double vg = 0.0;
#pragma unroll
            for (int a = 0; a < D; ++a) vg = __fma_rn(vi[a], g[a], vg);
            vg = __dmul_rn(k.vol / k.c_p, vg);
#pragma unroll
            for (int a = 0; a < D; ++a) A.pg[a] = __fma_rn(__dadd_rn(vi[a], vd[a]), vg, A.pg[a]);
        }
    }
#pragma unroll
    for (int a = 0; a < D; ++a) A.pg[a] = __fma_rn(pp, g[a], A.pg[a]);
}

// The rates with their factors (own lane's part), then summed over the L lanes.
template <int D, int L>
__device__ __forceinline__ void rates64(const Phys &P, const PairConst<double> &k, const Sums64<D> &A, double &ap,
                                        double *F)
{
    ap = __dmul_rn(k.c_div, A.vg);
    if (k.edac) ap = __fma_rn(k.c_edac, A.pF, ap);
    ap = __dmul_rn(ap, P.sig_h);
#pragma unroll
    for (int a = 0; a < D; ++a) F[a] = __dmul_rn(P.sig_h, __fma_rn(k.c_visc, A.Fv[a], -__dmul_rn(k.c_p, A.pg[a])));
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) {
        ap = __dadd_rn(ap, __shfl_xor_sync(0xffffffffu, ap, o));
#pragma unroll
        for (int a = 0; a < D; ++a) F[a] = __dadd_rn(F[a], __shfl_xor_sync(0xffffffffu, F[a], o));
    }
}

}  // namespace dtsph
