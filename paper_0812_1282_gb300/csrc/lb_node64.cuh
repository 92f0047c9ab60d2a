// FP64 per-node arithmetic of the step (Steps 1-3 of Sec. V), written for
// this GPU's FP64 pipe, which bounds every FP64 step.
//
// The pipe takes one warp instruction per 64 cycles from a scheduler, and
// all four schedulers together one per 16 cycles when every operand of a
// DFMA is a register, but only one per 19 when the instruction is a DADD or
// DMUL or has a constant among its operands (measured on independent
// chains, 1 to 16 warps).  So what counts is the number of operations, and
// each is best a DFMA on registers:
//  - the constants, among them 1, -1 and -0, come from shared memory (Node64),
//    where the compiler cannot fold them: add(x, y) is x * 1 + y and
//    mul(x, y) is x * y + (-0), exactly the sum and the product (2048^2, MRT:
//    832 us a step; 907 with plain sums and products; all constants held in
//    registers for a whole tile, two CTAs per SM instead of three: 996);
//  - opposite directions share their even part (E) and differ in the sign of
//    the odd one, which MRT leaves at its equilibrium;
//  - the two reciprocals 1/rho and 1/tau come from one of rho tau;
//  - constant factors of the stencils (kappa, 1/12, 1/6) are folded into the
//    node constants, and the stencils into running row values (lb_step64.cuh).
// 115.6 operations a node (counted, MRT) where the plain form has 203.6.  All products
// and sums are explicit fused operations, so every kernel that calls these
// functions gets the same bits.
#pragma once

#include <cuda_runtime.h>

#include <cmath>

namespace lbfe {

// Constants of one domain, computed once on the host (DomDesc::c64) and read
// from shared memory.  s = sqrt(kappa).
struct Node64 {
    double one, mone, nzero;   // 1, -1, -0
    double two, four, m4, m20;
    double q25, c3, c9, c12, m24;  // 1/4, 1/3, 1/9, 1/12, -1/24
    double sig;                // s / 12: scale of the phi values the stencils read
    double qa, ma6, cl;        // a/4, -a/6, -(2/3) s
    double ga, mga, gl;        // Gamma a / 3, -Gamma a / 3, -(2/3) Gamma s
    double t0, t1;             // tau = t0 + t1 phi
    double kg, og;             // 1 - 1/tau_phi, 1/tau_phi
    double lut_lo, lut_step, lut_inv, lut_kmax;
};
constexpr int kNode64 = int(sizeof(Node64) / sizeof(double));
static_assert(kNode64 <= 32, "one warp copies the constants");

inline Node64 make_node64(double a, double kappa, double gamma, double omega_phi, double tau_c0,
                          double tau_c1, double lut_lo, double lut_step, double lut_inv,
                          double lut_kmax)
{
    const double s = std::sqrt(kappa);
    Node64 c;
    c.one = 1.0;
    c.mone = -1.0;
    c.nzero = -0.0;
    c.two = 2.0;
    c.four = 4.0;
    c.m4 = -4.0;
    c.m20 = -20.0;
    c.q25 = 0.25;
    c.c3 = 1.0 / 3.0;
    c.c9 = 1.0 / 9.0;
    c.c12 = 1.0 / 12.0;
    c.m24 = -1.0 / 24.0;
    c.sig = s / 12.0;
    c.qa = 0.25 * a;
    c.ma6 = -a / 6.0;
    c.cl = -2.0 * s / 3.0;
    c.ga = gamma * a / 3.0;
    c.mga = -c.ga;
    c.gl = -2.0 * gamma * s / 3.0;
    c.t0 = tau_c0;
    c.t1 = tau_c1;
    c.kg = 1.0 - omega_phi;
    c.og = omega_phi;
    c.lut_lo = lut_lo;
    c.lut_step = lut_step;
    c.lut_inv = lut_inv;
    c.lut_kmax = lut_kmax;
    return c;
}

// All threads of a CTA (or the given range) copy the constants.
__device__ __forceinline__ void load_node64(Node64& dst, const double* src, int tid)
{
    if (tid < kNode64) reinterpret_cast<double*>(&dst)[tid] = src[tid];
}

// x + y, x - y, x y and x y + z as one DFMA each (C: a Node64)
#define LB64_ADD(x, y) __fma_rn((x), C.one, (y))
#define LB64_SUB(x, y) __fma_rn((y), C.mone, (x))
#define LB64_MUL(x, y) __fma_rn((x), (y), C.nzero)

// 1 / x: the hardware's seed (about 20 bits) and one third-order Newton-
// Raphson step, r (1 + e + e^2) with e = 1 - x r (relative error e^3,
// below the rounding of the last operation).
__device__ __forceinline__ double rcp64(const Node64& C, double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = __fma_rn(-x, r, C.one);
    return __fma_rn(r, __fma_rn(e, e, e), r);
}

// What m of a wall ghost row (lb_step64.cuh) is less than the m of the row it
// mirrors: phi is wet_k h less, 4 + 1 + 1 times, on the scaled phi.
__device__ __forceinline__ double ghost_shift64(double sig, int wet_k, double h)
{
    return __dmul_rn(6.0 * wet_k * h, sig);
}

// phi = sum of the nine pulled g, of which a node's collision wants g_0 and the
// sum of the others apart (collide_g64).
struct Phi64 {
    double g0, tail;
};
__device__ __forceinline__ double phi64(const Node64& C, const double (&g)[9], Phi64& s)
{
    s.g0 = g[0];
    s.tail = LB64_ADD(LB64_ADD(LB64_ADD(g[1], g[2]), LB64_ADD(g[3], g[4])),
                      LB64_ADD(LB64_ADD(g[5], g[6]), LB64_ADD(g[7], g[8])));
    return LB64_ADD(s.g0, s.tail);
}
__device__ __forceinline__ double phi64(const Node64& C, const double (&g)[9])
{
    Phi64 s;
    return phi64(C, g, s);
}

// Step 1 (Eq. moments) at one node: from its pulled f (deviation form) the sums
// s of opposite directions, rho - 1 and rho u; then, with phi, u and w = 1/tau.
struct Moments64 {
    double s1, s3, s5, s7, drho, jx, jy, w, ux, uy;
};
__device__ __forceinline__ void sums64(const Node64& C, const double (&f)[9], Moments64& m)
{
    m.s1 = LB64_ADD(f[1], f[2]);
    m.s3 = LB64_ADD(f[3], f[4]);
    m.s5 = LB64_ADD(f[5], f[6]);
    m.s7 = LB64_ADD(f[7], f[8]);
    const double d1 = LB64_SUB(f[1], f[2]), d3 = LB64_SUB(f[3], f[4]);
    const double d5 = LB64_SUB(f[5], f[6]), d7 = LB64_SUB(f[7], f[8]);
    m.drho = LB64_ADD(LB64_ADD(LB64_ADD(m.s1, m.s3), LB64_ADD(m.s5, m.s7)), f[0]);
    m.jx = LB64_ADD(d1, LB64_SUB(d5, d7));
    m.jy = LB64_ADD(d3, LB64_ADD(d5, d7));
}
// 1/rho and w from one reciprocal of rho tau.  Step 2 (s2) takes u_eq = 0, and
// with it 1/rho = 0.
__device__ __forceinline__ void velocity64(const Node64& C, double phi, bool s2, Moments64& m)
{
    // Eq. (tau), or the nearest tabulated one (lookup table of Sec. V)
    double tau = __fma_rn(C.t1, phi, C.t0);
    if (C.lut_kmax > 0.0) {
        const double k = fmin(fmax(rint((tau - C.lut_lo) * C.lut_inv), 0.0), C.lut_kmax);
        tau = __fma_rn(k, C.lut_step, C.lut_lo);
    }
    // 1/rho = tau / (rho tau), w = 1/tau = rho / (rho tau)
    const double r = rcp64(C, __fma_rn(tau, m.drho, tau));
    m.w = __fma_rn(m.drho, r, r);
    const double irho = s2 ? 0.0 : LB64_MUL(tau, r);
    m.ux = LB64_MUL(m.jx, irho);
    m.uy = LB64_MUL(m.jy, irho);
}

// The new f of a node: phi and its scaled derivatives X = s d_x phi, Y = s d_y
// phi, L = (s / 2) nabla^2 phi.  On Step-2 nodes the odd coefficients alpha
// (axis) and beta (diagonal) are those of the momentum rows' reading (MRT
// keeps j: 1/6; relaxing or BGK: 0).
template <bool MRT>
__device__ __forceinline__ void collide_f64(const Node64& C, const double (&f)[9],
                                            const Moments64& m, double phi, double phi2, double X,
                                            double Y, double L, bool s2, bool relax_j,
                                            double (&fo)[9])
{
    const double alpha = s2 ? (MRT && !relax_j ? 1.0 / 6.0 : 0.0) : C.c3;
    const double beta = s2 ? (MRT && !relax_j ? 1.0 / 6.0 : 0.0) : C.c12;
    const double jx = m.jx, jy = m.jy, w = m.w;
    // A9: a ninth of 3 [p0 - kappa phi lap] - rho (Eq. p0 less the rest pressure)
    const double A9 =
        __fma_rn(phi, __fma_rn(phi, __fma_rn(C.qa, phi2, C.ma6), LB64_MUL(C.cl, L)),
                 LB64_MUL(C.c9, m.drho));
    // rho u_a u_b and kappa d_a phi d_b phi: traces, and the two stress
    // moments of f^eq (rows 7, 8 of Eq. Matrix)
    const double rxx = LB64_MUL(jx, m.ux), R = __fma_rn(jy, m.uy, rxx);
    const double kxx = LB64_MUL(X, X), K = __fma_rn(Y, Y, kxx);
    const double S = LB64_ADD(R, K);
    const double m7e = __fma_rn(C.two, LB64_ADD(rxx, kxx), -S);
    const double m8e = __fma_rn(X, Y, LB64_MUL(jx, m.uy));
    // even parts of the axis and the diagonal directions (Appendix A)
    const double Pe = __fma_rn(C.c12, S, A9);
    const double Qe = __fma_rn(C.q25, A9, __fma_rn(C.c12, R, LB64_MUL(C.m24, K)));
    const double jp = LB64_ADD(jx, jy), jm = LB64_SUB(jy, jx);
    if (MRT) {
        // Step 3: the stress moments relax at w, the others are at equilibrium
        const double m7 = LB64_SUB(m.s1, m.s3), m8 = LB64_SUB(m.s5, m.s7);
        const double n7 = __fma_rn(w, LB64_SUB(m7e, m7), m7);
        const double n8 = __fma_rn(w, LB64_SUB(m8e, m8), m8);
        const double Ex = __fma_rn(C.q25, n7, Pe), Ey = __fma_rn(-C.q25, n7, Pe);
        const double Ed = __fma_rn(C.q25, n8, Qe), Ea = __fma_rn(-C.q25, n8, Qe);
        fo[1] = __fma_rn(alpha, jx, Ex);
        fo[2] = __fma_rn(-alpha, jx, Ex);
        fo[3] = __fma_rn(alpha, jy, Ey);
        fo[4] = __fma_rn(-alpha, jy, Ey);
        fo[5] = __fma_rn(beta, jp, Ed);
        fo[6] = __fma_rn(-beta, jp, Ed);
        fo[7] = __fma_rn(beta, jm, Ea);
        fo[8] = __fma_rn(-beta, jm, Ea);
        fo[0] = __fma_rn(C.m4, LB64_ADD(Pe, Qe), m.drho);
    } else {
        // f' = (1 - w) f + w f^eq
        const double k = LB64_SUB(C.one, w), aw = LB64_MUL(alpha, w), bw = LB64_MUL(beta, w);
        const double wx = LB64_MUL(w, __fma_rn(C.q25, m7e, Pe));
        const double wy = LB64_MUL(w, __fma_rn(-C.q25, m7e, Pe));
        const double wd = LB64_MUL(w, __fma_rn(C.q25, m8e, Qe));
        const double wa = LB64_MUL(w, __fma_rn(-C.q25, m8e, Qe));
        fo[1] = __fma_rn(k, f[1], __fma_rn(aw, jx, wx));
        fo[2] = __fma_rn(k, f[2], __fma_rn(-aw, jx, wx));
        fo[3] = __fma_rn(k, f[3], __fma_rn(aw, jy, wy));
        fo[4] = __fma_rn(k, f[4], __fma_rn(-aw, jy, wy));
        fo[5] = __fma_rn(k, f[5], __fma_rn(bw, jp, wd));
        fo[6] = __fma_rn(k, f[6], __fma_rn(-bw, jp, wd));
        fo[7] = __fma_rn(k, f[7], __fma_rn(bw, jm, wa));
        fo[8] = __fma_rn(k, f[8], __fma_rn(-bw, jm, wa));
        const double f0e = __fma_rn(C.m4, LB64_ADD(Pe, Qe), m.drho);
        fo[0] = __fma_rn(w, LB64_SUB(f0e, f[0]), f[0]);
    }
}

// The new g of a node.  g9 gives the pulled g, read only for tau_phi != 1.  g_0,
// which carries phi, advances by the difference of the others' sums before and
// after, so that a step rounds it once.  Phi less the others' new sum is an operation
// fewer (2048^2 829 and 834 us a step, 401 x 77 channel 8.8 and 9.0), but has the
// roundings of phi's own sum: the error of phi after 200 steps, against extended
// precision, 5.1e-16 rms and 2.4e-16 so.
template <class G9>
__device__ __forceinline__ void collide_g64(const Node64& C, const Moments64& m, double phi,
                                            double phi2, const Phi64& s, double L, G9 g9,
                                            double (&go)[9])
{
    // g^eq (Appendix A): a third of Gamma mu, then the velocity terms
    const double G3 = __fma_rn(phi, __fma_rn(C.ga, phi2, C.mga), LB64_MUL(C.gl, L));
    const double pux = LB64_MUL(phi, m.ux), puy = LB64_MUL(phi, m.uy);
    const double pxx = LB64_MUL(pux, m.ux), puu = __fma_rn(puy, m.uy, pxx);
    const double pd = __fma_rn(C.two, pxx, -puu), pxy = LB64_MUL(pux, m.uy);
    const double b = LB64_MUL(C.c12, puu);
    const double H = LB64_ADD(G3, b), D = __fma_rn(C.q25, G3, b);
    const double Gx = __fma_rn(C.q25, pd, H), Gy = __fma_rn(-C.q25, pd, H);
    const double Gd = __fma_rn(C.q25, pxy, D), Ga = __fma_rn(-C.q25, pxy, D);
    const double pp = LB64_ADD(pux, puy), pm = LB64_SUB(puy, pux);
    go[1] = __fma_rn(C.c3, pux, Gx);
    go[2] = __fma_rn(-C.c3, pux, Gx);
    go[3] = __fma_rn(C.c3, puy, Gy);
    go[4] = __fma_rn(-C.c3, puy, Gy);
    go[5] = __fma_rn(C.c12, pp, Gd);
    go[6] = __fma_rn(-C.c12, pp, Gd);
    go[7] = __fma_rn(C.c12, pm, Ga);
    go[8] = __fma_rn(-C.c12, pm, Ga);
    const double d = __fma_rn(C.m4, LB64_ADD(H, D), s.tail);
    go[0] = __fma_rn(C.og, d, s.g0);
    if (C.kg != 0.0) {
        // Eq. (gevo) with tau_phi != 1 (tau_phi = 1, Sec. III.B, leaves g' = g^eq)
        double g[9];
        g9(g);
#pragma unroll
        for (int i = 1; i < 9; ++i) go[i] = __fma_rn(C.kg, g[i] - go[i], go[i]);
    }
}

// One node: both.
template <bool MRT, class G9>
__device__ __forceinline__ void collide64(const Node64& C, const double (&f)[9], double phi,
                                          const Phi64& s, double X, double Y, double L, bool s2,
                                          bool relax_j, G9 g9, double (&fo)[9], double (&go)[9])
{
    Moments64 m;
    sums64(C, f, m);
    velocity64(C, phi, s2, m);
    const double phi2 = LB64_MUL(phi, phi);
    collide_f64<MRT>(C, f, m, phi, phi2, X, Y, L, s2, relax_j, fo);
    collide_g64(C, m, phi, phi2, s, L, g9, go);
}

}  // namespace lbfe
