// The FP32 per-node arithmetic of lb_node.cuh on two nodes at once, with
// the packed FP32 add, multiply and fused multiply-add of sm_100 and later
// (one instruction for both lanes, half the issue slots of the scalar
// form).  Each lane evaluates the same
// formulas as the scalar path for its own node (Appendix A equilibria,
// Eq. best stencils, Eq. chempot, Eq. tau, Steps 1-3 of Sec. V), with the
// same unbiased divisions by small constants; products that feed a sum are
// fused explicitly, so a lane can differ from the scalar path by rounding.
// The functions are templates on the number of lanes: V = f2, or f1 for the
// step of small lattices (lb_small.cuh), one node per thread.  A lane gets
// the same bits in both.
#pragma once

#include <cuda_runtime.h>

#include "lb_node.cuh"

namespace lbfe {

// Two FP32 lanes.
struct f2 {
    float2 v;
    __device__ __forceinline__ f2() {}
    __device__ __forceinline__ f2(float2 a) : v(a) {}
    __device__ __forceinline__ f2(float a, float b) : v(make_float2(a, b)) {}
    __device__ __forceinline__ explicit f2(float a) : v(make_float2(a, a)) {}
    __device__ __forceinline__ float lane(int l) const { return l ? v.y : v.x; }
};
__device__ __forceinline__ f2 operator+(f2 a, f2 b) { return f2(__fadd2_rn(a.v, b.v)); }
// a - b, one rounding (the product with -1 is exact)
__device__ __forceinline__ f2 operator-(f2 a, f2 b)
{
    return f2(__ffma2_rn(b.v, make_float2(-1.f, -1.f), a.v));
}
__device__ __forceinline__ f2 operator*(f2 a, f2 b) { return f2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ f2 operator*(float k, f2 b)
{
    return f2(__fmul2_rn(make_float2(k, k), b.v));
}
// a * b + c, one rounding
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return f2(__ffma2_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ f2 fma2(float k, f2 b, f2 c)
{
    return f2(__ffma2_rn(make_float2(k, k), b.v, c.v));
}

// One FP32 lane, with the operations of f2.
struct f1 {
    float v;
    __device__ __forceinline__ f1() {}
    __device__ __forceinline__ explicit f1(float a) : v(a) {}
    __device__ __forceinline__ float lane(int) const { return v; }
};
__device__ __forceinline__ f1 operator+(f1 a, f1 b) { return f1(__fadd_rn(a.v, b.v)); }
__device__ __forceinline__ f1 operator-(f1 a, f1 b) { return f1(__fsub_rn(a.v, b.v)); }
__device__ __forceinline__ f1 operator*(f1 a, f1 b) { return f1(__fmul_rn(a.v, b.v)); }
__device__ __forceinline__ f1 operator*(float k, f1 b) { return f1(__fmul_rn(k, b.v)); }
__device__ __forceinline__ f1 fma2(f1 a, f1 b, f1 c) { return f1(__fmaf_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ f1 fma2(float k, f1 b, f1 c) { return f1(__fmaf_rn(k, b.v, c.v)); }

// The node parameters P of the functions below are a NodeParams<float> or a
// volatile one (in shared memory, read at each use).

// x / K, unbiased (the residual step of div_const<K, float>)
template <int K, class V>
__device__ __forceinline__ V div_const2(V x)
{
    constexpr float r = 1.0f / float(K);
    const V q = r * x;
    return fma2(r, fma2(-float(K), q, x), q);
}

// correctly rounded reciprocal, lane by lane (no packed form)
__device__ __forceinline__ f2 rcp2(f2 x) { return f2(__frcp_rn(x.v.x), __frcp_rn(x.v.y)); }
__device__ __forceinline__ f1 rcp2(f1 x) { return f1(__frcp_rn(x.v)); }

// G0<float>::value / advance lane by lane (integer words)
__device__ __forceinline__ f2 g0_value2(f2 w)
{
    return 0x1p-29f *
           f2(__int2float_rn(__float_as_int(w.v.x)), __int2float_rn(__float_as_int(w.v.y)));
}
__device__ __forceinline__ f2 g0_advance2(f2 w, f2 d)
{
    const f2 s = 0x1p29f * d;
    return f2(__int_as_float(__float_as_int(w.v.x) + __float2int_rn(s.v.x)),
              __int_as_float(__float_as_int(w.v.y) + __float2int_rn(s.v.y)));
}

__device__ __forceinline__ f1 g0_value2(f1 w)
{
    return 0x1p-29f * f1(__int2float_rn(__float_as_int(w.v)));
}
__device__ __forceinline__ f1 g0_advance2(f1 w, f1 d)
{
    return f1(__int_as_float(__float_as_int(w.v) + __float2int_rn((0x1p29f * d).v)));
}

// the nearest tabulated viscosity of one lane (lookup table of Sec. V)
template <class PP>
__device__ __forceinline__ float lut_tau(PP& P, float tau)
{
    const float k = fminf(fmaxf(rintf((tau - P.lut_lo) * P.lut_inv), 0.f), P.lut_kmax);
    return P.lut_lo + k * P.lut_step;
}
template <class PP>
__device__ __forceinline__ f2 lut_tau2(PP& P, f2 tau)
{
    return f2(lut_tau(P, tau.v.x), lut_tau(P, tau.v.y));
}
template <class PP>
__device__ __forceinline__ f1 lut_tau2(PP& P, f1 tau)
{
    return f1(lut_tau(P, tau.v));
}

// Eq. (best) on absolute values, differences to the centre first (exact for
// nearby values, as in stencils<float>)
template <class V>
__device__ __forceinline__ void stencils2(V c, V e, V w, V n, V s, V ne, V nw, V se, V sw, V& dx,
                                          V& dy, V& lap)
{
    const V de = e - c, dw = w - c, dn = n - c, ds = s - c;
    const V dne = ne - c, dnw = nw - c, dse = se - c, dsw = sw - c;
    dx = div_const2<12>(fma2(4.f, de - dw, dne - dnw) + (dse - dsw));
    dy = div_const2<12>(fma2(4.f, dn - ds, dne - dse) + (dnw - dsw));
    lap = div_const2<6>(fma2(4.f, (de + dw) + (dn + ds), (dne + dnw) + (dse + dsw)));
}

// Appendix A equilibria for i = 1..8 in deviation form (f_equilibria)
template <class PP, class V>
__device__ __forceinline__ void f_equilibria2(PP& P, V drho, V phi, V jxe,
                                              V jye, V uxe, V uye, V dx, V dy, V lap,
                                              V (&fe)[9], V& m7eq, V& m8eq)
{
    const V phi2 = phi * phi;
    // 3 [p0 - kappa phi lap] - rho
    const V A3 = fma2(-3.f * P.kappa, phi * lap,
                       fma2(P.a * phi2, fma2(2.25f, phi2, V(-1.5f)), drho));
    const V rxx = jxe * uxe, ryy = jye * uye, rxy = jxe * uye;
    const V ruu = rxx + ryy;
    const V kdx = P.kappa * dx, kdy = P.kappa * dy;
    const V kxx = kdx * dx, kyy = kdy * dy, kxy = kdx * dy;
    const V ksum = kxx + kyy;
    m7eq = (rxx - ryy) + (kxx - kyy);
    m8eq = rxy + kxy;
    const V A4 = 4.f * A3, r6 = -6.f * ruu;
    const V Bx = A4 + fma2(18.f, rxx, r6) + fma2(12.f, kxx, -6.f * kyy);
    const V By = A4 + fma2(18.f, ryy, r6) + fma2(12.f, kyy, -6.f * kxx);
    const V Bb = fma2(-1.5f, ksum, fma2(3.f, ruu, A3));
    const V x9 = 9.f * (rxy + kxy);
    const V Bd = Bb + x9, Ba = Bb - x9;
    const V jp = jxe + jye, jm = jye - jxe;
    fe[1] = div_const2<36>(fma2(12.f, jxe, Bx));
    fe[2] = div_const2<36>(fma2(-12.f, jxe, Bx));
    fe[3] = div_const2<36>(fma2(12.f, jye, By));
    fe[4] = div_const2<36>(fma2(-12.f, jye, By));
    fe[5] = div_const2<36>(fma2(3.f, jp, Bd));
    fe[6] = div_const2<36>(fma2(-3.f, jp, Bd));
    fe[7] = div_const2<36>(fma2(3.f, jm, Ba));
    fe[8] = div_const2<36>(fma2(-3.f, jm, Ba));
}

// Gamma mu, Eq. (chempot)
template <class PP, class V>
__device__ __forceinline__ V gamma_mu2(PP& P, V phi, V lap)
{
    const V mu = fma2(-P.kappa, lap, P.a * fma2(phi * phi, phi, V(0.f) - phi));
    return P.gamma * mu;
}

// g equilibria for i = 1..8 (g_equilibria)
template <class V>
__device__ __forceinline__ void g_equilibria2(V phi, V G, V uxe, V uye, V (&ge)[9])
{
    const V pux = phi * uxe, puy = phi * uye;
    const V pxx = pux * uxe, pyy = puy * uye, pxy = pux * uye;
    const V puu = pxx + pyy;
    const V G4 = 4.f * G, p2 = -2.f * puu;
    const V Cx = G4 + fma2(6.f, pxx, p2);
    const V Cy = G4 + fma2(6.f, pyy, p2);
    const V Gp = G + puu, x3 = 3.f * pxy;
    const V Cd = Gp + x3, Ca = Gp - x3;
    const V sp = pux + puy, sm = puy - pux;
    ge[1] = div_const2<12>(fma2(4.f, pux, Cx));
    ge[2] = div_const2<12>(fma2(-4.f, pux, Cx));
    ge[3] = div_const2<12>(fma2(4.f, puy, Cy));
    ge[4] = div_const2<12>(fma2(-4.f, puy, Cy));
    ge[5] = div_const2<12>(Cd + sp);
    ge[6] = div_const2<12>(Cd - sp);
    ge[7] = div_const2<12>(Ca + sm);
    ge[8] = div_const2<12>(Ca - sm);
}

template <class V>
__device__ __forceinline__ V g_tail_sum2(const V (&g)[9])
{
    return (((g[1] + g[2]) + (g[3] + g[4])) + ((g[5] + g[6]) + (g[7] + g[8])));
}

// The f part of Steps 1-3 (collide_f) for two nodes of one row.  step2 and
// step2_relax_j are those of the row.
template <bool MRT, class PP, class V>
__device__ __forceinline__ void collide_f2(PP& P, const V (&f)[9], V phi,
                                           V dx, V dy, V lap, bool step2, bool step2_relax_j,
                                           V (&fo)[9], V& uxe_out, V& uye_out)
{
    const V drho = (((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7]))) + f[8];
    const V jx = (f[1] - f[2]) + (f[5] - f[6]) + (f[8] - f[7]);
    const V jy = (f[3] - f[4]) + (f[5] - f[6]) + (f[7] - f[8]);
    const V irho = rcp2(V(1.f) + drho);
    // Eq. (tau), with the lookup table of Sec. V lane by lane
    V tau = P.tau_c1 == 0.f ? V(P.tau_c0) : fma2(P.tau_c1, phi, V(P.tau_c0));
    if (P.lut_kmax > 0.f) tau = lut_tau2(P, tau);
    const V omega = rcp2(tau);
    // Step 2
    const V zero(0.f);
    const V jxe = step2 ? zero : jx, jye = step2 ? zero : jy;
    const V uxe = step2 ? zero : jx * irho, uye = step2 ? zero : jy * irho;
    V fe[9], m7eq, m8eq;
    f_equilibria2(P, drho, phi, jxe, jye, uxe, uye, dx, dy, lap, fe, m7eq, m8eq);
    // Step 3
    if (MRT) {
        const V m7 = ((f[1] + f[2]) - (f[3] + f[4])) - m7eq;
        const V m8 = ((f[5] + f[6]) - (f[7] + f[8])) - m8eq;
        const V s = fma2(-0.25f, omega, V(0.25f));  // (1 - w) / 4
        const V c7 = s * m7, c8 = s * m8;
        fo[1] = fe[1] + c7;
        fo[2] = fe[2] + c7;
        fo[3] = fe[3] - c7;
        fo[4] = fe[4] - c7;
        fo[5] = fe[5] + c8;
        fo[6] = fe[6] + c8;
        fo[7] = fe[7] - c8;
        fo[8] = fe[8] - c8;
        // momentum rows: j - j^eq is zero except on Step-2 rows, where the
        // literal rate 0 keeps it (the alternative reading relaxes it)
        if (step2 && !step2_relax_j) {
            const V cx = div_const2<6>(jx), cy = div_const2<6>(jy);
            const V cp = cx + cy, cm = cy - cx;
            fo[1] = fo[1] + cx;
            fo[2] = fo[2] - cx;
            fo[3] = fo[3] + cy;
            fo[4] = fo[4] - cy;
            fo[5] = fo[5] + cp;
            fo[6] = fo[6] - cp;
            fo[7] = fo[7] + cm;
            fo[8] = fo[8] - cm;
        }
    } else {
        const V k = V(1.f) - omega;
#pragma unroll
        for (int i = 1; i < 9; ++i) fo[i] = fma2(k, f[i] - fe[i], fe[i]);
    }
    fo[0] = drho - ((((fo[1] + fo[2]) + (fo[3] + fo[4])) + ((fo[5] + fo[6]) + (fo[7] + fo[8]))));
    uxe_out = uxe;
    uye_out = uye;
}

}  // namespace lbfe
