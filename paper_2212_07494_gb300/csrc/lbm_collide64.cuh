// lbm_collide64.cuh -- FP64 collisions with fewer FP64 instructions.
//
// GB300's FP64 pipe issues 2 fused multiply-adds per clock and SM (measured:
// 1.254 TFLOP/s on 152 SMs at 2.07 GHz), so an FP64 step is bound by the
// number of FP64 instructions per node and by nothing else: 136 per node for
// the shared trimmed collision on D2Q9 (4.6 GLUPS; HBM would allow 47).  The
// functions here are the same maps as collide_smrt_trim<D2Q9> and
// collide_bgk of lbm_device.cuh, factored so that each opposite pair of
// populations shares its even and odd parts and every D1Q3 reconstruction
// line takes four instructions: about 80 per node, for D2Q9.  Measured (us a
// step, before and after): 512^2 SMRT 63.4 and 46.5, 64 x 32 BGK (one warp per
// scheduler, 64 clocks an instruction) 7.65 and 4.26.  Against a long double
// reference one collision is closer than the shared form's (relative error
// 1.28e-16 against 1.72e-16 for SMRT, 1.49e-16 against 1.86e-16 for BGK).
// Runs of the two SMRT forms drift apart by more than that, 3.7e-13 after 600
// steps of a 50 x 200 channel: in double the line weights 1/6 + 2/3 + 1/6 add
// up to 1 - 5.6e-17, so the shared reconstruction, which multiplies by them,
// loses that share of mass and momentum per line and step (mean momentum lost
// per collision at j = 0.05: 7.6e-18 +- 0.1e-18; here 0 +- 0.07e-18), as does
// any reference written with those three constants.
#pragma once
#include "lbm_device.cuh"

namespace lbm {

// 1 / r without the division subroutine's FP64 instructions: a hardware
// estimate x0 (relative error e <= 2^-20) and one third-order step of
// Halley's iteration for the reciprocal, x0 (1 + e + e^2), whose remaining
// error e^3 = 2^-60 is below FP64 rounding.  Values whose estimate is zero,
// infinite or NaN take the plain division.
__host__ __device__ __forceinline__ double recip64(double r) {
#ifdef __CUDA_ARCH__
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(r));
    const unsigned ex = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
    if (ex == 0u || ex == 0x7ffu) return 1.0 / r;
#else
    const double x = (double)(1.0f / (float)r);
#endif
    const double e = fma(-r, x, 1.0);
    return fma(x, fma(e, e, e), x);
}

// one D1Q3 reconstruction line: t0 plain, t1 and t2 halved; out: populations
// for c = -1, 0, +1 with the weights 1/6, 2/3, 1/6 folded in
__host__ __device__ __forceinline__ void recon_line_half(double &t0, double &t1, double &t2) {
    const double e = fma(t0, 1.0 / 6.0, t2);
    const double z = fma(-2.0, e, t0);   // 2/3 t0 - 2 t2
    t0 = e - t1;
    t2 = e + t1;
    t1 = z;
}

// SMRT with tau_3 = tau_4 = 1 on D2Q9 (collide_smrt_trim): G on the 3 x 3
// velocity grid, x fastest
__host__ __device__ __forceinline__ void collide_smrt_trim64(double *G, double gx, double gy, double om2) {
    // projection: sums s, differences d along x per row, then along y
    const double sm = G[2] + G[0], dm = G[2] - G[0];
    const double s0 = G[5] + G[3], d0 = G[5] - G[3];
    const double sp = G[8] + G[6], dp = G[8] - G[6];
    const double nm = sm + G[1], n0 = s0 + G[4], np = sp + G[7];
    const double S = np + nm;
    const double drho = S + n0;
    const double jy = np - nm;
    const double jx = (dp + dm) + d0;
    const double m11 = dp - dm;
    const double m20 = fma(-1.0 / 3.0, drho, (sp + sm) + s0);   // sum of (2 s - z)/3 = s - n/3
    const double m02 = fma(-1.0 / 3.0, drho, S);
    const double rho = 1.0 + drho;
    const double inv = recip64(rho);
    const double hx = 0.5 * gx, hy = 0.5 * gy;
    const double ux = fma(jx, inv, hx), uy = fma(jy, inv, hy);   // Eq. (half_F)
    // second-order central moments, relaxed: with rho u = j + p, p = F/2,
    //   c20 = m20 - ux (2 jx - rho ux) = m20 - ux (jx - px)
    //   c11 = m11 - ux jy - uy jx + rho ux uy = m11 - ux jy + px uy
    const double px = rho * hx, py = rho * hy;
    const double k = 1.0 - om2, k2 = 0.5 * k, k4 = 0.25 * k;
    const double A = k2 * fma(-ux, jx - px, m20);          // c20 / 2
    const double C = k2 * fma(-uy, jy - py, m02);          // c02 / 2
    const double B = k4 * fma(px, uy, fma(-ux, jy, m11));  // c11 / 4
    // back to raw moments (shift by +u), first along x, then along y; a first
    // or second order along an axis is kept halved, which is what the
    // reconstruction line takes.  The first-order raw moments are the
    // momentum plus the force, j + 2 p, taken from j itself: the rounding of
    // 1 / rho then never enters the momentum of a later step
    const double qx = 0.5 * px, qy = 0.5 * py;             // c10 / 2, c01 / 2
    const double vx = 0.5 * ux, vy = 0.5 * uy;
    // rows of y-order 0: (rho, r1, r2), 1: (qy, s1, s2), 2: (C, t1, t2)
    const double r1 = fma(0.5, jx, px);
    const double r2 = fma(ux, r1 + qx, A);
    const double s1 = fma(vx, qy, B);
    const double s2 = ux * (s1 + B);
    const double t1 = vx * C;
    const double t2 = ux * t1;
    double M[9];
    M[0] = drho;                                           // deviation from the weights
    M[3] = fma(0.5, jy, py);
    M[6] = fma(uy, M[3] + qy, C);
    M[1] = r1;
    M[4] = fma(vy, r1, s1);
    M[7] = fma(uy, M[4] + s1, t1);
    M[2] = r2;
    M[5] = fma(vy, r2, s2);
    M[8] = fma(uy, M[5] + s2, t2);
#pragma unroll
    for (int r = 0; r < 3; ++r) recon_line_half(M[3 * r], M[3 * r + 1], M[3 * r + 2]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        recon_line_half(M[c], M[3 + c], M[6 + c]);
        G[c] = M[c];
        G[3 + c] = M[3 + c];
        G[6 + c] = M[6 + c];
    }
}

// BGK with the second-order equilibrium and Guo-form force (collide_bgk).
// Per opposite pair (i, i'), om deq + F = w (E +- O), with rho u = j + rho g/2:
//   O = c.h,                              h = 3 (om j + rho g)
//   E = om drho + (c.u)(c.k) - u.k / 3,   k = 1.5 h + 4.5 (1 - om/2) rho g
template <int L> __host__ __device__ __forceinline__ void collide_bgk64(double *G, double gx, double gy, double gz,
                                                                       double om) {
    constexpr int D = Lat<L>::D, Q = Lat<L>::Q;
    const double g[3] = {gx, gy, gz};
    double drho = G[gpos<L>(0)], j[3] = {0.0, 0.0, 0.0};
    static_for<Q>([&](auto I) {
        constexpr int i = decltype(I)::value, o = opp<L>(i);
        if constexpr (i > 0 && i < o) {
            const double s = G[gpos<L>(i)] + G[gpos<L>(o)], d = G[gpos<L>(i)] - G[gpos<L>(o)];
            drho += s;
            if constexpr (Lat<L>::cx(i) != 0) j[0] += Lat<L>::cx(i) > 0 ? d : -d;
            if constexpr (Lat<L>::cy(i) != 0) j[1] += Lat<L>::cy(i) > 0 ? d : -d;
            if constexpr (D == 3 && Lat<L>::cz(i) != 0) j[2] += Lat<L>::cz(i) > 0 ? d : -d;
        }
    });
    const double rho = 1.0 + drho, inv = recip64(rho);
    const double om3 = 3.0 * om, f15 = 1.5 - 0.75 * om, rho3 = 3.0 * rho;
    double u[3] = {0.0, 0.0, 0.0}, h[3] = {0.0, 0.0, 0.0}, k[3] = {0.0, 0.0, 0.0}, P[3] = {0.0, 0.0, 0.0};
    double sum = 0.0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        u[a] = fma(j[a], inv, 0.5 * g[a]);
        const double rg = rho3 * g[a];
        h[a] = fma(om3, j[a], rg);
        k[a] = fma(1.5, h[a], f15 * rg);
        P[a] = u[a] * k[a];
        sum = a == 0 ? P[a] : sum + P[a];
    }
    const double base = fma(-1.0 / 3.0, sum, om * drho);
    const double txy = fma(u[0], k[1], u[1] * k[0]);
    const double txz = D == 3 ? fma(u[0], k[2], u[2] * k[0]) : 0.0;
    const double tyz = D == 3 ? fma(u[1], k[2], u[2] * k[1]) : 0.0;
    const double keep = 1.0 - om;
    G[gpos<L>(0)] = fma(weight<L>(0), base, keep * G[gpos<L>(0)]);
    static_for<Q>([&](auto I) {
        constexpr int i = decltype(I)::value, o = opp<L>(i);
        if constexpr (i > 0 && i < o) {
            constexpr int cx = Lat<L>::cx(i), cy = Lat<L>::cy(i), cz = Lat<L>::cz(i);
            double E = base, O = 0.0;
            if constexpr (cx != 0) E += P[0];
            if constexpr (cy != 0) E += P[1];
            if constexpr (cz != 0) E += P[2];
            if constexpr (cx * cy != 0) E += cx * cy > 0 ? txy : -txy;
            if constexpr (cx * cz != 0) E += cx * cz > 0 ? txz : -txz;
            if constexpr (cy * cz != 0) E += cy * cz > 0 ? tyz : -tyz;
            if constexpr (cx != 0) O += cx > 0 ? h[0] : -h[0];
            if constexpr (cy != 0) O += cy > 0 ? h[1] : -h[1];
            if constexpr (cz != 0) O += cz > 0 ? h[2] : -h[2];
            constexpr double w = weight<L>(i);
            G[gpos<L>(i)] = fma(w, E + O, keep * G[gpos<L>(i)]);
            G[gpos<L>(o)] = fma(w, E - O, keep * G[gpos<L>(o)]);
        }
    });
}

}  // namespace lbm
