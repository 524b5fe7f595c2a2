// lbm_f64.cuh -- the FP64 node update for the two compile-time rate patterns
// (kRatesPaper, kRatesPaperRaw), written for the fewest FP64 operations.
//
// What bounds it: the FP64 pipe, which issues 1.6 operations per SM and cycle
// on this chip (integer instructions: about 100).  The general form of
// lbm_device.cuh takes 383 FP64 operations per node (0.71 ns of the whole GPU, 86 %
// of it that pipe).  Here (ncu counters, 32 batched cases of 1.89 M nodes, one
// step): 280 by the algebra below, 1342 -> 1005 us; 202 with the sums of
// populations and of the phi stencil in 64-bit integers (lbm_fix64.cuh), 724 us,
// the pipe still 87 % busy.  The integers also round once where the sums rounded
// at every addition: one step's error against 80-bit arithmetic fell from
// 1.25e-16 to 0.88e-16 (f) and from 2.1e-15 to 0.75e-15 (g) of their 2-norms on
// a 64 x 128 oscillating drop.
// The rate pattern fixes:
//   * the phase-field collision acts on four differences of populations, not
//     on nine moments: with t = s chi + (1 - s/2) R and T = r phi,
//       (f_1 - f_3)+ / 2 = (1 - s)/2 (f_1 - f_3) + t / 3, and the diagonal
//       part (1 - s)/4 e + t / 12, e = f_5 - f_7 - f_6 + f_8 (the same in r);
//       the even part is T w_i;
//   * a unit rate on the momenta gives m+ = J + F (the definition of u,
//     Eq. 32, in r rho u + F / 2), so Eq. 36's r rho u is never formed there;
//   * the interface normal enters as one factor of grad phi (Eq. 2, Eq. 38).
// Reciprocals and square roots start from the hardware's FP64 approximations
// (MUFU, 15.7 per SM and cycle) and take one third-order step, 3 and 5
// operations instead of the 4.5 and 7.6 of the rounded library forms.
#pragma once

#include "lbm_device.cuh"

namespace axilbm {

// One cell of the phi window: phi = m 2^(e - 1075), m with its sign.
struct Win64 {
    long long* m;
    int* e;
    __device__ __forceinline__ void put(int c, double x) const {
        const int hi = __double2hiint(x), ex = exp64(x);
        const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
        const long long v = (long long)(((unsigned long long)mh << 32) | (uint32_t)__double2loint(x));
        const long long sg = (long long)(hi >> 31);
        m[c] = ex == 0 ? 0ll : (v ^ sg) - sg;
        e[c] = ex;
    }
};

// The stencils of Eq. 39-40 in the block of their 17 values, times 72:
//   72 grad = 4 (8 X_1 - X_2) + (8 D_1 - D_2) with X, D the differences of the
// axis and diagonal values one and two links away,
//   72 lap = 4 (16 A_1 - A_2) + 16 B_1 - B_2 with A, B the sums of the axis and
// diagonal values minus four times the centre.
template <int LD>
__device__ __forceinline__ void stencil64(const Win64& W, int a, int b, double& gz, double& gr, double& lap) {
    constexpr int K = 3;  // |72 grad| <= 108 and 9 |lap| <= 80 largest values: below 2^63
    const int c = a * LD + b;
    int E = max(W.e[c], kMinE);
    int ex[2][9];
#pragma unroll
    for (int i = 1; i < 9; ++i) {
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            ex[n][i] = W.e[c + (n + 1) * (cz_of(i) * LD + cr_of(i))];
            E = max(E, ex[n][i]);
        }
    }
    long long x[2][9];
#pragma unroll
    for (int i = 1; i < 9; ++i) {
#pragma unroll
        for (int n = 0; n < 2; ++n)
            x[n][i] = (W.m[c + (n + 1) * (cz_of(i) * LD + cr_of(i))] << K) >> min(E - ex[n][i], 63);
    }
    const long long c4 = ((W.m[c] << K) >> min(E - W.e[c], 63)) * 4;
    long long X[2], Y[2], Z[2], R[2], A[2], B[2];
#pragma unroll
    for (int n = 0; n < 2; ++n) {
        const long long d57 = x[n][5] - x[n][7], d68 = x[n][6] - x[n][8];
        X[n] = x[n][1] - x[n][3];
        Y[n] = x[n][2] - x[n][4];
        Z[n] = d57 - d68;
        R[n] = d57 + d68;
        A[n] = (x[n][1] + x[n][3]) + (x[n][2] + x[n][4]) - c4;
        B[n] = (x[n][5] + x[n][7]) + (x[n][6] + x[n][8]) - c4;
    }
    const bool bad = E >= kBadE;
    gz = bad ? nan64() : unfix64<K>(X[0] * 32 - X[1] * 4 + Z[0] * 8 - Z[1], E);
    gr = unfix64<K>(Y[0] * 32 - Y[1] * 4 + R[0] * 8 - R[1], E);
    // 9 lap in units of the block, from values of at most 8 (A, B)
    lap = unfix64<K - 3>(A[0] * 8 - (A[1] >> 1) + B[0] * 2 - (B[1] >> 3), E);
}

// What the collisions take from a node's own populations.
struct Pre64 {
    double T;             // sum f = r phi
    double fz, fe, fr, fo;  // f_1 - f_3, f_5 - f_7 - f_6 + f_8, f_2 - f_4, f_5 - f_7 + f_6 - f_8
    double S0;            // g_1 + .. + g_8
    double q;             // the even moment that relaxes with 1/tau_g: M g's e, raw: sum c^2 g
    double Jz, Jr;        // sum c g
    double m7, m8;        // sum (c_z^2 - c_r^2) g, sum c_z c_r g
};

template <int RM>
__device__ __forceinline__ void pre64(const double* fd, const double* gd, Pre64& P) {
    {
        const int E = block_exp<9>(fd);
        long long f[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = fix64<kPopK>(fd[i], E);
        const double T = unfix64<kPopK>((f[0] + f[1] + f[2]) + (f[3] + f[4] + f[5]) + (f[6] + f[7] + f[8]), E);
        P.T = E >= kBadE ? nan64() : T;
        const long long f57 = f[5] - f[7], f68 = f[6] - f[8];
        P.fz = unfix64<kPopK>(f[1] - f[3], E);
        P.fe = unfix64<kPopK>(f57 - f68, E);
        P.fr = unfix64<kPopK>(f[2] - f[4], E);
        P.fo = unfix64<kPopK>(f57 + f68, E);
    }
    {
        const int E = block_exp<9>(gd);
        long long g[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = fix64<kPopK>(gd[i], E);
        const long long s13 = g[1] + g[3], s24 = g[2] + g[4], s57 = g[5] + g[7], s68 = g[6] + g[8];
        const long long d57 = g[5] - g[7], d68 = g[6] - g[8];
        const long long a14 = s13 + s24, a58 = s57 + s68;
        P.S0 = unfix64<kPopK>(a14 + a58, E);
        P.q = unfix64<kPopK>(RM == kRatesPaperRaw ? a58 * 2 + a14 : a58 * 2 - a14 - g[0] * 4, E);
        const double Jz = unfix64<kPopK>((g[1] - g[3]) + (d57 - d68), E);
        P.Jz = E >= kBadE ? nan64() : Jz;
        P.Jr = unfix64<kPopK>((g[2] - g[4]) + (d57 + d68), E);
        P.m7 = unfix64<kPopK>(s13 - s24, E);
        P.m8 = unfix64<kPopK>(s57 - s68, E);
    }
}

// What the update takes from a node's column, r = j + 1/2.
struct Col64 {
    double r, inv_r, i6, i4, i2, r03, r3, r72;  // r, 1/r, 0.6/r, -4/(15 r), -2/r, r/0.3, 3 r, r/72
};
__device__ __forceinline__ Col64 col64(int j, double inv_r) {
    const double r = (double)j + 0.5;
    return Col64{r, inv_r, 0.6 * inv_r, (-4.0 / 15.0) * inv_r, -2.0 * inv_r, (1.0 / 0.3) * r, 3.0 * r, (1.0 / 72.0) * r};
}
// The columns of a tile in shared memory, filled once per CTA (five operations
// per column instead of per node).
struct ColTab64 {
    double v[8][32];
    __device__ __forceinline__ void put(int x, const Col64& c) {
        v[0][x] = c.r, v[1][x] = c.inv_r, v[2][x] = c.i6, v[3][x] = c.i4, v[4][x] = c.i2, v[5][x] = c.r03, v[6][x] = c.r3, v[7][x] = c.r72;
    }
    __device__ __forceinline__ Col64 get(int x) const {
        return Col64{v[0][x], v[1][x], v[2][x], v[3][x], v[4][x], v[5][x], v[6][x], v[7][x]};
    }
};

// Macroscopic step, both collisions and both inverse transforms of a node of
// column constants K; the phi window is centred on (a, b).
template <int LD, int RM>
__device__ __forceinline__ void update64(const CaseDev& C, const Win64& W, int a, int b, double phi, const Col64& K,
                                         const Pre64& Q, double chz_prev, double chr_prev, double p_prev, double* fp,
                                         double* gp, double& chz, double& chr, double& p_out) {
    static_assert(RM == kRatesPaper || RM == kRatesPaperRaw, "a compile-time rate pattern");
    constexpr bool kRaw = RM == kRatesPaperRaw;
    const CaseReal<double>& P = C.pd;
    const Case64& H = C.p64;
    double gz, gr, lap;  // 72 grad phi, 72 lap phi
    stencil64<LD>(W, a, b, gz, gr, lap);
    const double rho = fma(phi, H.drho, P.rho_g);               // Eq. 17
    const double nu = fma(phi, H.dnu, P.nu_g);                  // Eq. 35
    const double tau = fma(3.0, nu, 0.5);                       // Eq. 34
    // 1 / tau_g, 1 / (r rho + nu rho / r) and 1 / (r rho) of Eq. 32
    const double s = rcp64(tau);
    const double rv = fma(nu, K.inv_r, K.r);
    const double D = rcp64(rho * rv);
    const double irr = K.inv_r * (D * rv);
    // Eq. 4, mu~ = mu - k d_r phi / r, and Eq. 30's F_z = r (F_s + G)_z
    const double w = fma(phi, phi - 1.5, 0.5);                  // (phi - 1)(phi - 1/2)
    const double mut = fma(H.beta4 * phi, w, H.mkappa * fma(gr, K.inv_r, lap));
    const double rm = K.r72 * mut;
    const double Fz = fma(rm, gz, K.r * ((rho - P.rho_l) * P.grav_z));
    const double rFsr = rm * gr;
    const double Z3 = H.drho3 * gz, R3 = H.drho3 * gr;          // 0.3 grad rho
    const double uz = fma(0.5, Fz, Q.Jz) * irr;                 // Eq. 32 (z)
    const double rz = rho * uz;
    // Eq. 33 with s_p = tau_g / 2 (raw: 3 tau_g / 2 - 1)
    const double A2 = 0.4 * rho;
    const double A0 = fma(uz, fma(-A2, uz, Z3), K.i6 * Q.S0);
    const double sp = kRaw ? fma(1.5, tau, -1.0) : 0.5 * tau;
    double ur, p, ps;
    if (C.p_coupling == 1) {
        ps = p_prev;
        ur = fma(0.5, rFsr + ps, Q.Jr) * D;
        p = fma(ur, fma(sp * rho, K.i4, fma(-A2, ur, R3)), A0);
    } else {
        // u_r = ca + D p / 2 and p = A0 + A1 u_r - A2 u_r^2 together
        const double ca = fma(0.5, rFsr, Q.Jr) * D;
        const double A1 = fma(sp * rho, K.i4, R3);
        const double t1 = A2 * ca;
        const double qb = fma(D, fma(-0.5, A1, t1), 1.0);
        const double qc = fma(ca, A1 - t1, A0);
        const double disc = fma((A2 * D) * D, qc, qb * qb);
        const bool two = __double2hiint(disc) >= 0;  // the sign bit: a comparison would take the FP64 pipe
        p = (two ? qc + qc : qc) * rcp64(two ? qb + sqrt64(disc) : qb);
        ps = p;
        ur = fma(0.5 * D, p, ca);
    }
    const double rr = rho * ur;
    const double Fr = fma(K.i2, nu * rr, rFsr + ps);    // Eq. 30 (r)
    p_out = p;
    // phase field (Eq. 19-23, 38): chi, then t / 3 of both directions
    chz = Q.T * uz;
    chr = fma(Q.T, ur, P.mob * phi);
    {
        // r lambda / (3 (|grad phi| + n_eps)): the normal's factor of grad phi
        const double lam = H.lam3 * (K.r * fma(-phi, phi, phi));
        const double L = lam * rcp64(sqrt64(fma(gz, gz, gr * gr)) + H.neps72);
        const double tz = fma(H.h3, fma(L, gz, -chz_prev), H.sh3 * chz);
        const double tr = fma(H.h3, fma(L, gr, -chr_prev), H.sh3 * chr);
        const double jz = fma(H.c2, Q.fz, tz), jr = fma(H.c2, Q.fr, tr);
        const double qz = fma(0.25, tz, H.c4 * Q.fe), qr = fma(0.25, tr, H.c4 * Q.fo);
        const double e = Q.T * (1.0 / 9.0), d = Q.T * (1.0 / 36.0);
        const double qp = qz + qr, qm = qz - qr;
        fp[0] = Q.T * (4.0 / 9.0);
        fp[1] = e + jz;
        fp[3] = e - jz;
        fp[2] = e + jr;
        fp[4] = e - jr;
        fp[5] = d + qp;
        fp[7] = d - qp;
        fp[8] = d + qm;
        fp[6] = d - qm;
    }
    // hydrodynamics (Eq. 24, 36-37)
    const double az = K.r03 * Z3, br = fma(K.r03, R3, rho);               // grad (r rho)
    const double P1 = uz * az, P2 = ur * br, udr = P1 + P2;
    const double E1 = rz * uz, E2 = rr * ur, E = E1 + E2;       // rho u^2
    const double pK = fma(2.0, p, E);
    const double c = 1.0 - s, h2 = 2.0 - s;                     // 1 - s, 2 (1 - s/2)
    const double h6 = h2 * (1.0 / 6.0);
    const double jz = Q.Jz + Fz, jr = Q.Jr + Fr;                // unit rates on the momenta
    const double m7 = fma(2.0 * h6, P1 - P2, fma(s, K.r * (E1 - E2), c * Q.m7));
    const double m8 = fma(h6, fma(uz, br, ur * az), fma(s, (K.r * rr) * uz, c * Q.m8));
    const double m0 = 0.5 * (udr - rr);
    double ep, em, dp, dm;
    if constexpr (kRaw) {
        // raw moments: k_3 = sum c^2 g relaxes with 1/tau_g, k_0 and k_8 take
        // equilibrium and half the source
        const double k3 = fma(2.0 * h6, fma(2.0, udr, -rr), fma(s, K.r * pK, c * Q.q));
        const double k8 = fma(K.r3 * (1.0 / 9.0), p + E, fma(3.0, udr, -rr) * (1.0 / 18.0));
        gp[0] = (m0 - k3) + k8;
        const double ax = fma(-0.5, k8, 0.25 * k3);
        ep = fma(0.25, m7, ax);
        em = fma(-0.25, m7, ax);
        dp = 0.25 * (k8 + m8);
        dm = 0.25 * (k8 - m8);
    } else {
        const double m1 = fma(h2, rr, fma(s, K.r3 * pK, c * Q.q));
        const double m2 = fma(-K.r3, pK + p, -(m0 + rr));
        const double n0 = m0 * (1.0 / 9.0);
        gp[0] = fma(1.0 / 9.0, m2 - m1, n0);
        const double e = fma(-1.0 / 36.0, m1, fma(-1.0 / 18.0, m2, n0));
        const double d = fma(1.0 / 18.0, m1, fma(1.0 / 36.0, m2, n0));
        ep = fma(0.25, m7, e);
        em = fma(-0.25, m7, e);
        dp = fma(0.25, m8, d);
        dm = fma(-0.25, m8, d);
    }
    const double q1 = jz + jr, q2 = jz - jr;
    gp[1] = fma(1.0 / 3.0, jz, ep);
    gp[3] = fma(-1.0 / 3.0, jz, ep);
    gp[2] = fma(1.0 / 3.0, jr, em);
    gp[4] = fma(-1.0 / 3.0, jr, em);
    gp[5] = fma(1.0 / 12.0, q1, dp);
    gp[7] = fma(-1.0 / 12.0, q1, dp);
    gp[8] = fma(1.0 / 12.0, q2, dm);
    gp[6] = fma(-1.0 / 12.0, q2, dm);
}

}  // namespace axilbm
