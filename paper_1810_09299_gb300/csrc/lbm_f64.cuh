// lbm_f64.cuh -- the FP64 node update for the two compile-time rate patterns
// (kRatesPaper, kRatesPaperRaw), written for the fewest FP64 operations.
//
// What bounds it: the FP64 pipe issues 1.6 operations per SM and cycle on this
// chip, the integer pipes about 100 instructions.  The general form of
// lbm_device.cuh takes 383 FP64 operations per node and is bound by that pipe.
// Here the sums of populations and of the phi stencil, both collisions, both
// inverse transforms, reciprocals and roots run in 64-bit integers
// (lbm_fix64.cuh); what depends on phi alone and the results' conversions stay
// on the FP64 pipe: 34.4 instructions per node there now (ncu, the phi ring's share
// and conversions included).  32 batched cases (1.89 M nodes), us a step; the counts
// are those written in the source, without the ring:
//   general form, 383 operations per node                          1342
//   the algebra below, 280                                         1005
//   sums of populations and of the stencil in integers, 202         724
//   collisions and inverse transforms in integers, 83               516
//   no IEEE fallbacks, cheaper conversions and normalisations, 55   408
//   shared alignments, the nine g converted on the FP64 pipe, 61    383
//   column constants from a table in device memory, 57              376
//   high-word multiplications; reciprocals and roots in integers, 29  331
//   every result converted on the FP64 pipe                         313
//   3 CTAs of 80 registers per SM                                   302
//   dropped bits given back on average, constants to 62 bits        309
// (Conversions in integers had been the better ones while the FP64 pipe was
// busier: 399 against 383 with all of them there, 61 operations.)  Now the ALU is 60 %
// and the FP64 pipe 34 % busy (ncu); timing-only copies without the
// mixed products of the multiplications, without the ring and without the
// sums' conversions ran 13, 6 and 6 % faster.
// The last line is for accuracy: integers that only drop bits err in one
// direction, which adds up over steps.  Error against 80-bit arithmetic, 2-norm,
// general form and here:
//                                        f                  g                  chi
//   drop 64 x 128, 1 step         1.25e-16 0.70e-16  2.1e-15 0.72e-15  2.5e-16 0.94e-16
//                   10 steps       5.8e-16  4.9e-16  1.6e-14  1.7e-15  1.9e-15  4.9e-16
//   bubble 96 x 300, 1 step       1.26e-16 0.72e-16  2.7e-16  1.1e-16  1.6e-16 0.88e-16
//                   10 steps       6.9e-16  5.0e-16  1.5e-15  1.0e-15  9.8e-16  5.8e-16
// The rate pattern fixes:
//   * the phase-field collision acts on four differences of populations, not
//     on nine moments: with t = s chi + (1 - s/2) R and T = r phi,
//       (f_1 - f_3)+ / 2 = (1 - s)/2 (f_1 - f_3) + t / 3, and the diagonal
//       part (1 - s)/4 e + t / 12, e = f_5 - f_7 - f_6 + f_8 (the same in r);
//       the even part is T w_i;
//   * a unit rate on the momenta gives m+ = J + F (the definition of u,
//     Eq. 32, in r rho u + F / 2), so Eq. 36's r rho u is never formed there;
//   * the interface normal enters as one factor of grad phi (Eq. 2, Eq. 38).
#pragma once

#include "lbm_device.cuh"

namespace axilbm {

constexpr int kWinK = 3;  // 72 grad of at most 108 and 9 lap of at most 80 largest values stay below 2^63
// One cell of the phi window: phi = m 2^(e - 1075 - kWinK), m with its sign.
struct Win64 {
    long long* m;
    int* e;
    __device__ __forceinline__ void put(int c, double x) const {
        const int hi = __double2hiint(x), ex = exp64(x);
        const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
        const long long v = (long long)((((unsigned long long)mh << 32) | (uint32_t)__double2loint(x)) << kWinK);
        const long long sg = (long long)(hi >> 31);
        m[c] = (v ^ sg) - sg;  // zero (ex = 0) leaves every block: E - ex >= kMinE
        e[c] = ex;
    }
};

// v 2^e with |v| < 2^63, normalised
__device__ __forceinline__ Sf norm_any(long long v, int e) { return norm(Sf{v >> 1, e + 1}); }

// The stencils of Eq. 39-40 in the block of their 17 values, times 72:
//   72 grad = 4 (8 X_1 - X_2) + (8 D_1 - D_2) with X, D the differences of the
// axis and diagonal values one and two links away,
//   72 lap = 4 (16 A_1 - A_2) + 16 B_1 - B_2 with A, B the sums of the axis and
// diagonal values minus four times the centre.
template <int LD>
__device__ __forceinline__ void stencil64(const Win64& W, int a, int b, Sf& gz, Sf& gr, Sf& lap, bool& bad) {
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
            x[n][i] = shr64(W.m[c + (n + 1) * (cz_of(i) * LD + cr_of(i))], E - ex[n][i]);
    }
    const long long c4 = shr64(W.m[c], E - W.e[c]) * 4;
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
    const int e = E - 1075 - kWinK;
    gz = norm_any(X[0] * 32 - X[1] * 4 + Z[0] * 8 - Z[1], e);
    gr = norm_any(Y[0] * 32 - Y[1] * 4 + R[0] * 8 - R[1], e);
    // 9 lap in units of the block, from values of at most 8 (A, B)
    lap = norm_any(A[0] * 8 - (A[1] >> 1) + B[0] * 2 - (B[1] >> 3), e + 3);
    bad = E >= kBadE;
}

// What the collisions take from a node's own populations: sum f = r phi as a
// double, the differences that the phase-field collision acts on in the block
// of f, and the moments of g.
struct Pre64 {
    double T;
    int Ef;                    // the block exponent of f
    bool bad;                  // a value out of the range of the sums, infinite or NaN
    long long t, fz, fe, fr, fo;  // sum f, f_1 - f_3, f_5 - f_7 - f_6 + f_8, f_2 - f_4, f_5 - f_7 + f_6 - f_8
    Sf S0;                     // g_1 + .. + g_8
    Sf q;                      // the even moment that relaxes with 1/tau_g: M g's e, raw: sum c^2 g
    Sf Jz, Jr;                 // sum c g
    Sf m7, m8;                 // sum (c_z^2 - c_r^2) g, sum c_z c_r g
};

__device__ __forceinline__ void pre64_f(const double* fd, Pre64& P) {
    const int E = block_exp<9>(fd);
    long long f[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = fix64<kPopK>(fd[i], E);
    P.Ef = E;
    P.t = (f[0] + f[1] + f[2]) + (f[3] + f[4] + f[5]) + (f[6] + f[7] + f[8]);
    P.T = unfix64<kPopK>(P.t, E);
    P.bad = E >= kBadE;
    if (P.bad) P.T = nan64();
    const long long f57 = f[5] - f[7], f68 = f[6] - f[8];
    P.fz = f[1] - f[3];
    P.fe = f57 - f68;
    P.fr = f[2] - f[4];
    P.fo = f57 + f68;
}
template <int RM>
__device__ __forceinline__ void pre64_g(const double* gd, Pre64& P) {
    const int E = block_exp<9>(gd);
    const int e = E - 1075 - kPopK;
    long long g[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = fix64<kPopK>(gd[i], E);
    const long long s13 = g[1] + g[3], s24 = g[2] + g[4], s57 = g[5] + g[7], s68 = g[6] + g[8];
    const long long d57 = g[5] - g[7], d68 = g[6] - g[8];
    const long long a14 = s13 + s24, a58 = s57 + s68;
    P.S0 = norm_any(a14 + a58, e);
    P.q = norm_any(RM == kRatesPaperRaw ? a58 * 2 + a14 : a58 * 2 - a14 - g[0] * 4, e);
    P.Jz = norm_any((g[1] - g[3]) + (d57 - d68), e);
    P.Jr = norm_any((g[2] - g[4]) + (d57 + d68), e);
    P.m7 = norm_any(s13 - s24, e);
    P.m8 = norm_any(s57 - s68, e);
    P.bad = P.bad || E >= kBadE;
}
template <int RM>
__device__ __forceinline__ void pre64(const double* fd, const double* gd, Pre64& P) {
    pre64_f(fd, P);
    pre64_g<RM>(gd, P);
}

// What the update takes from a node's column, r = j + 1/2.
struct Col64 {
    double r, inv_r;                          // r, 1/r
    Sf sr, s_inv_r, s_i6, s_i4, r03, r3, r72;  // r, 1/r, 0.6/r, -2/(15 r), r/0.3, 3 r, r/72
};
__device__ __forceinline__ Col64 col64(int j) {
    const double r = (double)j + 0.5;
    bool bad = false;
    const Sf s = sf_of(r), i = rcp(s, bad);
    return Col64{r, rcp_(r), s, i, norm(i * Sf{0x2666666666666666ll, -62}), neg(norm(i * Sf{0x2222222222222222ll, -64})),
                 norm(s * Sf{0x3555555555555555ll, -60}), sf_of(3.0 * r), norm(s * Sf{0x38e38e38e38e38e4ll, -68})};
}
constexpr int kColSf = 7;
// The columns 0 .. n - 1 of a handle in device memory, filled once when it is
// created: with them formed per tile in shared memory the window waited for a
// chain of FP64 operations behind a barrier of its own.
struct ColTab64 {
    const double* d;  // [2][n] doubles, then Sf [kColSf][n]
    int n;
    __device__ __forceinline__ double inv_r(int j) const { return __ldg(d + n + j); }
    __device__ __forceinline__ const longlong2* sf(int i) const {
        return reinterpret_cast<const longlong2*>(d + 2 * n) + (int64_t)i * n;
    }
    __device__ __forceinline__ struct ColRef64 at(int j) const;
};
// One column of the table, its values loaded where they are used.
struct ColRef64 {
    ColTab64 t;
    int j;
    __device__ __forceinline__ double dv(int i) const {
        double v;
        asm("ld.global.nc.f64 %0, [%1];" : "=d"(v) : "l"(t.d + i * t.n + j));
        return v;
    }
    __device__ __forceinline__ Sf sv(int i) const {
        long long m, e;
        asm("ld.global.nc.v2.s64 {%0, %1}, [%2];" : "=l"(m), "=l"(e) : "l"(t.sf(i) + j));
        return Sf{m, (int)e};
    }
    __device__ __forceinline__ double r() const { return dv(0); }
    __device__ __forceinline__ double inv_r() const { return dv(1); }
    __device__ __forceinline__ Sf sr() const { return sv(0); }
    __device__ __forceinline__ Sf s_inv_r() const { return sv(1); }
    __device__ __forceinline__ Sf s_i6() const { return sv(2); }
    __device__ __forceinline__ Sf s_i4() const { return sv(3); }
    __device__ __forceinline__ Sf r03() const { return sv(4); }
    __device__ __forceinline__ Sf r3() const { return sv(5); }
    __device__ __forceinline__ Sf r72() const { return sv(6); }
};
__device__ __forceinline__ ColRef64 ColTab64::at(int j) const { return ColRef64{*this, j}; }
// 16 bytes per column and Sf, 8 per double
constexpr size_t col_tab64_bytes(int n) { return (size_t)n * (2 * 8 + kColSf * 16); }

// a's integer in units of 2^e, e >= a.e
__device__ __forceinline__ long long in_units(Sf a, int e) { return shr64(a.m, e - a.e); }

// The macroscopic step of a node of column constants K; the phi window is
// centred on (a, b).  What depends on phi alone stays on the FP64 pipe,
// the rest runs beside it in integers.
struct Macro64 {
    Sf gz, gr, Z3, R3;     // 72 grad phi; 0.3 grad rho
    double nu;
    Sf rho, s;             // s = 1 / tau_g
    Sf uz, rz, ur, p, ps;  // rz = rho u_z; ps: the p of Eq. 30 and Eq. 32
    Sf rFsr;               // r F_s,r
    Two JFz;               // J_z and F_z (Eq. 30)
    bool bad;              // a value out of the range of the sums, infinite or NaN
};
template <int LD, int RM>
__device__ __forceinline__ Macro64 macros64(const CaseDev& C, const Win64& W, int a, int b, double phi, const ColRef64& K,
                                            const Pre64& Q, double p_prev) {
    static_assert(RM == kRatesPaper || RM == kRatesPaperRaw, "a compile-time rate pattern");
    constexpr bool kRaw = RM == kRatesPaperRaw;
    const CaseReal<double>& P = C.pd;
    const Case64& H = C.p64;
    Macro64 m;
    Sf lap;  // 72 lap phi
    stencil64<LD>(W, a, b, m.gz, m.gr, lap, m.bad);
    const Sf gz = m.gz, gr = m.gr;
    // of phi alone: Eq. 17, 35, 34, then 1 / tau_g, 1 / (r rho + nu rho / r) and 1 / (r rho) of Eq. 32
    const double rho_d = fma(phi, H.drho, P.rho_g);
    const double nu = fma(phi, H.dnu, P.nu_g);
    const double tau = fma(3.0, nu, 0.5);
    const double rv = fma(nu, K.inv_r(), K.r());
    const Sf rho = sf_of(rho_d), st = sf_of(tau), s = rcp(st, m.bad), srv = sf_of(rv), D = rcp(rho * srv, m.bad);
    const Sf irr = K.s_inv_r() * (D * srv), sphi = sf_of(phi);
    // Eq. 4: mu~ = mu - k d_r phi / r; Eq. 30's F_z = r (F_s + G)_z
    const Sf mut = norm29((Sf{H.beta4_m, H.beta4_e} * sphi) * sf_of(fma(phi, phi - 1.5, 0.5)) +
                          Sf{H.mkappa_m, H.mkappa_e} * norm29(gr * K.s_inv_r() + lap));
    const Sf rm = K.r72() * mut;
    Sf Fz = rm * gz;
    if (abs_hi(P.grav_z) != 0) Fz = Fz + K.sr() * (sf_of(rho_d - P.rho_l) * Sf{H.grav_m, H.grav_e});
    const Sf rFsr = rm * gr;
    const Sf d3{H.drho3_m, H.drho3_e};
    const Sf Z3 = d3 * gz, R3 = d3 * gr;  // 0.3 grad rho
    const Two JFz = align(Q.Jz, Fz);
    const Sf uz = norm29(Sf{JFz.a + (JFz.b >> 1), JFz.e}) * irr;  // Eq. 32 (z)
    const Sf rz = rho * uz;
    // Eq. 33 with s_p = tau_g / 2 (raw: 3 tau_g / 2 - 1)
    const Sf A2 = rho * Sf{0x3333333333333333ll, -63};  // 0.4 rho
    const Sf A0 = uz * norm29(Z3 - A2 * uz) + K.s_i6() * Q.S0;
    const Sf A1 = norm29(sf_of((kRaw ? fma(1.5, tau, -1.0) : tau) * rho_d) * scale2(K.s_i4(), kRaw ? 1 : 0) + R3);
    // numbers that are not finite do not exist in integers: seen here, put out as NaN
    int top = max(abs_hi(rho_d), abs_hi(nu));
    Sf ur, p, ps;
    if (C.p_coupling == 1) {
        ps = sf_of(p_prev);
        top = max(top, abs_hi(p_prev));
        ur = norm29(scale2(rFsr + ps, -1) + Q.Jr) * D;
        p = norm29(ur * norm29(A1 - A2 * ur) + A0);
    } else {
        // u_r = ca + D p / 2 and p = A0 + A1 u_r - A2 u_r^2 together
        const Sf ca = norm29(scale2(rFsr, -1) + Q.Jr) * D;
        const Sf t1 = A2 * ca;
        const Sf one{1ll << 61, -61};
        const Two tA = align(t1, A1);
        const Sf qb = norm29(one + D * norm29(Sf{tA.a - (tA.b >> 1), tA.e}));
        const Sf qc = norm29(A0 + ca * norm29(Sf{tA.b - tA.a, tA.e}));
        const Sf disc = qb * qb + ((A2 * D) * D) * qc;
        const bool two = disc.m >= 0;
        const Sf sum = qb + root(Sf{two ? disc.m : 0ll, disc.e});
        p = scale2(qc, two ? 1 : 0) * rcp(sum, m.bad);
        ps = p;
        ur = norm29(ca + scale2(D, -1) * p);
    }
    m.bad = m.bad || Q.bad || top >= 0x7ff00000;
    m.Z3 = Z3, m.R3 = R3, m.nu = nu, m.rho = rho, m.s = s;
    m.uz = uz, m.rz = rz, m.ur = ur, m.p = p, m.ps = ps, m.rFsr = rFsr, m.JFz = JFz;
    return m;
}

// The macroscopic step, both collisions and both inverse transforms.
template <int LD, int RM>
__device__ __forceinline__ void update64(const CaseDev& C, const Win64& W, int a, int b, double phi, const ColRef64& K,
                                         const Pre64& Q, double chz_prev, double chr_prev, double p_prev, double* fp,
                                         double* gp, double& chz_out, double& chr_out, double& p_out) {
    constexpr bool kRaw = RM == kRatesPaperRaw;
    const Case64& H = C.p64;
    const Macro64 m = macros64<LD, RM>(C, W, a, b, phi, K, Q, p_prev);
    bool bad = m.bad;
    int top = max(abs_hi(chz_prev), abs_hi(chr_prev));
    const Sf gz = m.gz, gr = m.gr, Z3 = m.Z3, R3 = m.R3, rho = m.rho, s = m.s, uz = m.uz, rz = m.rz, ur = m.ur, p = m.p;
    const Two JFz = m.JFz;
    const Sf rr = rho * ur;
    const Sf Fr = (m.rFsr + m.ps) - scale2(sf_of(m.nu) * K.s_inv_r() * rr, 1);  // Eq. 30 (r)
    p_out = double_of(p);
    // phase field (Eq. 19-23, 38): chi, then t / 3 of both directions
    const Sf T = norm_any(Q.t, Q.Ef - 1075 - kPopK);
    const Sf chz = T * uz, chr = T * ur + Sf{H.mob_m, H.mob_e} * sf_of(phi);
    chz_out = double_of(chz);
    chr_out = double_of(chr);
    {
        // r lambda / (3 (|grad phi| + n_eps)): the normal's factor of grad phi (72 in both)
        const Sf lam = Sf{H.lam3_m, H.lam3_e} * K.sr() * sf_of_or_zero(fma(-phi, phi, phi));
        const Sf L = lam * rcp(root(gz * gz + gr * gr) + Sf{H.neps72_m, H.neps72_e}, bad);
        const Sf h3{H.h3_m, H.h3_e}, sh3{H.sh3_m, H.sh3_e};
        const Sf tz = h3 * norm29(L * gz - sf_of_or_zero(chz_prev)) + sh3 * chz;
        const Sf tr = h3 * norm29(L * gr - sf_of_or_zero(chr_prev)) + sh3 * norm29(chr);
        // the sums of the inverse transform in units of the largest part, 2^E
        // (the block's values take up to 63 bits)
        const int eb = Q.Ef - 1075 - kPopK;
        const int E = max(max(max(tz.e, tr.e), eb), -990), sb = E - eb;
        bad = bad || E > 890;
        const long long e = ninth_double(shr64(Q.t, sb));
        const long long tz0 = in_units(tz, E), tr0 = in_units(tr, E);
        const auto part = [&](long long v, long long c) { return v == 0 ? 0ll : mul62(shr64(v, sb), c); };
        const long long jz = part(Q.fz, H.c2) + tz0, jr = part(Q.fr, H.c2) + tr0;
        const long long qz = part(Q.fe, H.c4) + (tz0 >> 2), qr = part(Q.fo, H.c4) + (tr0 >> 2);
        const long long d = (e + 2) >> 2, qp = qz + qr, qm = qz - qr;
        fp[0] = double_cvt(e, E + 2);
        fp[1] = double_cvt(e + jz, E);
        fp[3] = double_cvt(e - jz, E);
        fp[2] = double_cvt(e + jr, E);
        fp[4] = double_cvt(e - jr, E);
        fp[5] = double_cvt(d + qp, E);
        fp[7] = double_cvt(d - qp, E);
        fp[8] = double_cvt(d + qm, E);
        fp[6] = double_cvt(d - qm, E);
    }
    // hydrodynamics (Eq. 24, 36-37)
    const Sf az = K.r03() * Z3, br = norm29(K.r03() * R3 + rho);      // grad (r rho)
    const Two PP = align(uz * az, ur * br);
    const Sf udr{PP.a + PP.b, PP.e};
    const Two E12 = align(rz * uz, rr * ur);
    const Two pE = align(scale2(p, 1), Sf{E12.a + E12.b, E12.e});  // 2 p and rho u^2
    const Sf pK = norm29(Sf{pE.a + pE.b, pE.e});
    const Two s1 = align(Sf{1ll << 61, -61}, s);                // 1 - s, 2 (1 - s/2) and a sixth of that
    const Sf c = norm29(Sf{s1.a - s1.b, s1.e}), h2 = norm29(Sf{s1.a - (s1.b >> 1), s1.e + 1}), h6{third64(h2.m), h2.e - 1};
    const Sf jz{JFz.a + JFz.b, JFz.e}, jr = Q.Jr + Fr;                    // unit rates on the momenta
    const Sf m7 = (c * Q.m7 + s * (K.sr() * norm29(Sf{E12.a - E12.b, E12.e}))) + scale2(h6, 1) * norm29(Sf{PP.a - PP.b, PP.e});
    const Sf m8 = (c * Q.m8 + s * norm29((K.sr() * rr) * uz)) + h6 * norm29(uz * br + ur * az);
    const Sf m0 = scale2(udr - rr, -1);
    // no part reaches one unit: g is zero (in_units makes -1 of the negative ones)
    constexpr int kRestE = -990 - 62;
    bool rest;
    if constexpr (kRaw) {
        // raw moments: k_3 = sum c^2 g relaxes with 1/tau_g, k_0 and k_8 take
        // equilibrium and half the source
        const Sf rr3{third64(rr.m), rr.e};
        const Sf k3 = (c * Q.q + s * (K.sr() * pK)) + scale2(h6, 1) * norm29(scale2(udr, 1) - rr);
        const Sf w = K.r3() * norm29(Sf{(pE.a >> 1) + pE.b, pE.e});   // 3 r (p + rho u^2)
        const Sf v = udr - rr3;             // 6 times the rest of k_8
        const int top_e = max(max(max(k3.e, m0.e), max(w.e, v.e)), max(max(m7.e, m8.e), max(jz.e, jr.e)));
        const int E = max(-994, top_e) + 4;
        bad = bad || E > 890;
        rest = top_e < kRestE;
        const long long M0 = in_units(m0, E), K3 = in_units(k3, E), M7 = in_units(m7, E), M8 = in_units(m8, E);
        const long long K8 = ninth64(in_units(w, E)) + (third64(in_units(v, E)) >> 1);
        const long long JZ = in_units(jz, E), JR = in_units(jr, E);
        // 12 g in units of 2^E
        const long long ax = K3 * 3 - K8 * 6, p7 = M7 * 3;
        gp[0] = double_cvt(M0 - K3 + K8, E);
        gp[1] = double_cvt(third64<2>(ax + p7 + JZ * 4), E - 2);
        gp[3] = double_cvt(third64(ax + p7 - JZ * 4), E - 2);
        gp[2] = double_cvt(third64(ax - p7 + JR * 4), E - 2);
        gp[4] = double_cvt(third64<0>(ax - p7 - JR * 4), E - 2);
        const long long dp = (K8 + M8) * 3, dm = (K8 - M8) * 3;
        gp[5] = double_cvt(third64<2>(dp + JZ + JR), E - 2);
        gp[7] = double_cvt(third64<2>(dp - JZ - JR), E - 2);
        gp[8] = double_cvt(third64(dm + JZ - JR), E - 2);
        gp[6] = double_cvt(third64(dm - JZ + JR), E - 2);
    } else {
        const Sf m1 = (c * Q.q + s * (K.r3() * pK)) + h2 * rr;
        const Sf m2 = neg((K.r3() * norm29(Sf{((pE.a + pE.b) >> 1) + (pE.a >> 2), pE.e + 1})) + (m0 + rr));
        // 36 g = 4 m0 - m1 - 2 m2 +- 9 m7 +- 12 j (axes), 4 m0 + 2 m1 + m2 +- 9 m8
        // +- 3 j (diagonals), 4 (m0 - m1 + m2) (rest), in units of 2^E: the
        // coefficients add up to 28 at most.  in_units leaves half a unit out on
        // average; with its coefficient that is -11 to 10 units of 36 g, so the
        // quotients take 0 to 2 units back.
        const int top_e = max(max(max(m0.e, m1.e), max(m2.e, jz.e)), max(max(m7.e, m8.e), jr.e));
        const int E = max(-994, top_e) + 4;
        bad = bad || E > 890;
        rest = top_e < kRestE;
        const long long M0 = in_units(m0, E) * 4, M1 = in_units(m1, E), M2 = in_units(m2, E);
        const long long M7 = in_units(m7, E) * 9, M8 = in_units(m8, E) * 9;
        const long long JZ = in_units(jz, E) * 3, JR = in_units(jr, E) * 3;
        const long long ax = M0 - M1 - M2 * 2, dg = M0 + M1 * 2 + M2;
        gp[0] = double_cvt(ninth64(M0 - (M1 - M2) * 4), E - 2);
        gp[1] = double_cvt(ninth64<2>(ax + M7 + JZ * 4), E - 2);
        gp[3] = double_cvt(ninth64(ax + M7 - JZ * 4), E - 2);
        gp[2] = double_cvt(ninth64(ax - M7 + JR * 4), E - 2);
        gp[4] = double_cvt(ninth64<0>(ax - M7 - JR * 4), E - 2);
        gp[5] = double_cvt(ninth64<2>(dg + M8 + JZ + JR), E - 2);
        gp[7] = double_cvt(ninth64<2>(dg + M8 - JZ - JR), E - 2);
        gp[8] = double_cvt(ninth64(dg - M8 + JZ - JR), E - 2);
        gp[6] = double_cvt(ninth64(dg - M8 - JZ + JR), E - 2);
    }
    // not a number, or at rest: both rare, one branch around them
    const bool none = bad || top >= 0x7ff00000;
    if (none || rest) {
        const double v = none ? nan64() : 0.0;
#pragma unroll
        for (int i = 0; i < 9; ++i) gp[i] = v;
        if (none) {
#pragma unroll
            for (int i = 0; i < 9; ++i) fp[i] = v;
            chz_out = chr_out = p_out = v;
        }
    }
}

}  // namespace axilbm
