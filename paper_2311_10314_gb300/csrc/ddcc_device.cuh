// Device code shared by the DD-CCLB kernels (arXiv 2311.10314, Sec. 3).
//
// The per-node update is written once, against two small interfaces so the
// tile kernel and the row-sweep kernel feed it from their own shared-memory
// layouts:
//   accessor  C(j, dy, dx)  C_j (j < N-1) at the neighbour (x+dx, y+dy)
//             psi(dy, dx)   the characteristic function psi
//             mu(j, dy, dx) mu_j (j < N) of Eq. 2.14
//             grad_psi(P, gx, gy)  grad psi at the node
//             psi_rho(dy, dx)  psi rho
//             a(dy, dx)     the lagged antisymmetric-flux field a
//             lag(k)        lagged plane k at the node
//             f(i, p), g(p) pre-collision populations at the node
//   sink      f_out(i, p, v), g_out(p, v)   post-collision populations that
//                                           leave the node in direction p
//             lag_out(k, v)                 lagged plane k of the next step
//             macro(C, rho, ux, uy, P, mu)  read-out mode only
#pragma once

#include "ddcc_internal.h"

namespace ddcc {
namespace dev {

// Periodic wrap, or reflection about the outer wall half a node outside
// the first and last node (mirror ghost nodes).
__device__ __forceinline__ int map_index(int g, int n, int periodic) {
    if (periodic) {
        g %= n;
        return g < 0 ? g + n : g;
    }
    const int n2 = 2 * n;
    int m = g % n2;
    if (m < 0) m += n2;
    return m >= n ? n2 - 1 - m : m;
}

// The image of coordinate v (0 .. n-1) in the one-node ghost ring, as a step
// from v: periodic 0 -> n and n-1 -> -1, mirror 0 -> -1 and n-1 -> n; 0: none
// (n >= 3, so a node has at most one image along an axis).
__device__ __forceinline__ int ring_step(int v, int n, int periodic) {
    if (v == 0) return periodic ? n : -1;
    if (v == n - 1) return periodic ? -n : 1;
    return 0;
}

// g(C) = C^2 (C - 1)^2  =>  g'(C) = 2 C (C - 1) (2 C - 1)  (Sec. 2.1), with
// every factor exact to a rounding near its own root.
template <typename T>
__device__ __forceinline__ T gprime(T c) {
    return c * (c - T(1)) * (T(4) * c - T(2));
}

// Reciprocal and square root of the node update.  FP32: the hardware forms
// the build flags select.  FP64: the update is bound by the FP64 pipe, which
// takes 64 cycles a warp instruction (add, multiply and fused multiply-add
// alike), so both start from the hardware seed, whose relative error is below
// 2^-19.9 (measured by ddcc_selftest_math64, as are the figures below).
//  * rcp: with e = 1 - x r the reciprocal is r (1 + e + e^2 + ...) (geometric
//    series), cut after e^2: 3 FP64 instructions, where a division by the
//    operator took 8.8 (clock64, dependent chain).
//  * root: one of Goldschmidt's coupled steps, g -> sqrt(x) and h -> 1 / (2
//    sqrt(x)) from g = x y, h = y / 2, then the residual correction g + (x -
//    g^2) h: 7 FP64 instructions.
// Over all normal arguments and results rcp differs from the correctly
// rounded quotient by a unit in the last place for 0.2% of the arguments and
// root for none (below 2^-960 by a unit for some).  Zero, infinity and
// not-a-number give what the operators give; a subnormal argument counts as
// zero, and a reciprocal below 2^-1021 has the seed's accuracy or is zero.
// Chosen as integers, without a branch: with the operators behind a branch a
// 64 x 64 step of two phases took 18.8 us instead of 18.2.
__device__ __forceinline__ float rcp(float x) { return 1.0f / x; }
__device__ __forceinline__ double rcp(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    // |x| in [2^-1022, 2^1021); elsewhere the seed is infinite, zero, not a
    // number, or close to the end of the range
    return (unsigned)((__double2hiint(x) & 0x7ff00000) - (1 << 20)) < 2043u << 20 ? fma(r, fma(e, e, e), r) : r;
}
__device__ __forceinline__ float root(float x) { return sqrtf(x); }
__device__ __forceinline__ double root(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double g0 = x * y, h0 = 0.5 * y;
    const double r = fma(-g0, h0, 0.5);
    const double g = fma(g0, r, g0), h = fma(h0, r, h0);
    const double s = fma(fma(-g, g, x), h, g);
    const int hi = __double2hiint(x);
    if (hi == 0x7ff00000) return x;                       // infinity
    return (unsigned)(hi << 1) < 2u << 20 ? 0.0 : s;      // zero and subnormal
}
// x where x > 0, else 0 (not-a-number included), and x with the sign of s,
// without the FP64 pipe
__device__ __forceinline__ float clamp0(float x) { return fmaxf(x, 0.0f); }
__device__ __forceinline__ double clamp0(double x) { return (unsigned)__double2hiint(x) > 0x7ff00000u ? 0.0 : x; }
__device__ __forceinline__ bool positive(float x) { return x > 0.0f; }
__device__ __forceinline__ bool positive(double x) { return __double2hiint(x) > 0; }   // (subnormals count as zero)
__device__ __forceinline__ float signed_as(float x, float s) { return copysignf(x, s); }
__device__ __forceinline__ double signed_as(double x, double s) {
    return __hiloint2double((__double2hiint(s) & 0x80000000) | (__double2hiint(x) & 0x7fffffff),
                            __double2loint(x));
}

// Gradient stencil sum_p w_p c_p chi(x + c_p) / cs2 (isotropic, radius 1).
template <typename T, class A>
__device__ __forceinline__ void grad9(const KParams<T>& P, const A& chi, T& gx, T& gy) {
    // the two diagonals' differences serve both components
    const T ax = chi(0, 1) - chi(0, -1), ay = chi(1, 0) - chi(-1, 0);
    const T d1 = chi(1, 1) - chi(-1, -1), d2 = chi(-1, 1) - chi(1, -1);
    gx = P.gw1 * ax + P.gw2 * (d1 + d2);
    gy = P.gw1 * ay + P.gw2 * (d1 - d2);
}

// mu_i = psi mu_i / psi with psi mu_i of Eq. 2.14: beta_ij = 3 sigma_ij / eps,
// gradient term (3 eps / 4) sigma_ij div(psi grad C_j), wetting term
// 3 sigma_ij sum_{q != j} cos(theta_jq) C_j C_q |grad psi| with cos(theta_jq)
// from the N-1 angles theta_iN by Eq. 2.9 (cth holds cos(theta_iN)).  With
// several solids (Sec. 4.5) cth holds e_j = sum_k cos(theta^k_jN) |grad psi_k|
// and |grad psi| is replaced by 1: Eq. 2.9 is linear in the cosines, so
// sum_k cos(theta^k_jq) |grad psi_k| = (sigma_jN e_j - sigma_qN e_q) / sigma_jq.
// Cx(j, dy, dx) gives C_j for j < NP-1; Ps(dy, dx) gives psi.
//
// All three coefficients are multiples of sigma_ij, so with V_j = (3 eps / 4)
// div(psi grad C_j) + 3 C_j sum_q cos(theta_jq) C_q |grad psi| the sum over j
// is sum_j sigma_ij V_j once.  The pair terms g'(C_i + C_j) use
// g'(1 - c) = -g'(c) and sum_j C_j = 1: they vanish for two phases, are
// -g'(C_k) of the third for three, and for four three pairs give the other
// three.  For two phases mu_2 = -mu_1.
// mu_i of one node from the fractions and V_j = (3 eps / 4) div(psi grad C_j)
// of the N-1 evolved phases; agp3 = 3 |grad psi| (3 with several solids),
// inv_p0 = 1 / psi.  Any lattice: PT holds the model's constants.
template <typename T, int NP, class PT>
__device__ __forceinline__ void mu_of(const PT& P, const T* C, const T* Lk, const T* cth, T agp3, T inv_p0, T mu[NP]) {
    T Cv[NP], V[NP];
    T sumC = C[0], sumL = Lk[0];
#pragma unroll
    for (int j = 0; j < NP - 1; ++j) {
        Cv[j] = C[j];
        V[j] = Lk[j];
        if (j > 0) {
            sumC += C[j];
            sumL += Lk[j];
        }
    }
    Cv[NP - 1] = T(1) - sumC;
    V[NP - 1] = -sumL;
    // a_j = sigma_jN cos(theta_jN) (zero for j = N, sigma_NN = 0), so that
    // cos(theta_jq) = (a_j - a_q) / sigma_jq, antisymmetric in (j, q)
    if constexpr (NP == 2) {
        const T v = V[0] + agp3 * (cth[0] * (Cv[0] * Cv[1]));
        mu[0] = P.beta2[0][1] * gprime(Cv[0]) - P.sig[0][1] * v * inv_p0;
        mu[1] = -mu[0];
    } else {
        T aj[NP], gp[NP];
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            aj[j] = j < NP - 1 ? P.sigN[j] * cth[j] : T(0);
            gp[j] = gprime(Cv[j]);
        }
        T gpair[NP][NP], cpair[NP][NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) {
#pragma unroll
            for (int j = i + 1; j < NP; ++j) {
                if constexpr (NP == 3) {
                    gpair[i][j] = gpair[j][i] = -gp[3 - i - j];
                } else if (i == 0) {
                    const T h = gprime(Cv[0] + Cv[j]);
                    const int k = j == 1 ? 2 : 1, l = j == 3 ? 2 : 3;   // the other two phases
                    gpair[0][j] = gpair[j][0] = h;
                    gpair[k][l] = gpair[l][k] = -h;
                }
                const T c = j < NP - 1 ? (aj[i] - aj[j]) * P.invsig[i][j] : cth[i];
                cpair[i][j] = c;
                cpair[j][i] = -c;
            }
        }
        // V_j += 3 |grad psi| C_j sum_{q != j} cos(theta_jq) C_q
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            T acc = cpair[j][j == 0 ? 1 : 0] * Cv[j == 0 ? 1 : 0];
#pragma unroll
            for (int q = 1; q < NP; ++q)
                if (q != j && !(j == 0 && q == 1)) acc += cpair[j][q] * Cv[q];
            V[j] += agp3 * (Cv[j] * acc);
        }
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            T bulk = P.beta2s[i] * gp[i];
            T v = T(0);
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                if (j == i) continue;
                bulk -= P.beta2[i][j] * gpair[i][j];
                v = (j == 0 || (i == 0 && j == 1)) ? P.sig[i][j] * V[j] : v + P.sig[i][j] * V[j];
            }
            mu[i] = bulk + v * inv_p0;
        }
    }
}

// agp3 = 3 |grad psi| (3 with several solids) and inv_p0 = 1 / psi at the node.
template <typename T, int NP, class CA, class PA>
__device__ __forceinline__ void chem_pot_with(const KParams<T>& P, const CA& Cx, const PA& Ps,
                                              const T* cth, T agp3, T inv_p0, T mu[NP]) {
    const T p0 = Ps(0, 0);
    const T pE = Ps(0, 1), pW = Ps(0, -1), pN = Ps(1, 0), pS = Ps(-1, 0);
    const T pNE = Ps(1, 1), pNW = Ps(1, -1), pSW = Ps(-1, -1), pSE = Ps(-1, 1);
    T Cv[NP - 1], V[NP - 1];
#pragma unroll
    for (int j = 0; j < NP - 1; ++j) {
        const T c0 = Cx(j, 0, 0);
        // (3 eps / 4) div(psi grad C), div = sum_p w_p (psi + psi_p)(C_p - C) / cs2
        const T l = P.lk1 * ((p0 + pE) * (Cx(j, 0, 1) - c0) + (p0 + pW) * (Cx(j, 0, -1) - c0) +
                             (p0 + pN) * (Cx(j, 1, 0) - c0) + (p0 + pS) * (Cx(j, -1, 0) - c0)) +
                    P.lk2 * ((p0 + pNE) * (Cx(j, 1, 1) - c0) + (p0 + pNW) * (Cx(j, 1, -1) - c0) +
                             (p0 + pSW) * (Cx(j, -1, -1) - c0) + (p0 + pSE) * (Cx(j, -1, 1) - c0));
        Cv[j] = c0;
        V[j] = l;
    }
    mu_of<T, NP>(P, Cv, V, cth, agp3, inv_p0, mu);
}

template <typename T, int NP, class CA, class PA>
__device__ __forceinline__ void chem_pot(const KParams<T>& P, const CA& Cx, const PA& Ps,
                                         const T* cth, T mu[NP]) {
    T gpx, gpy;
    grad9(P, [&](int dy, int dx) { return Ps(dy, dx); }, gpx, gpy);
    // with several solids the angle planes already carry |grad psi_k|
    const T agp3 = T(3) * (P.wet_field ? T(1) : root(gpx * gpx + gpy * gpy));
    chem_pot_with<T, NP>(P, Cx, Ps, cth, agp3, rcp(Ps(0, 0)), mu);
}

// Hermite moments m_ab = sum_p v_p h_a(cx_p) h_b(cy_p), h = (1, c, c^2 - cs2),
// in the order (00, 10, 01, 20, 02, 11, 21, 12, 22).
// Returns the sum of the moving populations, m_00 - v_0.
template <typename T>
__device__ __forceinline__ T hermite_moments(const T v[9], T cs2, T m[9]) {
    // pass over cx in each row cy = -1, 0, +1 (populations (cx, cy)):
    //   A0 = sum, A1 = v(+1) - v(-1), A2 = v(+1) + v(-1) - cs2 A0
    const T sm0 = v[7] + v[8], sz0 = v[3] + v[1], sp0 = v[6] + v[5];
    const T A0m = sm0 + v[4], A0z = sz0 + v[0], A0p = sp0 + v[2];
    const T A1m = v[8] - v[7], A1z = v[1] - v[3], A1p = v[5] - v[6];
    const T A2m = sm0 - cs2 * A0m, A2z = sz0 - cs2 * A0z, A2p = sp0 - cs2 * A0p;
    // pass over cy with h_b(cy)
    const T moving = (A0m + sz0) + A0p;
    m[0] = moving + v[0];
    m[2] = A0p - A0m;
    m[4] = (A0p + A0m) - cs2 * m[0];
    m[1] = A1m + A1z + A1p;
    m[5] = A1p - A1m;
    m[7] = (A1p + A1m) - cs2 * m[1];
    m[3] = A2m + A2z + A2p;
    m[6] = A2p - A2m;
    m[8] = (A2p + A2m) - cs2 * m[3];
    return moving;
}

// Rounded to nearest and never fused or reassociated by the compiler.
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// B_p = sum_ab h_a(cx_p) h_b(cy_p) k_ab; out_p = v_p - w_p B_p.
// kConserve (the phase populations, which carry the conserved psi C, and
// whose k_00 is zero): the rest population holds nearly all of psi C, so
// v_0 - w_0 B_0 rounds at the ulp of psi C, and in a steady flow the same
// rounding repeats every step and drifts the phase mass.  Then w_0 B_0 and
// the subtraction are rounded explicitly, the exact error of the
// subtraction is recovered (TwoSum) and split evenly (halving is exact)
// between out_1 and out_3, the +x and -x populations, far smaller in
// magnitude: sum_p out_p keeps the exchange up to roundings at that smaller
// scale, and the recovered mass leaves the node in no preferred direction
// (a steady error put on one direction would carry phase mass along it
// every step).
template <typename T, bool kConserve = false>
__device__ __forceinline__ void hermite_relax_back(const T k[9], const KParams<T>& P, const T v[9], T out[9]) {
    const T cs2 = P.cs2, one_m = P.one_m_cs2;
    // R_a(cy) = k_a0 + cy k_a1 + (cy^2 - cs2) k_a2 for a = 0, 1, 2
    const T ka0[3] = {k[0], k[1], k[3]};
    const T ka1[3] = {k[2], k[5], k[6]};
    const T ka2[3] = {k[4], k[7], k[8]};
    T Rm[3], R0[3], Rp[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        T base;
        if (kConserve && a == 0) {
            base = one_m * ka2[0];
            R0[0] = -cs2 * ka2[0];
        } else {
            base = ka0[a] + one_m * ka2[a];
            R0[a] = ka0[a] - cs2 * ka2[a];
        }
        Rp[a] = base + ka1[a];
        Rm[a] = base - ka1[a];
    }
    // B(cx, cy) = R_0 + cx R_1 + (cx^2 - cs2) R_2; even parts once per row
    const T E0 = R0[0] + one_m * R0[2], Ep = Rp[0] + one_m * Rp[2], Em = Rm[0] + one_m * Rm[2];
    const T* w = kConserve ? P.wf : P.w9;
    const T w0 = w[0], wa = w[1], wd = w[2];
    out[1] = v[1] - wa * (E0 + R0[1]);
    out[3] = v[3] - wa * (E0 - R0[1]);
    if constexpr (kConserve) {
        const T t0 = mul_rn(w0, R0[0] - cs2 * R0[2]);
        const T o0 = add_rn(v[0], -t0);
        const T bb = add_rn(o0, -v[0]);                 // TwoSum(v_0, -t_0)
        const T err = add_rn(add_rn(v[0], -add_rn(o0, -bb)), add_rn(-t0, -bb));
        out[0] = o0;
        const T half = T(0.5) * err;
        out[1] = add_rn(out[1], half);
        out[3] = add_rn(out[3], half);
    } else {
        out[0] = v[0] - w0 * (R0[0] - cs2 * R0[2]);
    }
    out[2] = v[2] - wa * (Rp[0] - cs2 * Rp[2]);
    out[4] = v[4] - wa * (Rm[0] - cs2 * Rm[2]);
    out[5] = v[5] - wd * (Ep + Rp[1]);
    out[6] = v[6] - wd * (Ep - Rp[1]);
    out[7] = v[7] - wd * (Em - Rm[1]);
    out[8] = v[8] - wd * (Em + Rm[1]);
}

// The phase collision where one rate s holds for every moment of second and
// higher order (the paper's own choice, Secs. 4.1-4.4).  The rows are complete
// (sum_ab w_p h_ab(c_p) m_ab / N_ab = v_p), so relaxing all of them by s is
// (1 - s) v_p, and only the conserved and the first-order rows are put
// right; f^eq less its first order is w_p emu + X delta_p0, emu = eta psi mu,
// X = psi C - emu:
//   out_p = (1 - s) v_p + w_p (s emu + c_p . q) + s X delta_p0,
//   q = s j / cs2 - k_1,  k_1 = lambda_1 (j - psi C u) + cV V.
// What the rest population gives, t_0 = v_0 - out_0 = s (1 - w_0) emu - s m,
// is formed from the sum m of the moving populations: with psi C in its
// place the node's mass would change by s times the rounding of that sum
// (5e-17 rms at psi C = 1; so it is of the order of m's rounding, 2e-20 at
// moving populations of 1e-3).  Its rounding error is treated as in
// hermite_relax_back.  28 FP64 instructions a phase less than the transforms
// (FP64 only: FP32 is bound by memory).
template <typename T>
__device__ __forceinline__ void relax_one_rate(const KParams<T>& P, int i, const T v[9], T jx, T jy, T moving, T emu,
                                               T pcux, T pcuy, T Vx, T Vy, T out[9]) {
    const T lam = P.lamf[i][1];
    const T qx = P.qf[i] * jx + lam * pcux - P.cV[i] * Vx;
    const T qy = P.qf[i] * jy + lam * pcuy - P.cV[i] * Vy;
    const T se = P.sf * emu;
    const T a = P.wf[1] * se, ax = P.wf[1] * qx, ay = P.wf[1] * qy;
    const T d = P.wf[2] * se, dp = P.wf[2] * (qx + qy), dm = P.wf[2] * (qx - qy);
    const T k = P.one_m_sf;
    const T t0 = P.cse * emu - P.sf * moving;
    const T o0 = add_rn(v[0], -t0);
    const T bb = add_rn(o0, -v[0]);                 // TwoSum(v_0, -t_0)
    const T half = T(0.5) * add_rn(add_rn(v[0], -add_rn(o0, -bb)), add_rn(-t0, -bb));
    out[0] = o0;
    out[1] = add_rn(k * v[1] + (a + ax), half);
    out[3] = add_rn(k * v[3] + (a - ax), half);
    out[2] = k * v[2] + (a + ay);
    out[4] = k * v[4] + (a - ay);
    out[5] = k * v[5] + (d + dp);
    out[7] = k * v[7] + (d - dp);
    out[8] = k * v[8] + (d + dm);
    out[6] = k * v[6] + (d - dm);
}

// psi rho at a node, rho = rho_N + sum_j (rho_j - rho_N) C_j
template <typename T, int NP, class CA>
__device__ __forceinline__ T psi_rho(const KParams<T>& P, T psi, const CA& C) {
    T r = P.rho[NP - 1];
#pragma unroll
    for (int j = 0; j < NP - 1; ++j) r += P.drho[j] * C(j);
    return psi * r;
}

// One node of the step: order parameters and gradients (a1, a2), mobility
// flux and m^C (a4), force, the joint velocity / Eq. 19 pressure solve
// (a5, a6), then (MODE 0) both collisions in Hermite moment space (a7, a8)
// and the lagged fields (a10), or (MODE 1) the macroscopic read-out.
//
// sum_j C_j = 1 throughout (C_N is defined by it), so sums over all phases
// reduce to the N-1 evolved ones: rho and grad rho through rho_j - rho_N,
// the capillary force through mu_j - mu_N, and m^C = -m0 sum_j
// (rho_j - rho_N) Q_j because the Q_j add up to zero.  With the pair
// identities of chem_pot, psi rho formed once per node and the reciprocals
// above this is a fifth of the FP64 instructions less than sums over all
// phases, which is what FP64 is bound by; in FP32, bound by memory, it leaves
// the time as it is.
// kOneRate: the phase collision by relax_one_rate.
template <typename T, int NP, int MODE, bool kOneRate = false, class Acc, class Sink>
__device__ __forceinline__ void node_update(const KParams<T>& P, const Acc& A, Sink& out) {
    const T cs2 = P.cs2;
    const T psi = A.psi(0, 0);

    // ---- order parameters and their gradients -----------------------------
    T Cv[NP], gCx[NP - 1], gCy[NP - 1];
    T rho = P.rho[NP - 1], nu = P.nu[NP - 1], grx = T(0), gry = T(0);
    {
        T sC = T(0);
#pragma unroll
        for (int j = 0; j < NP - 1; ++j) {
            Cv[j] = A.C(j, 0, 0);
            grad9(P, [&](int dy, int dx) { return A.C(j, dy, dx); }, gCx[j], gCy[j]);
            sC = j == 0 ? Cv[0] : sC + Cv[j];
            rho += P.drho[j] * Cv[j];
            nu += P.dnu[j] * Cv[j];
            grx = j == 0 ? P.drho[0] * gCx[0] : grx + P.drho[j] * gCx[j];
            gry = j == 0 ? P.drho[0] * gCy[0] : gry + P.drho[j] * gCy[j];
        }
        Cv[NP - 1] = T(1) - sC;
    }
    // s21 and s22 from nu by Eq. 16
    const T inv_s21 = nu * P.nu_to_s21 + T(0.5);
    const T s21 = rcp(inv_s21);
    const T s22 = rcp(nu * P.nu_to_s22 + T(0.5));
    T gpx, gpy;
    A.grad_psi(P, gpx, gpy);
    T gprx, gpry;
    grad9(P, [&](int dy, int dx) { return A.psi_rho(dy, dx); }, gprx, gpry);

    // ---- chemical potentials, mobility flux, m^C --------------------------
    T mu[NP], gmx[NP], gmy[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        if (NP == 2 && j == 1) {
            mu[1] = -mu[0];
            gmx[1] = -gmx[0];
            gmy[1] = -gmy[0];
        } else {
            mu[j] = A.mu(j, 0, 0);
            grad9(P, [&](int dy, int dx) { return A.mu(j, dy, dx); }, gmx[j], gmy[j]);
        }
    }
    // Q_i = sum_j M_ij grad mu_j / m0 = C_i (grad mu_i - sum_j C_j grad mu_j)
    T Gx, Gy;
    if constexpr (NP == 2) {
        const T dC = Cv[0] - Cv[1];
        Gx = dC * gmx[0];
        Gy = dC * gmy[0];
    } else {
        Gx = Cv[0] * gmx[0];
        Gy = Cv[0] * gmy[0];
#pragma unroll
        for (int j = 1; j < NP; ++j) {
            Gx += Cv[j] * gmx[j];
            Gy += Cv[j] * gmy[j];
        }
    }
    T Qx[NP - 1], Qy[NP - 1];
    T mCx = T(0), mCy = T(0);   // psi m^C
#pragma unroll
    for (int i = 0; i < NP - 1; ++i) {
        Qx[i] = Cv[i] * (gmx[i] - Gx);
        Qy[i] = Cv[i] * (gmy[i] - Gy);
        mCx = i == 0 ? P.drho[0] * Qx[0] : mCx + P.drho[i] * Qx[i];
        mCy = i == 0 ? P.drho[0] * Qy[0] : mCy + P.drho[i] * Qy[i];
    }
    const T pm0 = -(P.m0 * psi);
    mCx *= pm0;
    mCy *= pm0;

    // ---- lagged fields of the previous step --------------------------------
    T dax, day;
    grad9(P, [&](int dy, int dx) { return A.a(dy, dx); }, dax, day);
    const T psimu_prev = A.lag(2 * NP + 2);

    // ---- flow populations, velocity and pressure ---------------------------
    T g[9], mg[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) g[p] = A.g(p);
    const T sum_g = hermite_moments(g, cs2, mg);
    const T Jx = mg[1], Jy = mg[2];
    T sx = rho * P.body[0], sy = rho * P.body[1];
#pragma unroll
    for (int j = 0; j < NP - 1; ++j) {
        const T dm = NP == 2 ? mu[0] + mu[0] : mu[j] - mu[NP - 1];
        sx += dm * gCx[j];
        sy += dm * gCy[j];
    }
    const T F0x = psi * sx + day;
    const T F0y = psi * sy - dax;
    const T psirho = psi * rho;
    const T dmp = P.damp - P.damp * psi;
    const T inv_den = rcp(psirho + T(0.5) * dmp);
    const T u0x = (Jx + T(0.5) * F0x) * inv_den;
    const T u0y = (Jy + T(0.5) * F0y) * inv_den;
    const T hi = T(0.5) * inv_den;
    const T ex = gpx * hi;
    const T ey = gpy * hi;
    const T Hs = P.Hfac - T(2) * P.Hfac * inv_s21;    // H / s21 = Hfac (s21 - 2) / s21
    const T Ap = P.A_P * psi;
    const T bx = Ap * grx + P.gam * mCx + Hs * gprx;
    const T by = Ap * gry + P.gam * mCy + Hs * gpry;
    const T gq = P.gam * psirho;
    const T G0 = sum_g - P.Kh * psimu_prev;
    // Eq. 19 with u = u0 + P e: cP (gq e.e) P^2 + (cP (b + 2 gq u0).e - psi) P
    // + cP (G0 + (b + gq u0).u0) = 0
    const T vx = bx + gq * u0x, vy = by + gq * u0y;
    const T wx = vx + gq * u0x, wy = vy + gq * u0y;
    const T qa = P.cP * gq * (ex * ex + ey * ey);
    const T qb = P.cP * (wx * ex + wy * ey) - psi;
    const T qc = P.cP * (G0 + vx * u0x + vy * u0y);
    const T disc = clamp0(qb * qb - T(4) * qa * qc);
    const T Pr = T(-2) * qc * rcp(qb + signed_as(root(disc), qb));
    const T ux = u0x + Pr * ex;
    const T uy = u0y + Pr * ey;

    if (MODE == 1) {
        out.macro(Cv, rho, ux, uy, Pr, mu);
        return;
    }
    const T Fx = F0x + Pr * gpx - dmp * ux;
    const T Fy = F0y + Pr * gpy - dmp * uy;

    // ---- phase LB, Eqs. 3.1, 3.5-3.7 ---------------------------------------
#pragma unroll
    for (int i = 0; i < NP - 1; ++i) {
        T v[9], m[9], k[9], o9[9], moving;
#pragma unroll
        for (int p = 0; p < 9; ++p) v[p] = A.f(i, p);
        if constexpr (kOneRate) {
            const T d1 = v[5] - v[7], d2 = v[8] - v[6];
            m[1] = (v[1] - v[3]) + (d1 + d2);
            m[2] = (v[2] - v[4]) + (d1 - d2);
            // in the order of hermite_moments
            moving = ((v[7] + v[8]) + v[4]) + (v[3] + v[1]) + ((v[6] + v[5]) + v[2]);
            m[0] = moving + v[0];
        } else {
            moving = hermite_moments(v, cs2, m);
        }
        const T psiC = m[0];
        const T pcux = psiC * ux, pcuy = psiC * uy;
        // V = d_t(psi C u) + cs2 eta (mu grad psi - S), S = psi (Q - grad mu)
        const T Vx = (pcux - A.lag(1 + 2 * i)) + P.ceta[i] * (mu[i] * gpx + psi * (gmx[i] - Qx[i]));
        const T Vy = (pcuy - A.lag(2 + 2 * i)) + P.ceta[i] * (mu[i] * gpy + psi * (gmy[i] - Qy[i]));
        if constexpr (kOneRate) {
            const T emu = P.eta[i] * (psi * mu[i]);
            relax_one_rate(P, i, v, m[1], m[2], moving, emu, pcux, pcuy, Vx, Vy, o9);
        } else {
            const T X = psiC - P.eta[i] * psi * mu[i];
            const T* lam = P.lamf[i];
            k[0] = T(0);
            k[1] = lam[1] * (m[1] - pcux) + P.cV[i] * Vx;
            k[2] = lam[2] * (m[2] - pcuy) + P.cV[i] * Vy;
            k[3] = lam[3] * (m[3] + cs2 * X);
            k[4] = lam[4] * (m[4] + cs2 * X);
            k[5] = lam[5] * m[5];
            k[6] = lam[6] * m[6];
            k[7] = lam[7] * m[7];
            k[8] = lam[8] * (m[8] - P.cs4 * X);
            hermite_relax_back<T, true>(k, P, v, o9);
        }
#pragma unroll
        for (int p = 0; p < 9; ++p) out.f_out(i, p, o9[p]);
        out.lag_out(1 + 2 * i, pcux);
        out.lag_out(2 + 2 * i, pcuy);
    }

    // ---- flow LB, Eqs. 3.2, 3.8, 3.10 --------------------------------------
    {
        T k[9], o9[9];
        const T psiP = psi * Pr;
        const T jx = psirho * ux, jy = psirho * uy;
        // T = psi (m^C u + u m^C) / 2, a = psi (m^C_x u_y - u_x m^C_y) / 2
        const T p1 = mCx * uy, p2 = ux * mCy;
        const T Txx = mCx * ux;
        const T Tyy = mCy * uy;
        const T Txy = T(0.5) * (p1 + p2);
        const T Axx = jx * ux + Txx;
        const T Ayy = jy * uy + Tyy;
        const T Axy = jx * uy + Txy;
        const T s1 = ux * gprx, s2 = uy * gpry;
        const T cu = P.c2m3cs2 * (s1 + s2);
        const T Mxx = (Txx - A.lag(2 * NP - 1)) + P.two_cs2 * s1 + cu;
        const T Myy = (Tyy - A.lag(2 * NP)) + P.two_cs2 * s2 + cu;
        const T Mxy = (Txy - A.lag(2 * NP + 1)) + cs2 * (ux * gpry + gprx * uy);
        const T a0 = psi * (ux * grx + uy * gry);
        const T l20 = s21 * P.invN20, l11 = s22 * P.invN11;
        const T c20 = T(0.5) * l20 - P.invN20, c11 = T(0.5) * l11 - P.invN11;
        k[0] = P.lg00 * mg[0] + P.cg0 * a0;
        k[1] = P.lg1 * (mg[1] - jx) + P.cg1 * Fx;
        k[2] = P.lg1 * (mg[2] - jy) + P.cg1 * Fy;
        k[3] = l20 * (mg[3] - (psiP + Axx)) + c20 * Mxx;
        k[4] = l20 * (mg[4] - (psiP + Ayy)) + c20 * Myy;
        k[5] = l11 * (mg[5] - Axy) + c11 * Mxy;
        k[6] = P.lg3 * mg[6];
        k[7] = P.lg3 * mg[7];
        k[8] = P.lg4 * (mg[8] + cs2 * psiP);
        hermite_relax_back(k, P, g, o9);
#pragma unroll
        for (int p = 0; p < 9; ++p) out.g_out(p, o9[p]);
        out.lag_out(0, T(0.5) * (p1 - p2));
        out.lag_out(2 * NP - 1, Txx);
        out.lag_out(2 * NP, Tyy);
        out.lag_out(2 * NP + 1, Txy);
        out.lag_out(2 * NP + 2, Axx + Ayy);
    }
}

}  // namespace dev
}  // namespace ddcc
