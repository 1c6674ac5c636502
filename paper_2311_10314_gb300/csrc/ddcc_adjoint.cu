// Discrete adjoint (reverse mode) of one DD-CCLB step and of the initial
// state (arXiv 2311.10314, Sec. 3): the transpose of the Jacobian of exactly
// the arithmetic the forward kernels perform, applied to an adjoint state.
//
// One reverse step n+1 -> n runs these kernels, each over every node (one
// thread per node; the ghost frames hold periodic or mirror copies exactly
// as in the forward step):
//   k_adj_fields             recompute C_i and mu_i of step n from the
//                            checkpointed state, on the domain and its
//                            1-node ghost ring
//   k_adj_node               the node update's VJP: adjoints of the node's
//                            own populations and lagged planes, and of every
//                            stencil output the update reads (grad C_j,
//                            grad psi, grad(psi rho), grad mu_j, grad a and
//                            the centre values); the streaming is transposed
//                            by pulling the adjoint from each push target
//   k_adj_gather3            transposed gradient stencils: adjoints of C_j,
//                            psi, mu_j and a at each node, followed in the
//                            same thread by the VJP of Eq. 2.14 per node
//                            (mu_node_at): adjoints of the centre C_j and
//                            psi, of div(psi grad C_j) and grad psi, and
//                            dJ/dcos(theta_iN) at the node
//   k_adj_gather2            transposed div(psi grad .) and grad psi stencils,
//                            then C_i = sum_p f^i_p / psi reversed, and
//                            dJ/dpsi
// A ghost-ring node copies a node of the domain, so what a transposed
// stencil leaves there belongs to the copied node.  Both gathers take that
// in through their shared-memory rings (load_ring): the sources beyond the
// edge are the wrapped or mirrored ones, with the sign of a vector's
// component across the wall reversed.
// The initial state (f = f^eq(psi C0, psi mu(C0), u = 0), g and the lagged
// planes zero) is reversed by k_adj_init_node followed by the same mu stage
// as a kernel of its own (k_adj_mu_node).
#include "ddcc_device.cuh"

namespace ddcc {
namespace {

using dev::map_index;
using dev::ring_step;

constexpr int AX = 32;   // threads (and nodes) along x of every kernel here
// Rows of a block.  FP64 is bound by FP64 warp instructions per SM
// sub-partition: blocks of two warps spread a small grid over every SM and
// leave shorter last waves (130 x 94, N = 3: as 32 x 8 blocks the grid was 60
// blocks on 60 of 152 SMs; with the shorter arithmetic 24 steps of the whole
// gradient went from 8.8 to 4.5 ms).  FP32 keeps eight rows, for the smaller share of
// ring nodes per node.
template <typename T>
__host__ __device__ constexpr int block_rows() { return sizeof(T) == 8 ? 2 : 8; }
// Whether a kernel of the reverse step lets the next one start early.
template <typename T>
__host__ __device__ constexpr bool overlaps() { return sizeof(T) == 4; }
// First node of the block.  FP64 counts the rows of blocks along grid x (grid
// y ends at 65535 blocks, short of the tallest grids in rows of two).
template <typename T>
__device__ __forceinline__ int first_x() { return (int)(sizeof(T) == 8 ? blockIdx.y : blockIdx.x) * AX; }
template <typename T>
__device__ __forceinline__ int first_y() { return (int)(sizeof(T) == 8 ? blockIdx.x : blockIdx.y) * block_rows<T>(); }
constexpr double kKinkGradPsi = 1e-6;

// D2Q9 velocities (Sec. 3): 0 rest, 1-4 axis, 5-8 diagonal.
__constant__ int aCx[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
__constant__ int aCy[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};

__device__ __forceinline__ int opp(int p) { return p == 0 ? 0 : (p <= 4 ? ((p + 1) & 3) + 1 : ((p - 3) & 3) + 5); }

// B_p = sum_ab h_a(cx_p) h_b(cy_p) k_ab (the transpose of hermite_moments).
template <typename T>
__device__ __forceinline__ void hermite_B(const T k[9], T cs2, T B[9]) {
    const T ka0[3] = {k[0], k[1], k[3]};
    const T ka1[3] = {k[2], k[5], k[6]};
    const T ka2[3] = {k[4], k[7], k[8]};
    T Rm[3], R0[3], Rp[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const T base = ka0[a] + (T(1) - cs2) * ka2[a];
        R0[a] = ka0[a] - cs2 * ka2[a];
        Rp[a] = base + ka1[a];
        Rm[a] = base - ka1[a];
    }
    const T one_m = T(1) - cs2;
    B[0] = R0[0] - cs2 * R0[2];
    B[1] = R0[0] + R0[1] + one_m * R0[2];
    B[2] = Rp[0] - cs2 * Rp[2];
    B[3] = R0[0] - R0[1] + one_m * R0[2];
    B[4] = Rm[0] - cs2 * Rm[2];
    B[5] = Rp[0] + Rp[1] + one_m * Rp[2];
    B[6] = Rp[0] - Rp[1] + one_m * Rp[2];
    B[7] = Rm[0] - Rm[1] + one_m * Rm[2];
    B[8] = Rm[0] + Rm[1] + one_m * Rm[2];
}

// g''(C) for g(C) = C^2 (C - 1)^2.
template <typename T>
__device__ __forceinline__ T gsecond(T c) {
    return T(12) * c * c - T(12) * c + T(2);
}

template <typename T>
__device__ __forceinline__ T wgt(const KParams<T>& P, int p) {
    return P.w1d[aCx[p] + 1] * P.w1d[aCy[p] + 1];
}

// ---------------------------------------------------------------------------
// recompute C_i and mu_i of step n
// ---------------------------------------------------------------------------

template <typename T>
struct PlaneAt {
    const T* base;
    long long plane, o;
    int pitch;
    __device__ T operator()(int j, int dy, int dx) const { return base[j * plane + o + (long long)dy * pitch + dx]; }
    __device__ T operator()(int dy, int dx) const { return base[o + (long long)dy * pitch + dx]; }
};

template <typename T, int NP>
__device__ __forceinline__ void node_cth(const KParams<T>& P, const T* cosf, long long o, T cth[NP]) {
#pragma unroll
    for (int i = 0; i < NP - 1; ++i) cth[i] = P.has_cos_field ? cosf[i * P.plane + o] : P.cos_uni[i];
    cth[NP - 1] = T(0);
}

// ---------------------------------------------------------------------------
// scratch planes (each a padded plane of T)
// ---------------------------------------------------------------------------

// Chemical-potential planes kept: for two phases mu_2 = -mu_1, so one, whose
// adjoint takes the second's with its sign reversed.
template <int NP>
__host__ __device__ constexpr int mu_planes() { return NP == 2 ? 1 : NP; }

template <typename T, int NP>
struct AdjPlanes {
    static constexpr int NM = mu_planes<NP>();
    static constexpr int NV = 2 * (NP + 2 + NM);   // planes of the gather3 ring
    T* C;     // N-1   C_i of step n
    T* mu;    // NM    mu_i of step n
    T* chi;   // 1     (FP64) psi rho of step n
    T* lC;    // N-1   node VJP: centre C_j
    T* lgC;   // 2(N-1)          grad C_j (x, y)
    T* lpsi;  // 1               centre psi
    T* lgp;   // 2               grad psi
    T* lgpr;  // 2               grad(psi rho)
    T* lmu;   // NM              centre mu_j
    T* lgm;   // 2 NM            grad mu_j
    T* lga;   // 2               grad a
    T* LC;    // N-1   gathered adjoint of C_j
    T* Lpsi;  // 1                         psi
    T* Lmu;   // NM                        mu_j (the initial state's reverse only)
    T* mC;    // N-1   mu VJP: centre C_j
    T* mL;    // N-1           (3 eps / 4) div(psi grad C_j)
    T* mpsi;  // 1             centre psi
    T* mgp;   // 2             grad psi
    const T* a;   // lagged plane a of step n (the state's own plane, ghost ring filled)
    __host__ static AdjPlanes carve(T* base, long long plane) {
        AdjPlanes A;
        T* q = base;
        auto take = [&](int n) { T* r = q; q += (long long)n * plane; return r; };
        A.C = take(NP - 1);   // first: adjoint_c_planes
        A.mu = take(NM);
        A.chi = take(sizeof(T) == 8 ? 1 : 0);
        A.lC = take(NP - 1);
        A.lpsi = take(1);
        A.lmu = take(NM);
        // the vector pairs the first gather reads, consecutive
        A.lgC = take(2 * (NP - 1));
        A.lgp = take(2);
        A.lgpr = take(2);
        A.lgm = take(2 * NM);
        A.lga = take(2);
        A.LC = take(NP - 1);
        A.Lpsi = take(1);
        A.Lmu = take(NM);
        A.mC = take(NP - 1);
        A.mpsi = take(1);
        A.mL = take(NP - 1);
        A.mgp = take(2);
        A.a = nullptr;
        return A;
    }
    // 7 (N-1) + 5 NM + 11 planes
    __host__ __device__ static constexpr int planes() { return 7 * (NP - 1) + 5 * NM + 11 + (sizeof(T) == 8 ? 1 : 0); }
};

// Coordinate v in [-1, n] of the ring taken into the domain (values of v
// beyond, in the unused part of a block, land anywhere inside).
__device__ __forceinline__ int ring_index(int v, int n, int periodic) {
    if (v < 0) v = periodic ? v + n : -1 - v;
    else if (v >= n) v = periodic ? v - n : 2 * n - 1 - v;
    return min(max(v, 0), n - 1);
}

// C and mu of one state in one launch: C on the block's nodes and one node
// around them in shared memory, mu on the nodes, both written to the node and
// to its copies in the ghost ring.  From the populations, or (kC0) from the
// C planes themselves, as the initial state's reverse has them.
template <typename T, int NP, bool kC0>
__global__ void __launch_bounds__(AX * block_rows<T>()) k_adj_fields(KParams<T> P, const T* f,
                                                                     const T* __restrict__ psi,
                                                                     const T* __restrict__ cosf, T* C,
                                                                     T* __restrict__ mu, T* __restrict__ chi) {
    constexpr int AY = block_rows<T>(), NT = AX * AY, W = AX + 2, H = AY + 2;
    __shared__ T sC[NP - 1][H][W], sP[H][W];
    if constexpr (overlaps<T>()) wait_for_previous();
    const int x0 = first_x<T>(), y0 = first_y<T>();
    const int tid = threadIdx.y * AX + threadIdx.x;
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    const long long pl = P.plane;
    const long long sx = ring_step(x, P.nx, P.px), sy = (long long)ring_step(y, P.ny, P.py) * P.pitch;
    auto put = [&](T* base, long long o, T v) {
        base[o] = v;
        if (sx) base[o + sx] = v;
        if (sy) base[o + sy] = v;
        if (sx && sy) base[o + sx + sy] = v;
    };
    // all the loads of a thread before the first use of one, so that they are
    // in flight together (beyond the last ring node they repeat it)
    constexpr int R = (H * W + NT - 1) / NT, NF = kC0 ? NP - 1 : 9 * (NP - 1);
    T ps[R], v[R][NF];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int k = min(tid + r * NT, H * W - 1), ly = k / W, lx = k - ly * W;
        const long long o = P.org + (long long)ring_index(y0 + ly - 1, P.ny, P.py) * P.pitch +
                            ring_index(x0 + lx - 1, P.nx, P.px);
        ps[r] = psi[o];
#pragma unroll
        for (int q = 0; q < NF; ++q) v[r][q] = kC0 ? C[q * pl + o] : f[q * pl + o];
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int k = min(tid + r * NT, H * W - 1), ly = k / W, lx = k - ly * W;
        sP[ly][lx] = ps[r];
        const T inv = kC0 ? T(1) : dev::rcp(ps[r]);
#pragma unroll
        for (int i = 0; i < NP - 1; ++i) {
            if constexpr (kC0) {
                sC[i][ly][lx] = v[r][i];
            } else {
                T s = v[r][9 * i];
#pragma unroll
                for (int p = 1; p < 9; ++p) s += v[r][9 * i + p];
                sC[i][ly][lx] = s * inv;
            }
        }
    }
    __syncthreads();
    if constexpr (overlaps<T>()) dependents_may_start();
    if (x >= P.nx || y >= P.ny) return;
    const int ly = threadIdx.y + 1, lx = threadIdx.x + 1;
    const long long o = P.org + (long long)y * P.pitch + x;
    T cth[NP], m[NP];
    node_cth<T, NP>(P, cosf, o, cth);
    dev::chem_pot<T, NP>(P, [&](int j, int dy, int dx) { return sC[j][ly + dy][lx + dx]; },
                         [&](int dy, int dx) { return sP[ly + dy][lx + dx]; }, cth, m);
    if (!kC0) {
#pragma unroll
        for (int i = 0; i < NP - 1; ++i) put(C + i * pl, o, sC[i][ly][lx]);
    }
#pragma unroll
    for (int i = 0; i < mu_planes<NP>(); ++i) put(mu + i * pl, o, m[i]);
    if (sizeof(T) == 8 && !kC0)
        put(chi, o, dev::psi_rho<T, NP>(P, sP[ly][lx], [&](int j) { return sC[j][ly][lx]; }));
}

// ---------------------------------------------------------------------------
// VJP of the node update (a1-a10 at one node)
// ---------------------------------------------------------------------------
// The transpose of dev::node_update in the same variables (mC holds psi m^C,
// s the capillary and body force over psi, v = b + gq u0, w = v + gq u0).
// The pressure's derivative is that of the root of qa P^2 + qb P + qc = 0.
// Bound: FP64 by its pipe, FP32 by latency at two blocks of 128 registers per
// SM.  (With the update's older form, in sums over all N phases, the FP32
// kernel spilled 168 bytes a thread at N = 4 and 60 at N = 3; now 112 and 4.)

template <typename T, int NP>
__global__ void __launch_bounds__(AX * block_rows<T>(), sizeof(T) == 4 ? 2 : 4)
    k_adj_node(KParams<T> P, const T* __restrict__ psi_pl, const T* st_pop,
               const T* st_lag, const T* ad_pop_in, const T* ad_lag_in,
               T* __restrict__ ad_pop_out, T* __restrict__ ad_lag_out, AdjPlanes<T, NP> W) {
    constexpr int M = NP - 1, NM = mu_planes<NP>();
    if constexpr (overlaps<T>()) {
        wait_for_previous();
        dependents_may_start();
    }
    const int x = first_x<T>() + threadIdx.x, y = first_y<T>() + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    const long long pl = P.plane;
    const long long o = P.org + (long long)y * P.pitch + x;
    const PlaneAt<T> Ca{W.C, pl, o, P.pitch}, Pa{psi_pl, pl, o, P.pitch}, Ma{W.mu, pl, o, P.pitch},
        Aa{W.a, pl, o, P.pitch};
    auto grad = [&](auto chi, T& gx, T& gy) { dev::grad9(P, chi, gx, gy); };
    const T cs2 = P.cs2;
    const T* st_g = st_pop + (long long)9 * M * pl;

    // ---- forward recomputation (the arithmetic of dev::node_update) -------
    const T psi = Pa(0, 0);
    T Cv[NP], gCx[M], gCy[M];
    T rho = P.rho[M], nu = P.nu[M], grx = T(0), gry = T(0);
    {
        T sC = T(0);
#pragma unroll
        for (int j = 0; j < M; ++j) {
            Cv[j] = Ca(j, 0, 0);
            grad([&](int dy, int dx) { return Ca(j, dy, dx); }, gCx[j], gCy[j]);
            sC += Cv[j];
            rho += P.drho[j] * Cv[j];
            nu += P.dnu[j] * Cv[j];
            grx += P.drho[j] * gCx[j];
            gry += P.drho[j] * gCy[j];
        }
        Cv[M] = T(1) - sC;
    }
    const T inv_s21 = nu * P.nu_to_s21 + T(0.5);
    const T s21 = dev::rcp(inv_s21);
    const T s22 = dev::rcp(nu * P.nu_to_s22 + T(0.5));
    T gpx, gpy;
    grad([&](int dy, int dx) { return Pa(dy, dx); }, gpx, gpy);
    T gprx, gpry;
    if constexpr (sizeof(T) == 8) {
        const PlaneAt<T> Xa{W.chi, pl, o, P.pitch};
        grad([&](int dy, int dx) { return Xa(dy, dx); }, gprx, gpry);
    } else {
        grad([&](int dy, int dx) { return dev::psi_rho<T, NP>(P, Pa(dy, dx), [&](int j) { return Ca(j, dy, dx); }); },
             gprx, gpry);
    }
    T mu[NM], gmx[NM], gmy[NM];
#pragma unroll
    for (int j = 0; j < NM; ++j) {
        mu[j] = Ma(j, 0, 0);
        grad([&](int dy, int dx) { return Ma(j, dy, dx); }, gmx[j], gmy[j]);
    }
    T Gx, Gy;
    if constexpr (NP == 2) {
        const T dC = Cv[0] - Cv[1];
        Gx = dC * gmx[0];
        Gy = dC * gmy[0];
    } else {
        Gx = Gy = T(0);
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            Gx += Cv[j] * gmx[j];
            Gy += Cv[j] * gmy[j];
        }
    }
    T Qx[M], Qy[M], tQx = T(0), tQy = T(0);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        Qx[i] = Cv[i] * (gmx[i] - Gx);
        Qy[i] = Cv[i] * (gmy[i] - Gy);
        tQx += P.drho[i] * Qx[i];
        tQy += P.drho[i] * Qy[i];
    }
    const T pm0 = -(P.m0 * psi);
    const T mCx = pm0 * tQx, mCy = pm0 * tQy;   // psi m^C
    T dax, day;
    grad([&](int dy, int dx) { return Aa(dy, dx); }, dax, day);
    auto lag = [&](int k) { return st_lag[k * pl + o]; };
    T mg[9], sum_g;
    {
        T g[9];
#pragma unroll
        for (int p = 0; p < 9; ++p) g[p] = st_g[p * pl + o];
        sum_g = dev::hermite_moments(g, cs2, mg);
    }
    T dm[M];   // mu_j - mu_N
    T sx = rho * P.body[0], sy = rho * P.body[1];
#pragma unroll
    for (int j = 0; j < M; ++j) {
        if constexpr (NP == 2) dm[0] = mu[0] + mu[0];
        else dm[j] = mu[j] - mu[NM - 1];
        sx += dm[j] * gCx[j];
        sy += dm[j] * gCy[j];
    }
    const T F0x = psi * sx + day, F0y = psi * sy - dax;
    const T psirho = psi * rho;
    const T dmp = P.damp - P.damp * psi;
    const T inv_den = dev::rcp(psirho + T(0.5) * dmp);
    const T u0x = (mg[1] + T(0.5) * F0x) * inv_den, u0y = (mg[2] + T(0.5) * F0y) * inv_den;
    const T hi = T(0.5) * inv_den;
    const T ex = gpx * hi, ey = gpy * hi;
    const T Hs = P.Hfac - T(2) * P.Hfac * inv_s21;
    const T Ap = P.A_P * psi;
    const T gq = P.gam * psirho;
    const T vx = Ap * grx + P.gam * mCx + Hs * gprx + gq * u0x;
    const T vy = Ap * gry + P.gam * mCy + Hs * gpry + gq * u0y;
    const T wx = vx + gq * u0x, wy = vy + gq * u0y;
    const T ee = ex * ex + ey * ey;
    const T qa = P.cP * gq * ee;
    const T qb = P.cP * (wx * ex + wy * ey) - psi;
    const T qc = P.cP * (sum_g - P.Kh * lag(2 * NP + 2) + vx * u0x + vy * u0y);
    const T disc = dev::clamp0(qb * qb - T(4) * qa * qc);
    const T sroot = dev::signed_as(dev::root(disc), qb);
    const T inv_D = dev::rcp(qb + sroot);
    const T Pr = T(-2) * qc * inv_D;
    const T ux = u0x + Pr * ex, uy = u0y + Pr * ey;

    // ---- adjoints of the outputs: transposed push streaming -------------
    // (the forward sends population p of this node to tgt in direction tdir)
    long long tgt[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        int tx = x + aCx[p], ty = y + aCy[p];
        bool bounce = false;
        if (tx < 0 || tx >= P.nx) {
            if (P.px) tx = tx < 0 ? tx + P.nx : tx - P.nx;
            else bounce = true;
        }
        if (ty < 0 || ty >= P.ny) {
            if (P.py) ty = ty < 0 ? ty + P.ny : ty - P.ny;
            else bounce = true;
        }
        tgt[p] = bounce ? opp(p) * pl + o : p * pl + P.org + (long long)ty * P.pitch + tx;
    }
    auto lo_lag = [&](int k) { return ad_lag_in[k * pl + o]; };
    auto lo_g = [&](int p) { return ad_pop_in[(long long)9 * M * pl + tgt[p]]; };

    // accumulators of the intermediate adjoints
    T l_psi, l_ux, l_uy, l_gprx, l_gpry, l_mCx, l_mCy, l_Fx, l_Fy, l_psiP, l_psirho, l_grx, l_gry;
    T l_s21, l_s22, lmg[9];

    // ---- flow LB (Eqs. 3.2, 3.8, 3.10) reversed ---------------------------
    {
        T lk[9];
        {
            T wl[9];
#pragma unroll
            for (int p = 0; p < 9; ++p) wl[p] = -(P.w9[p == 0 ? 0 : p <= 4 ? 1 : 2] * lo_g(p));
            dev::hermite_moments(wl, cs2, lk);
        }
        const T jx = psirho * ux, jy = psirho * uy;
        const T p1 = mCx * uy, p2 = ux * mCy;
        const T Txx = mCx * ux, Tyy = mCy * uy, Txy = T(0.5) * (p1 + p2);
        const T s1 = ux * gprx, s2 = uy * gpry;
        const T cu = P.c2m3cs2 * (s1 + s2);
        const T Mxx = (Txx - lag(2 * NP - 1)) + P.two_cs2 * s1 + cu;
        const T Myy = (Tyy - lag(2 * NP)) + P.two_cs2 * s2 + cu;
        const T Mxy = (Txy - lag(2 * NP + 1)) + cs2 * (ux * gpry + gprx * uy);
        const T psiP = psi * Pr;
        const T l20 = s21 * P.invN20, l11 = s22 * P.invN11;
        const T R3 = mg[3] - (psiP + jx * ux + Txx) + T(0.5) * Mxx;
        const T R4 = mg[4] - (psiP + jy * uy + Tyy) + T(0.5) * Myy;
        const T R5 = mg[5] - (jx * uy + Txy) + T(0.5) * Mxy;
        const T c20 = T(0.5) * l20 - P.invN20, c11 = T(0.5) * l11 - P.invN11;
        lmg[0] = P.lg00 * lk[0];
        lmg[1] = P.lg1 * lk[1];
        lmg[2] = P.lg1 * lk[2];
        lmg[3] = l20 * lk[3];
        lmg[4] = l20 * lk[4];
        lmg[5] = l11 * lk[5];
        lmg[6] = P.lg3 * lk[6];
        lmg[7] = P.lg3 * lk[7];
        lmg[8] = P.lg4 * lk[8];
        const T l_a0 = P.cg0 * lk[0];
        T l_jx = -lmg[1], l_jy = -lmg[2];
        l_Fx = P.cg1 * lk[1];
        l_Fy = P.cg1 * lk[2];
        l_psiP = cs2 * lmg[8] - (lmg[3] + lmg[4]);
        l_s21 = P.invN20 * (R3 * lk[3] + R4 * lk[4]);
        l_s22 = P.invN11 * (R5 * lk[5]);
        const T l_Mxx = c20 * lk[3], l_Myy = c20 * lk[4], l_Mxy = c11 * lk[5];
        ad_lag_out[(2 * NP - 1) * pl + o] = -l_Mxx;
        ad_lag_out[(2 * NP) * pl + o] = -l_Myy;
        ad_lag_out[(2 * NP + 1) * pl + o] = -l_Mxy;
        // (psi m . u)_new = A_xx + A_yy, A = j u + T
        const T lpm = lo_lag(2 * NP + 2);
        const T l_Axx = lpm - lmg[3], l_Ayy = lpm - lmg[4], l_Axy = -lmg[5];
        // a0 = psi (u . grad rho)
        const T pa = psi * l_a0;
        l_psi = (ux * grx + uy * gry) * l_a0;
        l_ux = grx * pa;
        l_uy = gry * pa;
        l_grx = ux * pa;
        l_gry = uy * pa;
        // M^2G
        const T l_cu = P.c2m3cs2 * (l_Mxx + l_Myy);
        const T l_s1 = P.two_cs2 * l_Mxx + l_cu, l_s2 = P.two_cs2 * l_Myy + l_cu;
        const T cxy = cs2 * l_Mxy;
        l_ux += gprx * l_s1 + gpry * cxy;
        l_uy += gpry * l_s2 + gprx * cxy;
        l_gprx = ux * l_s1 + uy * cxy;
        l_gpry = uy * l_s2 + ux * cxy;
        // A
        l_jx += ux * l_Axx + uy * l_Axy;
        l_jy += uy * l_Ayy;
        l_ux += jx * l_Axx;
        l_uy += jy * l_Ayy + jx * l_Axy;
        // T, and a_new = (p1 - p2) / 2
        const T l_Txx = l_Mxx + l_Axx + lo_lag(2 * NP - 1);
        const T l_Tyy = l_Myy + l_Ayy + lo_lag(2 * NP);
        const T l_Txy = l_Mxy + l_Axy + lo_lag(2 * NP + 1);
        const T la = lo_lag(0);
        const T l_p1 = T(0.5) * (l_Txy + la), l_p2 = T(0.5) * (l_Txy - la);
        l_mCx = ux * l_Txx + uy * l_p1;
        l_mCy = uy * l_Tyy + ux * l_p2;
        l_ux += mCx * l_Txx + mCy * l_p2;
        l_uy += mCy * l_Tyy + mCx * l_p1;
        // j = psi rho u
        l_psirho = ux * l_jx + uy * l_jy;
        l_ux += psirho * l_jx;
        l_uy += psirho * l_jy;
    }

    // ---- phase LB (Eqs. 3.1, 3.5-3.7) reversed, one phase at a time ------
    T l_mu[NM], l_gmx[NM], l_gmy[NM], l_Qx[M], l_Qy[M], l_gpx = T(0), l_gpy = T(0);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        T lout[9], lm[9], lk[9];
        T psiC;
        {
            T v[9];
#pragma unroll
            for (int p = 0; p < 9; ++p) v[p] = st_pop[(long long)(9 * i + p) * pl + o];
            psiC = (((v[7] + v[8]) + v[4]) + (v[3] + v[1]) + ((v[6] + v[5]) + v[2])) + v[0];
        }
        {
            T wl[9];
#pragma unroll
            for (int p = 0; p < 9; ++p) {
                lout[p] = ad_pop_in[(long long)9 * i * pl + tgt[p]];
                wl[p] = -(P.w9[p == 0 ? 0 : p <= 4 ? 1 : 2] * lout[p]);
            }
            dev::hermite_moments(wl, cs2, lk);
        }
        const T* lam = P.lamf[i];
#pragma unroll
        for (int a = 1; a < 9; ++a) lm[a] = lam[a] * lk[a];
        const T l_Vx = P.cV[i] * lk[1], l_Vy = P.cV[i] * lk[2];
        const T l_pcux = l_Vx - lm[1] + lo_lag(1 + 2 * i), l_pcuy = l_Vy - lm[2] + lo_lag(2 + 2 * i);
        // X = psi C - eta psi mu_i
        const T l_X = cs2 * (lm[3] + lm[4]) - P.cs4 * lm[8];
        const T el = P.eta[i] * l_X;
        // V = dt(psi C u) + cs2 eta (mu grad psi + psi (grad mu - Q))
        const T cx = P.ceta[i] * l_Vx, cy = P.ceta[i] * l_Vy;
        l_mu[i] = gpx * cx + gpy * cy - psi * el;
        l_gpx += mu[i] * cx;
        l_gpy += mu[i] * cy;
        l_psi += (gmx[i] - Qx[i]) * cx + (gmy[i] - Qy[i]) * cy - mu[i] * el;
        l_gmx[i] = psi * cx;
        l_gmy[i] = psi * cy;
        l_Qx[i] = -l_gmx[i];
        l_Qy[i] = -l_gmy[i];
        ad_lag_out[(1 + 2 * i) * pl + o] = -l_Vx;
        ad_lag_out[(2 + 2 * i) * pl + o] = -l_Vy;
        lm[0] = l_X + ux * l_pcux + uy * l_pcuy;
        l_ux += psiC * l_pcux;
        l_uy += psiC * l_pcuy;
        T Bm[9];
        hermite_B(lm, cs2, Bm);
#pragma unroll
        for (int p = 0; p < 9; ++p) ad_pop_out[(long long)(9 * i + p) * pl + o] = lout[p] + Bm[p];
    }
    if constexpr (NP > 2) l_mu[NM - 1] = l_gmx[NM - 1] = l_gmy[NM - 1] = T(0);

    // ---- velocity, force and the Eq. 19 pressure reversed ---------------
    // F = F0 + P grad psi - dmp u, psi P, u = u0 + P e
    l_psi += Pr * l_psiP;
    l_gpx += Pr * l_Fx;
    l_gpy += Pr * l_Fy;
    T l_dmp = -(ux * l_Fx + uy * l_Fy);
    T l_u0x = l_ux - dmp * l_Fx, l_u0y = l_uy - dmp * l_Fy;
    const T l_Pr = psi * l_psiP + gpx * l_Fx + gpy * l_Fy + ex * l_u0x + ey * l_u0y;
    T l_ex = Pr * l_u0x, l_ey = Pr * l_u0y;
    // dP = -(P^2 dqa + P dqb + dqc) / (2 qa P + qb), and 2 qa P + qb is the
    // signed root; where the discriminant was clamped P = -2 qc / qb
    T l_qa, l_qb, l_qc;
    if (dev::positive(disc)) {
        l_qc = -l_Pr * dev::rcp(sroot);
        l_qb = Pr * l_qc;
        l_qa = Pr * l_qb;
    } else {
        l_qc = T(-2) * inv_D * l_Pr;
        l_qb = -Pr * inv_D * l_Pr;
        l_qa = T(0);
    }
    const T cA = P.cP * l_qa, cB = P.cP * l_qb, l_G0 = P.cP * l_qc;
    l_psi -= l_qb;
    const T l_wx = cB * ex, l_wy = cB * ey;
    const T g2 = T(2) * gq * cA;
    l_ex += cB * wx + g2 * ex;
    l_ey += cB * wy + g2 * ey;
    const T l_vx = l_G0 * u0x + l_wx, l_vy = l_G0 * u0y + l_wy;
    l_u0x += l_G0 * vx + gq * (l_wx + l_vx);
    l_u0y += l_G0 * vy + gq * (l_wy + l_vy);
    l_psirho += P.gam * (cA * ee + u0x * (l_wx + l_vx) + u0y * (l_wy + l_vy));
    ad_lag_out[(2 * NP + 2) * pl + o] = -P.Kh * l_G0;
    // b = A_P psi grad rho + gamma psi m^C + Hs grad(psi rho), l_b = l_v
    l_psi += P.A_P * (grx * l_vx + gry * l_vy);
    l_grx += Ap * l_vx;
    l_gry += Ap * l_vy;
    l_mCx += P.gam * l_vx;
    l_mCy += P.gam * l_vy;
    l_gprx += Hs * l_vx;
    l_gpry += Hs * l_vy;
    const T l_inv_s21 = T(-2) * P.Hfac * (gprx * l_vx + gpry * l_vy) - s21 * s21 * l_s21;
    // e = grad psi / (2 den), u0 = (J + F0 / 2) / den, den = psi rho + dmp / 2
    l_gpx += hi * l_ex;
    l_gpy += hi * l_ey;
    const T l_den = -inv_den * (hi * (gpx * l_ex + gpy * l_ey) + u0x * l_u0x + u0y * l_u0y);
    const T l_Jx = inv_den * l_u0x, l_Jy = inv_den * l_u0y;
    const T l_F0x = l_Fx + T(0.5) * l_Jx, l_F0y = l_Fy + T(0.5) * l_Jy;
    l_psirho += l_den;
    l_dmp += T(0.5) * l_den;
    l_psi -= P.damp * l_dmp;
    // the flow populations: J and sum_{p>0} g_p are moments too
    {
        T Bm[9];
        lmg[0] += l_G0;
        lmg[1] += l_Jx;
        lmg[2] += l_Jy;
        hermite_B(lmg, cs2, Bm);
        Bm[0] -= l_G0;
        T* ad_g = ad_pop_out + (long long)9 * M * pl;
#pragma unroll
        for (int p = 0; p < 9; ++p) ad_g[p * pl + o] = lo_g(p) + Bm[p];
    }
    W.lga[o] = -l_F0y;
    W.lga[pl + o] = l_F0x;
    W.lgp[o] = l_gpx;
    W.lgp[pl + o] = l_gpy;
    W.lgpr[o] = l_gprx;
    W.lgpr[pl + o] = l_gpry;
    // F0 = psi s + (d_y a, -d_x a), s = rho b + sum_j (mu_j - mu_N) grad C_j
    l_psi += sx * l_F0x + sy * l_F0y + rho * l_psirho;
    const T l_sx = psi * l_F0x, l_sy = psi * l_F0y;
    const T l_rho = P.body[0] * l_sx + P.body[1] * l_sy + psi * l_psirho;
    const T l_nu = P.nu_to_s21 * l_inv_s21 - P.nu_to_s22 * (s22 * s22 * l_s22);
#pragma unroll
    for (int j = 0; j < M; ++j) {
        const T d = gCx[j] * l_sx + gCy[j] * l_sy;
        if constexpr (NP == 2) {
            l_mu[0] += d + d;
        } else {
            l_mu[j] += d;
            l_mu[NM - 1] -= d;
        }
        W.lgC[(2 * j) * pl + o] = dm[j] * l_sx + P.drho[j] * l_grx;
        W.lgC[(2 * j + 1) * pl + o] = dm[j] * l_sy + P.drho[j] * l_gry;
    }
    // psi m^C = -m0 psi sum_i (rho_i - rho_N) Q_i, Q_i = C_i (grad mu_i - G)
    l_psi -= P.m0 * (tQx * l_mCx + tQy * l_mCy);
    W.lpsi[o] = l_psi;
    const T mx = pm0 * l_mCx, my = pm0 * l_mCy;
    T l_C[M], l_Gx = T(0), l_Gy = T(0);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        const T qx = l_Qx[i] + P.drho[i] * mx, qy = l_Qy[i] + P.drho[i] * my;
        l_C[i] = (gmx[i] - Gx) * qx + (gmy[i] - Gy) * qy + P.drho[i] * l_rho + P.dnu[i] * l_nu;
        const T cx = Cv[i] * qx, cy = Cv[i] * qy;
        l_gmx[i] += cx;
        l_gmy[i] += cy;
        l_Gx -= cx;
        l_Gy -= cy;
    }
    // G = sum_j C_j grad mu_j, C_N = 1 - sum_j C_j
    if constexpr (NP == 2) {
        const T d = gmx[0] * l_Gx + gmy[0] * l_Gy, dC = Cv[0] - Cv[1];
        l_C[0] += d + d;
        l_gmx[0] += dC * l_Gx;
        l_gmy[0] += dC * l_Gy;
    } else {
        const T dN = gmx[NM - 1] * l_Gx + gmy[NM - 1] * l_Gy;
#pragma unroll
        for (int j = 0; j < M; ++j) l_C[j] += gmx[j] * l_Gx + gmy[j] * l_Gy - dN;
#pragma unroll
        for (int j = 0; j < NM; ++j) {
            l_gmx[j] += Cv[j] * l_Gx;
            l_gmy[j] += Cv[j] * l_Gy;
        }
    }
#pragma unroll
    for (int j = 0; j < M; ++j) W.lC[j * pl + o] = l_C[j];
#pragma unroll
    for (int j = 0; j < NM; ++j) {
        W.lmu[j * pl + o] = l_mu[j];
        W.lgm[(2 * j) * pl + o] = l_gmx[j];
        W.lgm[(2 * j + 1) * pl + o] = l_gmy[j];
    }
}

// Shared-memory copy of planes over a block plus a 1-node ring: entry
// (k, ly, lx) holds plane k at node (x0 - 1 + lx, y0 - 1 + ly), wrapped or
// mirrored at the domain's edge (ring_index).  kPairs: the planes are (x, y)
// components in turn, and a mirror reverses the component across its wall:
// the source s = (x, 0) reaches the ghost node (x, -1) by c_p with c_py = -1,
// weight gw_p (c_px v_x - v_y), which is what a source (v_x, -v_y) at (x, -1)
// gives the node (x, 0) by c_py = +1; scalars carry over unchanged.  (With
// zeros beyond the edge and the images gathered from memory by the edge
// nodes, gather3 took 18.6 us at 256 x 256 in FP32, N = 2, and gather2 11.)
// Plain loads, all of a call's before its first shared-memory store, so that
// they are in flight at once.  (Not the read-only path: the kernel before
// this one may still write these planes when this one starts, see
// wait_for_previous.)
template <typename T>
struct Ring {
    static constexpr int AY = block_rows<T>(), W = AX + 2, H = AY + 2, N = W * H, NT = AX * AY, R = (N + NT - 1) / NT;
    long long g[R];      // offsets of this thread's ring nodes (beyond the last they repeat it)
    bool mx[R], my[R];   // mirrored along x, y
    __device__ Ring(const KParams<T>& P, int x0, int y0) {
        const int tid = threadIdx.y * AX + threadIdx.x;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int k = min(tid + r * NT, N - 1), ly = k / W, lx = k - ly * W;
            const int X = x0 - 1 + lx, Y = y0 - 1 + ly;
            mx[r] = !P.px && (X < 0 || X >= P.nx);
            my[r] = !P.py && (Y < 0 || Y >= P.ny);
            g[r] = P.org + (long long)ring_index(Y, P.ny, P.py) * P.pitch + ring_index(X, P.nx, P.px);
        }
    }
};
template <typename T, int NPL, bool kPairs>
__device__ __forceinline__ void load_ring(const KParams<T>& P, const Ring<T>& ring, T* sm, const T* base) {
    using R = Ring<T>;
    const int tid = threadIdx.y * AX + threadIdx.x;
    T v[R::R][NPL];
#pragma unroll
    for (int r = 0; r < R::R; ++r)
#pragma unroll
        for (int q = 0; q < NPL; ++q) v[r][q] = base[q * P.plane + ring.g[r]];
#pragma unroll
    for (int r = 0; r < R::R; ++r) {
        const int k = min(tid + r * R::NT, R::N - 1);
#pragma unroll
        for (int q = 0; q < NPL; ++q)
            sm[q * R::N + k] = kPairs && (q % 2 ? ring.my[r] : ring.mx[r]) ? -v[r][q] : v[r][q];
    }
}
// sum_p gw_p (c_p . (vx, vy))(q - c_p) from the ring copy, q = thread's node
template <typename T>
__device__ __forceinline__ T grad_T_sm(const KParams<T>& P, const T* vx, const T* vy, int lx, int ly) {
    constexpr int W = Ring<T>::W;
    const int c = (ly + 1) * W + lx + 1;
    // the axis neighbours, and per diagonal direction both components
    const T ax = (vx[c - 1] - vx[c + 1]) + (vy[c - W] - vy[c + W]);
    const T d1 = (vx[c - W - 1] - vx[c + W + 1]) + (vy[c - W - 1] - vy[c + W + 1]);
    const T d2 = (vx[c + W - 1] - vx[c - W + 1]) + (vy[c - W + 1] - vy[c + W - 1]);
    return P.gw1 * ax + P.gw2 * (d1 + d2);
}

// ---- transposed stencils of the node update -------------------------------
// LC_j, Lpsi, Lmu_j at every node, and the adjoint of the lagged plane a
// straight into the output state.  Ring copies (shared memory) of the vector
// pairs: grad C_j (N-1), grad psi, grad(psi rho), grad mu_j, grad a.
template <typename T, int NP>
__device__ __forceinline__ void mu_node_at(const KParams<T>& P, const T* __restrict__ psi_pl,
                                           const T* __restrict__ cosf, const AdjPlanes<T, NP>& W,
                                           double* dJ_dcos, int x, int y,
                                           const T (&Lmu_kept)[mu_planes<NP>()]);

// The chemical-potential VJP (mu_node_at) of the node follows in the same
// thread from the gathered adjoint of mu, which then never reaches memory
// (the initial state's reverse runs k_adj_mu_node on its own).
template <typename T, int NP>
__global__ void __launch_bounds__(AX * block_rows<T>()) k_adj_gather3(KParams<T> P, const T* __restrict__ psi_pl,
                                                     AdjPlanes<T, NP> W, T* __restrict__ ad_lag_out,
                                                     const T* __restrict__ cosf, double* dJ_dcos) {
    constexpr int NM = mu_planes<NP>(), NV = AdjPlanes<T, NP>::NV, RN = Ring<T>::N;
    extern __shared__ __align__(16) unsigned char g3_raw[];
    T* sm = reinterpret_cast<T*>(g3_raw);
    wait_for_previous();
    const long long pl = P.plane;
    const int x0 = first_x<T>(), y0 = first_y<T>();
    load_ring<T, NV, true>(P, Ring<T>(P, x0, y0), sm, W.lgC);
    __syncthreads();
    if constexpr (overlaps<T>()) dependents_may_start();
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    const int lx = threadIdx.x, ly = threadIdx.y;
    const long long o = P.org + (long long)y * P.pitch + x;
    auto gT = [&](int k) { return grad_T_sm(P, sm + k * RN, sm + (k + 1) * RN, lx, ly); };
    constexpr int kC = 0, kP = 2 * (NP - 1), kR = kP + 2, kM = kR + 2, kA = kM + 2 * NM;
    T LC[NP - 1], Lmu[NM];
    const T psiq = psi_pl[o];
    const T lchi = gT(kR), plchi = psiq * lchi;
    T rq = P.rho[NP - 1];
#pragma unroll
    for (int j = 0; j < NP - 1; ++j) {
        rq += P.drho[j] * W.C[j * pl + o];
        LC[j] = W.lC[j * pl + o] + gT(kC + 2 * j) + P.drho[j] * plchi;
    }
    const T Lpsi = W.lpsi[o] + gT(kP) + rq * lchi;
#pragma unroll
    for (int j = 0; j < NM; ++j) Lmu[j] = W.lmu[j * pl + o] + gT(kM + 2 * j);
    ad_lag_out[o] = gT(kA);
#pragma unroll
    for (int j = 0; j < NP - 1; ++j) W.LC[j * pl + o] = LC[j];
    W.Lpsi[o] = Lpsi;
    mu_node_at<T, NP>(P, psi_pl, cosf, W, dJ_dcos, x, y, Lmu);
}

// ---- VJP of the chemical potential (Eq. 2.14) per node ---------------------
template <typename T, int NP>
__device__ __forceinline__ void mu_node_at(const KParams<T>& P, const T* __restrict__ psi_pl,
                                           const T* __restrict__ cosf, const AdjPlanes<T, NP>& W,
                                           double* dJ_dcos, int x, int y,
                                           const T (&Lmu_kept)[mu_planes<NP>()]) {
    const long long pl = P.plane;
    const long long o = P.org + (long long)y * P.pitch + x;
    const PlaneAt<T> Ca{W.C, pl, o, P.pitch}, Ps{psi_pl, pl, o, P.pitch};
    T Lmu[NP];   // two phases: mu_1 alone is kept, mu_2 = -mu_1 carries none of its own
#pragma unroll
    for (int i = 0; i < NP; ++i) Lmu[i] = i < mu_planes<NP>() ? Lmu_kept[i < mu_planes<NP>() ? i : 0] : T(0);
    T cth[NP];
    node_cth<T, NP>(P, cosf, o, cth);
    // forward (dev::chem_pot: mu_i = bulk_i + v_i / psi, bulk_i = sum_j 2
    // beta_ij (g'(C_i) - g'(C_i + C_j)), v_i = sum_j sigma_ij V_j, V_j = (3 eps
    // / 4) div(psi grad C_j) + 3 |grad psi| W_j, W_j = C_j sum_q cos_jq C_q)
    const T p0 = Ps(0, 0);
    // summed side by side, not by diagonals as grad9: FP32 rounding decides
    // which nodes of the fluid bulk pass kKinkGradPsi below, and this order is
    // the one the FP32 gradients are stated for
    const T pE = Ps(0, 1), pW = Ps(0, -1), pN = Ps(1, 0), pS = Ps(-1, 0);
    const T pNE = Ps(1, 1), pNW = Ps(1, -1), pSW = Ps(-1, -1), pSE = Ps(-1, 1);
    const T gpx = P.gw1 * (pE - pW) + P.gw2 * ((pNE - pNW) + (pSE - pSW));
    const T gpy = P.gw1 * (pN - pS) + P.gw2 * ((pNE + pNW) - (pSE + pSW));
    const T agp = dev::root(gpx * gpx + gpy * gpy);
    T Cv[NP], V[NP];
    {
        T sC = T(0), sL = T(0);
#pragma unroll
        for (int j = 0; j < NP - 1; ++j) {
            const T c0 = Ca(j, 0, 0);
            const T l = P.lk1 * ((p0 + Ps(0, 1)) * (Ca(j, 0, 1) - c0) + (p0 + Ps(0, -1)) * (Ca(j, 0, -1) - c0) +
                                 (p0 + Ps(1, 0)) * (Ca(j, 1, 0) - c0) + (p0 + Ps(-1, 0)) * (Ca(j, -1, 0) - c0)) +
                        P.lk2 * ((p0 + Ps(1, 1)) * (Ca(j, 1, 1) - c0) + (p0 + Ps(1, -1)) * (Ca(j, 1, -1) - c0) +
                                 (p0 + Ps(-1, -1)) * (Ca(j, -1, -1) - c0) + (p0 + Ps(-1, 1)) * (Ca(j, -1, 1) - c0));
            Cv[j] = c0;
            V[j] = l;
            sC = j == 0 ? c0 : sC + c0;
            sL = j == 0 ? l : sL + l;
        }
        Cv[NP - 1] = T(1) - sC;
        V[NP - 1] = -sL;
    }
    T cpair[NP][NP], acc[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i)
#pragma unroll
        for (int j = i + 1; j < NP; ++j) {
            const T c = j < NP - 1 ? (P.sigN[i] * cth[i] - P.sigN[j] * cth[j]) * P.invsig[i][j] : cth[i];
            cpair[i][j] = c;
            cpair[j][i] = -c;
        }
    const T agp3 = T(3) * agp;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        T a = T(0);
#pragma unroll
        for (int q = 0; q < NP; ++q)
            if (q != j) a = q == (j == 0 ? 1 : 0) ? cpair[j][q] * Cv[q] : a + cpair[j][q] * Cv[q];
        acc[j] = a;
        V[j] += agp3 * (Cv[j] * a);
    }
    const T inv_p0 = dev::rcp(p0);
    // reverse: l_v_i = Lmu_i / psi, l_V_j = sum_i sigma_ij l_v_i
    T lv[NP], l_V[NP];
    T l_inv = T(0);   // sum_i v_i l_v_i = sum_j V_j l_V_j
#pragma unroll
    for (int i = 0; i < NP; ++i) lv[i] = Lmu[i] * inv_p0;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        T t = T(0);
#pragma unroll
        for (int i = 0; i < NP; ++i)
            if (i != j) t = i == (j == 0 ? 1 : 0) ? P.sig[i][j] * lv[i] : t + P.sig[i][j] * lv[i];
        l_V[j] = t;
        l_inv = j == 0 ? V[0] * t : l_inv + V[j] * t;
    }
    const T l_p0 = -inv_p0 * l_inv;
    T l_agp = T(0), l_Cv[NP], l_W[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        const T ca = Cv[j] * acc[j];
        l_agp = j == 0 ? ca * l_V[0] : l_agp + ca * l_V[j];
        l_W[j] = agp3 * l_V[j];
    }
    l_agp *= T(3);
    // bulk: g'(C_i) with weight sum_j 2 beta_ij, and the pairs; what adds the
    // same to every l_C drops out below (C_N = 1 - sum C_j), so g'(C_i + C_j)
    // counts once per pair of complements (none for two phases, -g'(C_k) for
    // three)
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        T l_gp = P.beta2s[i] * Lmu[i];
        if constexpr (NP == 3) {
            const int a = i == 0 ? 1 : 0, b = i == 2 ? 1 : 2;
            l_gp += P.beta2[a][b] * (Lmu[a] + Lmu[b]);
        }
        l_Cv[i] = gsecond(Cv[i]) * l_gp + acc[i] * l_W[i];
    }
    if constexpr (NP == 4) {
#pragma unroll
        for (int j = 1; j < 4; ++j) {
            const int k = j == 1 ? 2 : 1, l = j == 3 ? 2 : 3;
            const T t = gsecond(Cv[0] + Cv[j]) *
                        (P.beta2[k][l] * (Lmu[k] + Lmu[l]) - P.beta2[0][j] * (Lmu[0] + Lmu[j]));
            l_Cv[0] += t;
            l_Cv[j] += t;
        }
    }
    // W_j = C_j sum_{q != j} cos_jq C_q, cos_jq = (a_j - a_q) / sigma_jq
    T l_aj[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) l_aj[j] = T(0);
#pragma unroll
    for (int j = 0; j < NP; ++j)
#pragma unroll
        for (int q = j + 1; q < NP; ++q) {
            const T d = l_W[j] - l_W[q];
            // d W_j / d C_q = cos_jq C_j, d W_q / d C_j = -cos_jq C_q; the
            // terms cos_jq C_q of W_j's own C_j are in acc above
            l_Cv[q] += cpair[j][q] * Cv[j] * l_W[j];
            l_Cv[j] -= cpair[j][q] * Cv[q] * l_W[q];
            const T lc = Cv[j] * Cv[q] * d * P.invsig[j][q];
            l_aj[j] += lc;
            if (q < NP - 1) l_aj[q] -= lc;
        }
    const long long node = (long long)y * P.nx + x;
    const long long nn = (long long)P.nx * P.ny;
#pragma unroll
    for (int j = 0; j < NP - 1; ++j) dJ_dcos[j * nn + node] += (double)(P.sigN[j] * l_aj[j]);
    // |grad psi| has a kink at grad psi = 0.  In the fluid bulk psi is 1 up
    // to rounding, and the direction of a rounding-level gradient would
    // carry the wetting term's full weight into dJ/dpsi there; below
    // kKinkGradPsi the derivative is taken as zero, the value central
    // differences give at the kink.
    T l_gpx = T(0), l_gpy = T(0);
    if (agp > T(kKinkGradPsi)) {
        const T r = dev::rcp(agp) * l_agp;
        l_gpx = gpx * r;
        l_gpy = gpy * r;
    }
#pragma unroll
    for (int j = 0; j < NP - 1; ++j) {
        W.mC[j * pl + o] = l_Cv[j] - l_Cv[NP - 1];
        W.mL[j * pl + o] = l_V[j] - l_V[NP - 1];   // of (3 eps / 4) div(psi grad C_j)
    }
    W.mpsi[o] = l_p0;
    W.mgp[o] = l_gpx;
    W.mgp[pl + o] = l_gpy;
}

template <typename T, int NP>
__global__ void __launch_bounds__(AX * block_rows<T>()) k_adj_mu_node(KParams<T> P, const T* __restrict__ psi_pl,
                                                     const T* __restrict__ cosf, AdjPlanes<T, NP> W,
                                                     double* __restrict__ dJ_dcos) {
    const int x = first_x<T>() + threadIdx.x, y = first_y<T>() + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    const long long o = P.org + (long long)y * P.pitch + x;
    T Lmu[mu_planes<NP>()];
#pragma unroll
    for (int i = 0; i < mu_planes<NP>(); ++i) Lmu[i] = W.Lmu[i * P.plane + o];
    mu_node_at<T, NP>(P, psi_pl, cosf, W, dJ_dcos, x, y, Lmu);
}

// ---- transposed div(psi grad C_j) and grad psi stencils, then
//      C_i = sum_p f^i_p / psi reversed and dJ/dpsi ------------------------------
// Ring copies: grad psi pair, mL_j (N-1), psi, C_j (N-1).
template <typename T, int NP>
__global__ void __launch_bounds__(AX * block_rows<T>()) k_adj_gather2(KParams<T> P, const T* __restrict__ psi_pl,
                                                     AdjPlanes<T, NP> W, T* ad_pop_out,
                                                     double* dJ_dpsi, int initial) {
    extern __shared__ __align__(16) unsigned char g2_raw[];
    constexpr int RN = Ring<T>::N, RW = Ring<T>::W;
    T* sm = reinterpret_cast<T*>(g2_raw);
    wait_for_previous();
    const long long pl = P.plane;
    const int x0 = first_x<T>(), y0 = first_y<T>();
    T* sG = sm;
    T* sL = sG + 2 * RN;
    T* sP = sL + (NP - 1) * RN;
    T* sC = sP + RN;
    const Ring<T> ring(P, x0, y0);
    load_ring<T, 2, true>(P, ring, sG, W.mgp);
    load_ring<T, NP - 1, false>(P, ring, sL, W.mL);
    load_ring<T, 1, false>(P, ring, sP, psi_pl);
    load_ring<T, NP - 1, false>(P, ring, sC, W.C);
    __syncthreads();
    if constexpr (overlaps<T>()) dependents_may_start();
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    const int lx = threadIdx.x, ly = threadIdx.y;
    const long long o = P.org + (long long)y * P.pitch + x;
    const int rc = (ly + 1) * RW + lx + 1;
    const T psio = sP[rc];
    T lC[NP - 1];
    T lpsi = W.Lpsi[o] + W.mpsi[o] + grad_T_sm(P, sG, sG + RN, lx, ly);
    // node o as the neighbour of s, and as the centre with neighbour s: with
    // t_s = (psi_s + psi_o) and m_s = mL_s - mL_o,
    //   l_C_j += sum_s lk t_s m_s, l_psi += sum_s lk (C_o - C_s) m_s
    // (the stencil of the centre contributes -mL_o and the neighbours' mL_s)
#pragma unroll
    for (int j = 0; j < NP - 1; ++j) {
        const T *L = sL + j * RN, *C = sC + j * RN;
        const T mo = L[rc], co = C[rc];
        T c1 = T(0), c2 = T(0), p1 = T(0), p2 = T(0);
#pragma unroll
        for (int p = 1; p < 9; ++p) {
            const int r = rc - aCy[p] * RW - aCx[p];
            const T m = L[r] - mo, t = psio + sP[r], d = co - C[r];
            if (p == 1) {
                c1 = t * m;
                p1 = d * m;
            } else if (p == 5) {
                c2 = t * m;
                p2 = d * m;
            } else if (p <= 4) {
                c1 += t * m;
                p1 += d * m;
            } else {
                c2 += t * m;
                p2 += d * m;
            }
        }
        lC[j] = W.LC[j * pl + o] + W.mC[j * pl + o] + P.lk1 * c1 + P.lk2 * c2;
        lpsi += P.lk1 * p1 + P.lk2 * p2;
    }
    if (!initial) {
        // C_i = sum_p f^i_p / psi
        const T inv = dev::rcp(psio);
#pragma unroll
        for (int i = 0; i < NP - 1; ++i) {
            const T d = lC[i] * inv;
            // all nine loads before any store (the compiler cannot tell the
            // planes apart, so interleaved read-modify-writes would serialise)
            T v[9];
#pragma unroll
            for (int p = 0; p < 9; ++p) v[p] = ad_pop_out[(9 * i + p) * pl + o];
#pragma unroll
            for (int p = 0; p < 9; ++p) ad_pop_out[(9 * i + p) * pl + o] = v[p] + d;
            lpsi -= d * sC[i * RN + rc];
        }
    }
    dJ_dpsi[(long long)y * P.nx + x] += (double)lpsi;
}

// ---- initial state reversed: f^i_p = w_p eta_i psi mu_i (p > 0),
//      f^i_0 = (w_0 - 1) eta_i psi mu_i + psi C0_i ------------------------------
template <typename T, int NP>
__global__ void __launch_bounds__(AX * block_rows<T>()) k_adj_init_node(KParams<T> P, const T* __restrict__ psi_pl,
                                                       const T* __restrict__ ad_pop0, AdjPlanes<T, NP> W) {
    const int x = first_x<T>() + threadIdx.x, y = first_y<T>() + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    const long long pl = P.plane;
    const long long o = P.org + (long long)y * P.pitch + x;
    const T psi = psi_pl[o];
    T lpsi = T(0);
#pragma unroll
    for (int i = 0; i < NP - 1; ++i) {
        T lemu = T(0);
#pragma unroll
        for (int p = 0; p < 9; ++p) lemu += wgt(P, p) * ad_pop0[(9 * i + p) * pl + o];
        const T l0 = ad_pop0[(9 * i) * pl + o];
        lemu -= l0;
        lpsi += W.C[i * pl + o] * l0 + P.eta[i] * W.mu[i * pl + o] * lemu;
        W.Lmu[i * pl + o] = P.eta[i] * psi * lemu;
    }
    if (NP > 2) W.Lmu[(NP - 1) * pl + o] = T(0);
    W.Lpsi[o] = lpsi;
}

// ---- objective: phase centroid J = sum_x x m(x) / sum_x m(x), m = sum_p f^i_p
template <typename T>
__global__ void __launch_bounds__(256) k_centroid_partial(KParams<T> P, const T* __restrict__ f,
                                                          double* __restrict__ part) {
    double s0 = 0.0, s1 = 0.0;
    const long long n = (long long)P.nx * P.ny;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int y = (int)(idx / P.nx), x = (int)(idx - (long long)y * P.nx);
        const long long o = P.org + (long long)y * P.pitch + x;
        double m = 0.0;
        for (int p = 0; p < 9; ++p) m += (double)f[p * P.plane + o];
        s0 += m;
        s1 += (double)x * m;
    }
    __shared__ double r0[256], r1[256];
    r0[threadIdx.x] = s0;
    r1[threadIdx.x] = s1;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            r0[threadIdx.x] += r0[threadIdx.x + w];
            r1[threadIdx.x] += r1[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = r0[0];
        part[2 * blockIdx.x + 1] = r1[0];
    }
}

// one warp; every lane sums every 32nd pair of partials, then the lanes in a
// fixed order (one thread adding all 304 pairs took 30 us)
__global__ void k_centroid_final(const double* __restrict__ part, int nblocks, double* __restrict__ out) {
    double s0 = 0.0, s1 = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += 32) {
        s0 += part[2 * b];
        s1 += part[2 * b + 1];
    }
    for (int d = 16; d > 0; d >>= 1) {
        s0 += __shfl_down_sync(0xffffffffu, s0, d);
        s1 += __shfl_down_sync(0xffffffffu, s1, d);
    }
    if (threadIdx.x != 0) return;
    out[0] = s1 / s0;   // J
    out[1] = s0;        // M
}

template <typename T>
__global__ void __launch_bounds__(AX * block_rows<T>()) k_centroid_seed(KParams<T> P, const double* __restrict__ JM,
                                                       T* __restrict__ lf) {
    const int x = first_x<T>() + threadIdx.x, y = first_y<T>() + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    const long long o = P.org + (long long)y * P.pitch + x;
    const T v = (T)(((double)x - JM[0]) / JM[1]);
#pragma unroll
    for (int p = 0; p < 9; ++p) lf[p * P.plane + o] = v;
}

template <typename T>
dim3 node_grid(int nx, int ny) {
    const unsigned bx = (nx + AX - 1) / AX, by = (ny + block_rows<T>() - 1) / block_rows<T>();
    return sizeof(T) == 8 ? dim3(by, bx) : dim3(bx, by);
}
template <typename T>
dim3 node_block() { return dim3(AX, block_rows<T>()); }

template <typename T, int NP>
cudaError_t gather_smem_attrs() {
    cudaError_t e = cudaFuncSetAttribute(k_adj_gather3<T, NP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(sizeof(T) * Ring<T>::N * AdjPlanes<T, NP>::NV));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_adj_gather2<T, NP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(sizeof(T) * Ring<T>::N * (2 * (NP - 1) + 3)));
}

template <typename T, int NP>
cudaError_t adjoint_step_n(const AdjStepArgs<T>& a, cudaStream_t s) {
    const KParams<T>& k = *a.kp;
    // the shared-memory limit is a per-device attribute: set it on every call
    const cudaError_t attrs = gather_smem_attrs<T, NP>();
    if (attrs != cudaSuccess) return attrs;
    AdjPlanes<T, NP> W = AdjPlanes<T, NP>::carve(a.scratch, k.plane);
    W.a = a.st_lag;   // lagged plane 0
    const dim3 blk = node_block<T>(), grd = node_grid<T>(k.nx, k.ny);
    cudaError_t e;
    if ((e = launch_dependent(overlaps<T>(), k_adj_fields<T, NP, false>, grd, blk, 0, s, k, a.st_pop, a.psi, a.cosf, W.C, W.mu, W.chi)) !=
            cudaSuccess ||
        (e = launch_dependent(overlaps<T>(), k_adj_node<T, NP>, grd, blk, 0, s, k, a.psi, a.st_pop, a.st_lag, a.ad_pop_in, a.ad_lag_in,
                              a.ad_pop_out, a.ad_lag_out, W)) != cudaSuccess ||
        (e = launch_dependent(overlaps<T>(), k_adj_gather3<T, NP>, grd, blk, sizeof(T) * Ring<T>::N * AdjPlanes<T, NP>::NV, s, k,
                              a.psi, W, a.ad_lag_out, a.cosf, a.dJ_dcos)) != cudaSuccess)
        return e;
    return launch_dependent(overlaps<T>(), k_adj_gather2<T, NP>, grd, blk, sizeof(T) * Ring<T>::N * (2 * (NP - 1) + 3), s, k, a.psi, W,
                            a.ad_pop_out, a.dJ_dpsi, 0);
}

template <typename T, int NP>
cudaError_t adjoint_initial_n(const AdjStepArgs<T>& a, cudaStream_t s) {
    const KParams<T>& k = *a.kp;
    // the shared-memory limit is a per-device attribute: set it on every call
    const cudaError_t attrs = gather_smem_attrs<T, NP>();
    if (attrs != cudaSuccess) return attrs;
    const AdjPlanes<T, NP> W = AdjPlanes<T, NP>::carve(a.scratch, k.plane);
    const dim3 blk = node_block<T>(), grd = node_grid<T>(k.nx, k.ny);
    cudaError_t e;
    // the caller has put C0 into W.C
    if ((e = launch_fill_ghosts<T>(W.C, NP - 1, k, s, 1, 1)) != cudaSuccess) return e;
    k_adj_fields<T, NP, true><<<grd, blk, 0, s>>>(k, nullptr, a.psi, a.cosf, W.C, W.mu, W.chi);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(W.LC, 0, sizeof(T) * k.plane * (NP - 1), s)) != cudaSuccess) return e;
    k_adj_init_node<T, NP><<<grd, blk, 0, s>>>(k, a.psi, a.ad_pop_in, W);
    k_adj_mu_node<T, NP><<<grd, blk, 0, s>>>(k, a.psi, a.cosf, W, a.dJ_dcos);
    k_adj_gather2<T, NP><<<grd, blk, sizeof(T) * Ring<T>::N * (2 * (NP - 1) + 3), s>>>(k, a.psi, W, nullptr,
                                                                              a.dJ_dpsi, 1);
    return cudaGetLastError();
}

}  // namespace

template <typename T>
size_t adjoint_scratch_planes(int N) {
    const int nm = N == 2 ? 1 : N;   // AdjPlanes::planes()
    return (size_t)(7 * (N - 1) + 5 * nm + 11 + (sizeof(T) == 8 ? 1 : 0));
}

template <typename T>
T* adjoint_c_planes(T* scratch) {
    return scratch;   // W.C is the first block of the scratch
}

#define DDCC_ADJ_DISPATCH(fn, ...)                            \
    switch (a.kp->N) {                                        \
        case 2: return fn<T, 2>(__VA_ARGS__);                 \
        case 3: return fn<T, 3>(__VA_ARGS__);                 \
        case 4: return fn<T, 4>(__VA_ARGS__);                 \
        default: return cudaErrorInvalidValue;                \
    }

template <typename T>
cudaError_t launch_adjoint_step(const AdjStepArgs<T>& a, cudaStream_t s) {
    DDCC_ADJ_DISPATCH(adjoint_step_n, a, s);
}

template <typename T>
cudaError_t launch_adjoint_initial(const AdjStepArgs<T>& a, cudaStream_t s) {
    DDCC_ADJ_DISPATCH(adjoint_initial_n, a, s);
}

template <typename T>
cudaError_t launch_centroid(const KParams<T>& kp, const T* f_phase, double* part, double* JM,
                            T* seed_f_phase, cudaStream_t s) {
    k_centroid_partial<T><<<kMassBlocks, 256, 0, s>>>(kp, f_phase, part);
    k_centroid_final<<<1, 32, 0, s>>>(part, kMassBlocks, JM);
    if (seed_f_phase)
        k_centroid_seed<T><<<node_grid<T>(kp.nx, kp.ny), node_block<T>(), 0, s>>>(kp, JM, seed_f_phase);
    return cudaGetLastError();
}

#define DDCC_ADJ_INSTANTIATE(T)                                                                      \
    template size_t adjoint_scratch_planes<T>(int);                                                  \
    template T* adjoint_c_planes<T>(T*);                                                             \
    template cudaError_t launch_adjoint_step<T>(const AdjStepArgs<T>&, cudaStream_t);                \
    template cudaError_t launch_adjoint_initial<T>(const AdjStepArgs<T>&, cudaStream_t);             \
    template cudaError_t launch_centroid<T>(const KParams<T>&, const T*, double*, double*, T*,       \
                                            cudaStream_t);

DDCC_ADJ_INSTANTIATE(float)
DDCC_ADJ_INSTANTIATE(double)

}  // namespace ddcc
