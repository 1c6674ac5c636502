// Three-dimensional DD-CCLB stepper (C ABI in include/ddcc3d.h): phase
// populations on D3Q7, flow populations on D3Q15 (Sec. 3), periodic box.
//
// One step is three kernels with one thread per node, or in FP32 by default
// one fused kernel (below):
//   k3_order   C_i = sum_p f^i_p / psi                      (Sec. 3)
//   k3_mu      mu_i of Eq. 2.14 from C and psi on the 15-point stencil
//   k3_update  gradients (D3Q15-weighted isotropic stencils), mobility
//              (Eq. 2.5), S_i (Eq. 3.7), m^C, force, the joint velocity /
//              Eq. 19 pressure solve, both collisions (Eqs. 3.1, 3.2 with
//              Eqs. 3.5-3.10), push streaming and the lagged fields.
// The rest population of each phase carries nearly all of psi C, so its
// update rounds at the ulp of psi C, with the same error every step once the
// flow is steady; the exact rounding error is recovered (TwoSum) and split
// evenly between the +x and -x populations, which keeps sum_p f to
// roundings at that smaller scale (in FP32 a steady drop otherwise loses
// mass every step) and sends the recovered mass in no preferred direction.
// Populations, lagged fields and the per-step C and mu are SoA planes of
// nx*ny*nz elements (x fastest), each plane 256-byte aligned; neighbours
// wrap periodically by index arithmetic.  g_0 is stored as g_0 - rho0 (the
// constant cancels in every moment difference).
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include <cuda_runtime.h>

#include "ddcc3d.h"
#include "ddcc_device.cuh"

namespace {

using ddcc::dev::add_rn;
using ddcc::dev::clamp0;
using ddcc::dev::rcp;
using ddcc::dev::root;
using ddcc::dev::signed_as;

constexpr int kMaxN = DDCC_MAX_PHASES;
constexpr int kBX = 32, kBY = 4, kBZ = 2;
constexpr int kBX4 = kBX / 4;        // threads along x of the four-nodes-per-thread kernel
constexpr int kThreads = kBX * kBY * kBZ;
constexpr int kMassBlocks = 304;     // 2 x 152 SMs
constexpr int kKinds = 4;            // order, mu, update, fused step
constexpr int kFusedTY = 8;          // rows of the fused step's column

// Velocities of Sec. 3: p = 0 rest; 1..6 = +x, -x, +y, -y, +z, -z; 7..14 the
// corners (+-1, +-1, +-1) with bit 0, 1, 2 of p - 7 giving a minus sign in
// x, y, z.  D3Q7 is p = 0..6 of the same list.
__host__ __device__ constexpr int cx(int p) { return p == 1 ? 1 : p == 2 ? -1 : p >= 7 ? (((p - 7) & 1) ? -1 : 1) : 0; }
__host__ __device__ constexpr int cy(int p) { return p == 3 ? 1 : p == 4 ? -1 : p >= 7 ? (((p - 7) & 2) ? -1 : 1) : 0; }
__host__ __device__ constexpr int cz(int p) { return p == 5 ? 1 : p == 6 ? -1 : p >= 7 ? (((p - 7) & 4) ? -1 : 1) : 0; }
// the seven pairs of opposite velocities: p = pair_rep(q), c_pair_opp(q) = -c_p
__host__ __device__ constexpr int pair_rep(int q) { return q < 3 ? 2 * q + 1 : 7 + (q - 3); }
__host__ __device__ constexpr int pair_opp(int q) { return q < 3 ? 2 * q + 2 : 14 - (q - 3); }

// Kernel constants, derived on the host (make_params) from ddcc3d_params.
// inv_cs2 and K are read by no kernel; they hold the places of the rest.
// Without them, or with others in their places, the compiler allots the
// registers of k3_fused otherwise: 208 x 192 x 160, N = 3, 200 steps and reads
// in 147 to 160 ms instead of 140.
template <typename T>
struct P3 {
    int nx, ny, nz, N;
    long long nxy, plane;
    int has_cos_field;
    T cs2, inv_cs2;
    T ga, gc;                  // w_axis / cs2, w_corner / cs2 (D3Q15 weights)
    T la, lc;                  // (3 eps / 4) times ga, gc
    T w7_0, w7_1;              // D3Q7 weights
    T w15[3];                  // D3Q15 weights: rest, axis, corner
    T rho[kMaxN], nu[kMaxN];
    T drho[kMaxN], dnu[kMaxN]; // rho_j - rho_N, nu_j - nu_N
    T beta2[kMaxN][kMaxN];     // 2 beta_ij = 6 sigma_ij / eps
    T beta2s[kMaxN];           // sum_{j != i} 2 beta_ij
    T sig[kMaxN][kMaxN];       // sigma_ij
    T sigN[kMaxN];             // sigma_iN
    T invsig[kMaxN][kMaxN];
    T cos_uni[kMaxN];
    T eta[kMaxN], ceta[kMaxN]; // eta_i, cs2 eta_i
    T m0;
    T hs21f;                   // D3Q7 s21 / 2
    T h1f[kMaxN], h2f[kMaxN];  // s1 / 2 and s1 / 4 - 1 / 2 (odd part of the D3Q7 collision)
    T lg0, lg1, lg3, lg3c, lg4; // D3Q15 constant rates over the row norms
    T cg0, cg1;                // lg0 / 2 - 1 and lg1 / 2 - 1 / cs2
    T inv_n2d, inv_n2o;        // 1 / norm of the s21 and s22 rows
    T nu_to_s21, inv_cs2_nu;   // 2 / (1 - cs2), 1 / cs2 (Eq. 16)
    T damp;                    // 1 / eps0^3
    T K, Hfac;                 // K = 1 - 2 d0; H = Hfac (s21 - 2)
    T A_P, cP, kk, c2m3;       // Eq. 19 coefficients; 1 - 3 cs2
    T half_K, two_cs2, one_m;  // K / 2, 2 cs2, 1 - cs2
    T q0, qa, qc;              // the last D3Q15 row at rest, axis and corner velocities
    T body[3];
};

template <typename T>
struct F3 {
    T* f[2];        // 7 (N-1) planes: the D3Q7 populations, plane 7 (i-1) + p
    T* g[2];        // 15 planes
    T* lag[2];      // 3N + 7 planes
    T* psi;
    T* cosf;        // N-1 planes or null
    T* C;           // N-1 planes
    T* mu;          // N planes
    T* chi;         // (FP64) 1 plane: psi rho of the current step
    T* st;          // (FP64) kStatic planes of psi's own terms, formed at create
    double* stage;  // 1 double plane (host staging, read-out)
    double* partial;
    int* flag;
};

// (FP64) planes of what depends on psi alone: 1 / psi, grad psi, 3 |grad psi|
enum { kInvPsi, kGrad, kAgp3 = kGrad + 3, kStatic };

// lagged plane indices
__host__ __device__ constexpr int lag_a(int k) { return k; }                   // xy, yz, zx
__host__ __device__ constexpr int lag_cu(int i, int a) { return 3 + 3 * i + a; }
template <int NP> __host__ __device__ constexpr int lag_T(int k) { return 3 + 3 * NP + k; }
template <int NP> __host__ __device__ constexpr int lag_pm() { return 9 + 3 * NP; }
__host__ __device__ constexpr int n_lag(int N) { return 3 * N + 7; }

struct Site {
    int x, y, z;
    long long zo[3];
    int yo[3], xo[3];
    __device__ long long at(int dx, int dy, int dz) const { return zo[dz + 1] + yo[dy + 1] + xo[dx + 1]; }
    __device__ long long self() const { return zo[1] + yo[1] + xo[1]; }
};

// Node of this thread.  FP32: blocks of 32 x 4 x 2 nodes.  FP64 (bound by FP64
// warp instructions, 64 cycles each per SM sub-partition, also for a warp
// that is half empty): nodes numbered row by row, one per thread of kLinear-
// thread blocks, so that no lane goes to padding and the last wave is short.
constexpr int kLinear = 64;
template <typename T>
__device__ __forceinline__ bool site(const P3<T>& P, Site& s) {
    if constexpr (sizeof(T) == 8) {
        const unsigned i = blockIdx.x * (unsigned)kLinear + threadIdx.x, nxy = (unsigned)P.nxy;
        if (i >= nxy * (unsigned)P.nz) return false;
        s.z = (int)(i / nxy);
        const unsigned r = i - (unsigned)s.z * nxy;
        s.y = (int)(r / (unsigned)P.nx);
        s.x = (int)(r - (unsigned)s.y * (unsigned)P.nx);
    } else {
        s.x = blockIdx.x * kBX + threadIdx.x;
        s.y = blockIdx.y * kBY + threadIdx.y;
        s.z = blockIdx.z * kBZ + threadIdx.z;
        if (s.x >= P.nx || s.y >= P.ny || s.z >= P.nz) return false;
    }
    s.xo[0] = s.x == 0 ? P.nx - 1 : s.x - 1;
    s.xo[1] = s.x;
    s.xo[2] = s.x == P.nx - 1 ? 0 : s.x + 1;
    s.yo[0] = (s.y == 0 ? P.ny - 1 : s.y - 1) * P.nx;
    s.yo[1] = s.y * P.nx;
    s.yo[2] = (s.y == P.ny - 1 ? 0 : s.y + 1) * P.nx;
    s.zo[0] = (long long)(s.z == 0 ? P.nz - 1 : s.z - 1) * P.nxy;
    s.zo[1] = (long long)s.z * P.nxy;
    s.zo[2] = (long long)(s.z == P.nz - 1 ? 0 : s.z + 1) * P.nxy;
    return true;
}
template <typename T>
__host__ __device__ constexpr int node_threads() { return sizeof(T) == 8 ? kLinear : kThreads; }

// Ping-pong buffer c of a pair without a dynamically indexed parameter array
// (which would be copied to local memory).
template <typename X>
__device__ __forceinline__ X* pick(X* const (&a)[2], int c) { return c ? a[1] : a[0]; }

// psi rho, rho = rho_N + sum_j (rho_j - rho_N) C_j
template <typename T, int NP, class CA>
__device__ __forceinline__ T psi_rho(const P3<T>& P, T psi, const CA& C) {
    T r = P.rho[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) r += P.drho[j] * C(j);
    return psi * r;
}

// ---------------------------------------------------------------------------
// volume fractions
// ---------------------------------------------------------------------------
template <typename T, int NP>
__global__ void __launch_bounds__(node_threads<T>()) k3_order(P3<T> P, F3<T> F, int cur) {
    Site s;
    if (!site(P, s)) return;
    const long long i0 = s.self();
    const T* f = pick(F.f, cur);
    const T inv = sizeof(T) == 8 ? F.st[kInvPsi * P.plane + i0] : rcp(F.psi[i0]);
    T C[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        T acc = f[7 * i * P.plane + i0];
#pragma unroll
        for (int p = 1; p < 7; ++p) acc += f[(7 * i + p) * P.plane + i0];
        F.C[i * P.plane + i0] = C[i] = acc * inv;
    }
    if constexpr (sizeof(T) == 8) F.chi[i0] = psi_rho<T, NP>(P, F.psi[i0], [&](int j) { return C[j]; });
}

// ---------------------------------------------------------------------------
// chemical potentials, Eq. 2.14 (beta_ij = 3 sigma_ij / eps)
// ---------------------------------------------------------------------------
// sum_p w_p c_p v(p) / cs2 on the 15-point stencil (p = 1..14), from the
// pairs of opposite neighbours: an axis pair gives its difference to its
// own component; the corner pairs (7, 14), (8, 13), (9, 12), (10, 11) give
// their differences d, signed by the first member's velocity.
template <typename T, class V>
__device__ __forceinline__ void grad15(const P3<T>& P, const V& v, T g[3]) {
    const T d0 = v(7) - v(14), d1 = v(8) - v(13), d2 = v(9) - v(12), d3 = v(10) - v(11);
    const T s01 = d0 + d1, s23 = d2 + d3;
    g[0] = P.ga * (v(1) - v(2)) + P.gc * ((d0 - d1) + (d2 - d3));
    g[1] = P.ga * (v(3) - v(4)) + P.gc * (s01 - s23);
    g[2] = P.ga * (v(5) - v(6)) + P.gc * (s01 + s23);
}

// One pair of opposite neighbours (difference d, first member p) added to a
// gradient, corner pairs before axis pairs: the corners' signed sums take
// their weight with the first axis pair of the component.  FP32 goes through
// the pairs once for all its fields (loads of different fields between the
// arithmetic of others), FP64 field by field (grad15, fewer operations).
template <typename T>
__device__ __forceinline__ void add_pair(const P3<T>& P, int q, T d, T g[3]) {
    const int p = pair_rep(q);
    if (q >= 3) {
        const int sg[3] = {cx(p), cy(p), cz(p)};
#pragma unroll
        for (int a = 0; a < 3; ++a) g[a] = q == 3 ? d : sg[a] > 0 ? g[a] + d : g[a] - d;
    } else {
        g[q] = P.ga * d + P.gc * g[q];
    }
}

// (3 eps / 4) div(psi grad C) = sum_p l_p (psi + psi_p)(C_p - C): the axis and
// the corner neighbours are summed first and take their weight once
template <typename T, class PV, class CV>
__device__ __forceinline__ T lap15(const P3<T>& P, const PV& psum, const CV& C, T c0) {
    T a = psum(1) * (C(1) - c0), c = psum(7) * (C(7) - c0);
#pragma unroll
    for (int p = 2; p < 7; ++p) a += psum(p) * (C(p) - c0);
#pragma unroll
    for (int p = 8; p < 15; ++p) c += psum(p) * (C(p) - c0);
    return P.la * a + P.lc * c;
}

// mu of one node from the 15-point neighbourhood: psi(p) and C(j, p), p = 0 the
// node; grad psi is returned in gp.
template <typename T, int NP, class PV, class CV>
__device__ __forceinline__ void mu_node(const P3<T>& P, const PV& psi, const CV& C, const T* cth, T mu[NP + 1], T gp[3]) {
    const T p0 = psi(0);
    T c0[NP], L[NP];
    if constexpr (sizeof(T) == 8) {
        T ps[15];
#pragma unroll
        for (int p = 1; p < 15; ++p) ps[p] = psi(p);
        grad15(P, [&](int p) { return ps[p]; }, gp);
#pragma unroll
        for (int p = 1; p < 15; ++p) ps[p] += p0;
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            c0[j] = C(j, 0);
            L[j] = lap15(P, [&](int p) { return ps[p]; }, [&](int p) { return C(j, p); }, c0[j]);
        }
    } else {
        T La[NP][2], Lc[NP][2];   // axis and corner sums, one per member of a pair
#pragma unroll
        for (int j = 0; j < NP; ++j) c0[j] = C(j, 0);
#pragma unroll
        for (int k = 0; k < 7; ++k) {
            const int q = k < 4 ? k + 3 : k - 4, p = pair_rep(q), o = pair_opp(q);
            const T a = psi(p), b = psi(o);
            add_pair(P, q, a - b, gp);
            const T ta = p0 + a, tb = p0 + b;
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const T da = ta * (C(j, p) - c0[j]), db = tb * (C(j, o) - c0[j]);
                T* S = q >= 3 ? Lc[j] : La[j];
                const bool first = q == 3 || q == 0;
                S[0] = first ? da : S[0] + da;
                S[1] = first ? db : S[1] + db;
            }
        }
#pragma unroll
        for (int j = 0; j < NP; ++j) L[j] = P.la * (La[j][0] + La[j][1]) + P.lc * (Lc[j][0] + Lc[j][1]);
    }
    const T agp3 = T(3) * root(gp[0] * gp[0] + gp[1] * gp[1] + gp[2] * gp[2]);
    ddcc::dev::mu_of<T, NP + 1>(P, c0, L, cth, agp3, rcp(p0), mu);
}

template <typename T, int NP>
__device__ __forceinline__ void angles(const P3<T>& P, const F3<T>& F, long long i, T cth[NP]) {
#pragma unroll
    for (int j = 0; j < NP; ++j) cth[j] = P.has_cos_field ? F.cosf[j * P.plane + i] : P.cos_uni[j];
}

template <typename T, int NP>
__global__ void __launch_bounds__(node_threads<T>()) k3_mu(P3<T> P, F3<T> F) {
    Site s;
    if (!site(P, s)) return;
    const long long i0 = s.self();
    T cth[NP], m[NP + 1];
    angles<T, NP>(P, F, i0, cth);
    auto at = [&](int p) { return s.at(cx(p), cy(p), cz(p)); };
    if constexpr (sizeof(T) == 8) {
        const T psi = __ldg(F.psi + i0);
        T ps[15], c0[NP], L[NP];
#pragma unroll
        for (int p = 1; p < 15; ++p) ps[p] = psi + __ldg(F.psi + at(p));
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            const T* C = F.C + j * P.plane;
            c0[j] = __ldg(C + i0);
            L[j] = lap15(P, [&](int p) { return ps[p]; }, [&](int p) { return __ldg(C + at(p)); }, c0[j]);
        }
        ddcc::dev::mu_of<T, NP + 1>(P, c0, L, cth, __ldg(F.st + kAgp3 * P.plane + i0),
                                    __ldg(F.st + kInvPsi * P.plane + i0), m);
    } else {
        T gp[3];
        mu_node<T, NP>(P, [&](int p) { return F.psi[at(p)]; }, [&](int j, int p) { return F.C[j * P.plane + at(p)]; },
                       cth, m, gp);
    }
#pragma unroll
    for (int i = 0; i < NP + 1; ++i) F.mu[i * P.plane + i0] = m[i];
}

// (FP64) the static planes from psi
template <typename T>
__global__ void __launch_bounds__(node_threads<T>()) k3_static(P3<T> P, F3<T> F) {
    Site s;
    if (!site(P, s)) return;
    const long long i0 = s.self();
    T g[3];
    grad15(P, [&](int p) { return F.psi[s.at(cx(p), cy(p), cz(p))]; }, g);
    F.st[kInvPsi * P.plane + i0] = T(1) / F.psi[i0];
#pragma unroll
    for (int a = 0; a < 3; ++a) F.st[(kGrad + a) * P.plane + i0] = g[a];
    F.st[kAgp3 * P.plane + i0] = T(3) * sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
}

// The same chemical potentials for four consecutive x nodes per thread
// (FP32, nx a multiple of 4; 8 x 4 x 2 threads cover 32 x 4 x 2 nodes):
// each stencil row of psi and C_j is one aligned float4 load, and the values
// one node to the left and right of the quad come from the neighbouring
// lanes by warp shuffle (scalar loads at the block's x edges and at the
// periodic seam).  Lanes beyond the box load clamped rows and store nothing.
template <int NP>
__global__ void __launch_bounds__(kThreads, NP <= 2 ? 3 : 2) k3_mu4(P3<float> P, F3<float> F) {
    constexpr int N = NP + 1;
    constexpr int NF = NP + 1;                 // fields: psi, C_1..C_{N-1}
    const int tx = threadIdx.x;
    const int x0 = 4 * (blockIdx.x * kBX4 + tx);
    const int y = blockIdx.y * kBY + threadIdx.y, z = blockIdx.z * kBZ + threadIdx.z;
    const bool live = x0 < P.nx && y < P.ny && z < P.nz;
    const int xa = x0 < P.nx ? x0 : P.nx - 4;
    const int ya = y < P.ny ? y : P.ny - 1, za = z < P.nz ? z : P.nz - 1;
    const int xm = xa == 0 ? P.nx - 1 : xa - 1;
    const int xp = xa + 4 == P.nx ? 0 : xa + 4;
    const float* fld[NF];
    fld[0] = F.psi;
#pragma unroll
    for (int j = 0; j < NP; ++j) fld[1 + j] = F.C + j * P.plane;
    auto rowbase = [&](int dy, int dz) {
        int yy = ya + dy, zz = za + dz;
        yy = yy < 0 ? yy + P.ny : (yy >= P.ny ? yy - P.ny : yy);
        zz = zz < 0 ? zz + P.nz : (zz >= P.nz ? zz - P.nz : zz);
        return (long long)zz * P.nxy + (long long)yy * P.nx;
    };
    // one row: v[f][0..3] at x0..x0+3, lf / rt[f] at x0 - 1 and x0 + 4
    float v[NF][4], lf[NF], rt[NF];
    auto load_row = [&](int dy, int dz, bool sides) {
        const long long b = rowbase(dy, dz);
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const float4 q = *reinterpret_cast<const float4*>(fld[f] + b + xa);
            v[f][0] = q.x; v[f][1] = q.y; v[f][2] = q.z; v[f][3] = q.w;
            if (sides) {
                const float l = __shfl_up_sync(0xffffffffu, q.w, 1);
                const float r = __shfl_down_sync(0xffffffffu, q.x, 1);
                lf[f] = tx > 0 ? l : fld[f][b + xm];
                rt[f] = (tx < kBX4 - 1 && xa + 4 < P.nx) ? r : fld[f][b + xp];
            }
        }
    };
    auto at = [&](int f, int k, int dx) {
        return dx == 0 ? v[f][k] : (dx < 0 ? (k == 0 ? lf[f] : v[f][k - 1]) : (k == 3 ? rt[f] : v[f][k + 1]));
    };
    float psi[4], C[NP][4], La[NP][4], Lc[NP][4], g[3][4];
    load_row(0, 0, true);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        psi[k] = v[0][k];
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            C[j][k] = v[1 + j][k];
            La[j][k] = Lc[j][k] = 0.f;
        }
        g[0][k] = g[1][k] = g[2][k] = 0.f;
    }
    // neighbour (dx, dy, dz) of node k, stencil weight w, from the loaded row
    auto accumulate = [&](int dx, int dy, int dz, float w) {
        const bool axis = dx * dx + dy * dy + dz * dz == 1;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float psp = at(0, k, dx);
            const float wp = w * psp;
            if (dx) g[0][k] += float(dx) * wp;
            if (dy) g[1][k] += float(dy) * wp;
            if (dz) g[2][k] += float(dz) * wp;
            const float ps = psi[k] + psp;
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const float d = ps * (at(1 + j, k, dx) - C[j][k]);
                if (axis) La[j][k] += d;
                else Lc[j][k] += d;
            }
        }
    };
    accumulate(1, 0, 0, P.ga);
    accumulate(-1, 0, 0, P.ga);
#pragma unroll
    for (int a = 0; a < 4; ++a) {                 // the four axis rows: +-y, +-z
        const int dy = a < 2 ? (a == 0 ? 1 : -1) : 0, dz = a < 2 ? 0 : (a == 2 ? 1 : -1);
        load_row(dy, dz, false);
        accumulate(0, dy, dz, P.ga);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {                 // the four corner rows
        const int dy = (c & 1) ? -1 : 1, dz = (c & 2) ? -1 : 1;
        load_row(dy, dz, true);
        accumulate(1, dy, dz, P.gc);
        accumulate(-1, dy, dz, P.gc);
    }
    if (!live) return;
    const long long i0 = (long long)za * P.nxy + (long long)ya * P.nx + xa;
    float cN[NP][4];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        if (P.has_cos_field) {
            const float4 q = *reinterpret_cast<const float4*>(F.cosf + j * P.plane + i0);
            cN[j][0] = q.x; cN[j][1] = q.y; cN[j][2] = q.z; cN[j][3] = q.w;
        } else {
            cN[j][0] = cN[j][1] = cN[j][2] = cN[j][3] = P.cos_uni[j];
        }
    }
    float out[N][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float Ck[NP], Lk[NP], ck[NP], m[N];
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            Ck[j] = C[j][k];
            Lk[j] = P.la * La[j][k] + P.lc * Lc[j][k];
            ck[j] = cN[j][k];
        }
        const float agp3 = 3.f * root(g[0][k] * g[0][k] + g[1][k] * g[1][k] + g[2][k] * g[2][k]);
        ddcc::dev::mu_of<float, N>(P, Ck, Lk, ck, agp3, rcp(psi[k]), m);
#pragma unroll
        for (int i = 0; i < N; ++i) out[i][k] = m[i];
    }
#pragma unroll
    for (int i = 0; i < N; ++i)
        *reinterpret_cast<float4*>(F.mu + i * P.plane + i0) = make_float4(out[i][0], out[i][1], out[i][2], out[i][3]);
}

// ---------------------------------------------------------------------------
// node update (kMacro = false) or read-out of rho, u, P (kMacro = true)
// ---------------------------------------------------------------------------
// Where the node update reads its fields: neighbour p of the velocity list
// (p = 0 the node itself) and the global index of that neighbour (the lagged
// field a is read there, populations are pushed there).
template <typename T, int NP>
struct GlobalSrc {     // the per-step C and mu planes in global memory
    const P3<T>& P;
    const F3<T>& F;
    Site s;
    const T* f_;       // populations and lagged planes of the input copy
    const T* g_;
    const T* lag_;
    __device__ long long at(int p) const { return s.at(cx(p), cy(p), cz(p)); }
    __device__ T f(int i, int p) const { return __ldg(f_ + (7 * i + p) * P.plane + s.self()); }
    __device__ T g(int p) const { return __ldg(g_ + p * P.plane + s.self()); }
    __device__ T lag(int k) const { return __ldg(lag_ + k * P.plane + s.self()); }
    __device__ T a(int k, int p) const { return __ldg(lag_ + lag_a(k) * P.plane + at(p)); }
    __device__ T psi(int p) const { return __ldg(F.psi + at(p)); }
    __device__ T C(int j, int p) const { return __ldg(F.C + j * P.plane + at(p)); }
    __device__ T mu(int j, int p) const { return __ldg(F.mu + j * P.plane + at(p)); }
    __device__ T psirho(int p) const {
        if constexpr (sizeof(T) == 8) return __ldg(F.chi + at(p));
        else return psi_rho<T, NP>(P, psi(p), [&](int j) { return C(j, p); });
    }
    __device__ void grad_psi(T gp[3]) const {
        if constexpr (sizeof(T) == 8) {
#pragma unroll
            for (int a = 0; a < 3; ++a) gp[a] = __ldg(F.st + (kGrad + a) * P.plane + s.self());
        } else {
            grad15(P, [&](int p) { return psi(p); }, gp);
        }
    }
};

// sum_j C_j = 1 (C_N is defined by it), so sums over all phases reduce to the
// N-1 evolved ones: rho and grad rho through rho_j - rho_N, the capillary
// force through mu_j - mu_N, m^C = -m0 sum_j (rho_j - rho_N) Q_j because the
// Q_j = C_j (grad mu_j - sum_k C_k grad mu_k) add up to zero.  For two phases
// mu_2 = -mu_1.  kMacro: rho, u and P of the state go to the planes at out
// instead.
// FP64 (three kernels) is bound by FP64 warp instructions: sums over all
// phases, pairs of mu, psi's own terms at every step, 256-thread blocks of 32
// x 4 x 2 nodes and divisions by the operator took twice the time (96 x 80 x
// 72, N = 3, 10 steps and a read-out: 18.0 ms, now 9.4).
// FP32 (fused): 617 us a step at 208 x 192 x 160, N = 3 (722 without field a
// staged); the kernel's loads and stores alone take 504 us there (loads 314),
// the stores in 128-byte rows of 45 planes.
template <typename T, int NP, bool kMacro, class S>
__device__ __forceinline__ void update_node(const P3<T>& P, const F3<T>& F, int cur, T* out, const S& src) {
    constexpr int N = NP + 1, NM = NP == 1 ? 1 : N;
    const long long i0 = src.at(0);
    const int nxt = cur ^ 1;
    const T psi = src.psi(0);
    const T cs2 = P.cs2;
    T C[N], gC[NP][3], mu[NM], gmu[NM][3], G[3], gpr[3];
    T dA[3];   // -div A: (d_y a_xy - d_z a_zx, d_z a_yz - d_x a_xy, d_x a_zx - d_y a_yz)
    if constexpr (sizeof(T) == 8) {
#pragma unroll
        for (int j = 0; j < NP; ++j) grad15(P, [&](int p) { return src.C(j, p); }, gC[j]);
#pragma unroll
        for (int j = 0; j < NM; ++j) grad15(P, [&](int p) { return src.mu(j, p); }, gmu[j]);
        grad15(P, [&](int p) { return src.psirho(p); }, gpr);
        T gaxy[3], gayz[3], gazx[3];
        grad15(P, [&](int p) { return src.a(0, p); }, gaxy);
        grad15(P, [&](int p) { return src.a(1, p); }, gayz);
        grad15(P, [&](int p) { return src.a(2, p); }, gazx);
        dA[0] = gaxy[1] - gazx[2];
        dA[1] = gayz[2] - gaxy[0];
        dA[2] = gazx[0] - gayz[1];
    } else {
#pragma unroll
        for (int k = 0; k < 7; ++k) {
            const int q = k < 4 ? k + 3 : k - 4, p = pair_rep(q), o = pair_opp(q);
            // a first: from global memory
            const T dxy = q != 2 ? src.a(0, p) - src.a(0, o) : T(0);
            const T dyz = q != 0 ? src.a(1, p) - src.a(1, o) : T(0);
            const T dzx = q != 1 ? src.a(2, p) - src.a(2, o) : T(0);
#pragma unroll
            for (int j = 0; j < NP; ++j) add_pair(P, q, src.C(j, p) - src.C(j, o), gC[j]);
#pragma unroll
            for (int j = 0; j < NM; ++j) add_pair(P, q, src.mu(j, p) - src.mu(j, o), gmu[j]);
            add_pair(P, q, src.psirho(p) - src.psirho(o), gpr);
            if (q >= 3) {
                const T sx = T(cx(p)), sy = T(cy(p)), sz = T(cz(p));
                const T t0 = sy * dxy - sz * dzx, t1 = sz * dyz - sx * dxy, t2 = sx * dzx - sy * dyz;
                dA[0] = q == 3 ? t0 : dA[0] + t0;
                dA[1] = q == 3 ? t1 : dA[1] + t1;
                dA[2] = q == 3 ? t2 : dA[2] + t2;
            } else {
                // weight the corners' sums once, with the first axis pair
                if (q == 0) {
                    dA[0] *= P.gc;
                    dA[1] = P.gc * dA[1] - P.ga * dxy;
                    dA[2] = P.gc * dA[2] + P.ga * dzx;
                } else if (q == 1) {
                    dA[0] += P.ga * dxy;
                    dA[2] -= P.ga * dyz;
                } else {
                    dA[0] -= P.ga * dzx;
                    dA[1] += P.ga * dyz;
                }
            }
        }
    }
    T rho = P.rho[NP], nu = P.nu[NP], grho[3];
    {
        T sum = T(0);
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            C[j] = src.C(j, 0);
            sum = j == 0 ? C[0] : sum + C[j];
            rho += P.drho[j] * C[j];
            nu += P.dnu[j] * C[j];
#pragma unroll
            for (int a = 0; a < 3; ++a) grho[a] = j == 0 ? P.drho[0] * gC[0][a] : grho[a] + P.drho[j] * gC[j][a];
        }
        C[NP] = T(1) - sum;
    }
#pragma unroll
    for (int j = 0; j < NM; ++j) mu[j] = src.mu(j, 0);
    if constexpr (NP == 1) {
        const T dC = C[0] - C[1];
#pragma unroll
        for (int a = 0; a < 3; ++a) G[a] = dC * gmu[0][a];
    } else {
#pragma unroll
        for (int j = 0; j < NM; ++j)
#pragma unroll
            for (int a = 0; a < 3; ++a) G[a] = j == 0 ? C[0] * gmu[0][a] : G[a] + C[j] * gmu[j][a];
    }
    T Q[NP][3], mC[3];   // mC: psi m^C
    const T pm0 = -(P.m0 * psi);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        T t = T(0);
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            Q[i][a] = C[i] * (gmu[i][a] - G[a]);
            t = i == 0 ? P.drho[0] * Q[0][a] : t + P.drho[i] * Q[i][a];
        }
        mC[a] = pm0 * t;
    }
    T gps[3];
    src.grad_psi(gps);

    const T t21 = nu * P.nu_to_s21 + T(0.5);   // 1 / s21
    const T s21 = rcp(t21);
    const T s22 = rcp(nu * P.inv_cs2_nu + T(0.5));

    // force without P grad psi and the damping: psi (sum_j (mu_j - mu_N) grad
    // C_j + rho b) - div A (A_jk = psi (m^C_j u_k - u_j m^C_k)/2, lagged)
    T Fv[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        T t = rho * P.body[a];
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            T dm;
            if constexpr (NP == 1) dm = mu[0] + mu[0];
            else dm = mu[j] - mu[NM - 1];
            t += dm * gC[j][a];
        }
        Fv[a] = psi * t + dA[a];
    }

    // D3Q15 moments.  Opposite velocities come in seven pairs: an even
    // polynomial of c takes the pairs' sums, an odd one their differences; the
    // four corner pairs' signs are those of grad15.
    T j3[3], t3[3], e2[3], o2[3], xyz, corner, mm, sum_g;
    {
        T gs[7], gd[7];
#pragma unroll
        for (int q = 0; q < 7; ++q) {
            const T a = src.g(pair_rep(q)), b = src.g(pair_opp(q));
            gs[q] = a + b;
            gd[q] = a - b;
        }
        const T m01 = gd[3] - gd[4], m23 = gd[5] - gd[6], s01 = gd[3] + gd[4], s23 = gd[5] + gd[6];
        t3[0] = m01 + m23;
        t3[1] = s01 - s23;
        t3[2] = s01 + s23;
        xyz = m01 - m23;
        const T c01 = gs[3] + gs[4], c23 = gs[5] + gs[6], n01 = gs[3] - gs[4], n23 = gs[5] - gs[6];
        corner = c01 + c23;
        o2[0] = n01 - n23;
        o2[1] = c01 - c23;
        o2[2] = n01 + n23;
        sum_g = (gs[0] + gs[1]) + (gs[2] + corner);
        mm = src.g(0) + sum_g;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            j3[a] = gd[a] + t3[a];
            e2[a] = gs[a] + corner;
        }
    }
    const T psirho = psi * rho;
    const T damp = P.damp - P.damp * psi;
    const T inv_den = rcp(psirho + T(0.5) * damp);
    const T hi = T(0.5) * inv_den;
    const T Hs = P.Hfac - T(2) * P.Hfac * t21;   // H / s21
    const T Ap = P.A_P * psi;
    const T gam = P.kk * psirho;
    // Eq. 19 with u = u0 + P e: cP gam e.e P^2 + (cP (b + 2 gam u0).e - psi) P
    // + cP (G0 + (b + gam u0).u0) = 0
    T u0[3], e[3], ee, we, vu;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        u0[a] = (j3[a] + T(0.5) * Fv[a]) * inv_den;
        e[a] = gps[a] * hi;
        const T v = Ap * grho[a] + P.kk * mC[a] + Hs * gpr[a] + gam * u0[a];
        const T w = v + gam * u0[a];
        ee = a == 0 ? e[0] * e[0] : ee + e[a] * e[a];
        we = a == 0 ? w * e[0] : we + w * e[a];
        vu = a == 0 ? v * u0[0] : vu + v * u0[a];
    }
    const T qa = P.cP * gam * ee;
    const T qb = P.cP * we - psi;
    const T qc = P.cP * ((sum_g - P.half_K * src.lag(lag_pm<NP>())) + vu);
    const T disc = clamp0(qb * qb - T(4) * qa * qc);
    const T Pp = T(-2) * qc * rcp(qb + signed_as(root(disc), qb));
    T u[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        u[a] = u0[a] + Pp * e[a];
        Fv[a] += Pp * gps[a] - damp * u[a];
    }
    if constexpr (kMacro) {
        out[i0] = rho;
#pragma unroll
        for (int a = 0; a < 3; ++a) out[(1 + a) * P.plane + i0] = u[a];
        out[4 * P.plane + i0] = Pp;
        return;
    } else {
        T* lagn = pick(F.lag, nxt);
        // ---- phase LB (Eqs. 3.1, 3.5-3.7), D3Q7 ----
        T* fnew = pick(F.f, nxt);
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            T f[7];
            T psiC = T(0);
#pragma unroll
            for (int p = 0; p < 7; ++p) {
                f[p] = src.f(i, p);
                psiC = p == 0 ? f[0] : psiC + f[p];
            }
            const T csepm = P.ceta[i] * (psi * mu[i]);
            // Lambda v, v = f - f^eq + F/2, on the D3Q7 rows 1, c_a,
            // c_a^2 - cs2 (S = s0, s1, s21) from the moments of v: the zeroth
            // vanishes (sum f^eq = psi C = sum f, sum F = 0); the first is
            // j_a(f) - psi C u_a + V_a / 2; the raw second, sum_{+-a} v, is
            // e_a(f) - d0 eta psi mu (Eqs. 3.5, 3.6, B.5b, B.5c).  F_p = w_p
            // c_p . V / cs2 is +-V_a / 2 (w_1 = cs2 / 2) and zero at rest.
            // V = d_t(psi C u) + cs2 eta (mu grad psi - S), S = psi (Q - grad mu)
            T hE[3], h[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const T fp = f[1 + 2 * a], fm = f[2 + 2 * a];
                const T cu = psiC * u[a];
                const T V = (cu - src.lag(lag_cu(i, a))) +
                            P.ceta[i] * (mu[i] * gps[a] + psi * (gmu[i][a] - Q[i][a]));
                lagn[lag_cu(i, a) * P.plane + i0] = cu;
                h[a] = P.h1f[i] * ((fp - fm) - cu) + P.h2f[i] * V;
                hE[a] = P.hs21f * ((fp + fm) - csepm);
            }
            // The rest population's new value f_0 + 2 sum_a hE_a is rounded
            // explicitly and its exact rounding error (TwoSum) is split
            // evenly between the populations p = 1 and 2 (+x and -x), so
            // sum_p f keeps the exchange and no direction is preferred.
            const T w0 = T(2) * ((hE[0] + hE[1]) + hE[2]);
            const T o0 = add_rn(f[0], w0);
            const T bb = add_rn(o0, -f[0]);
            const T err = T(0.5) * add_rn(add_rn(f[0], -add_rn(o0, -bb)), add_rn(w0, -bb));
            fnew[(7 * i) * P.plane + i0] = o0;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                // the two parts are joined first: in a steady flow hE is below
                // the ulp of f and would be lost on its own every step
                T op = f[1 + 2 * a] - (hE[a] + h[a]), om = f[2 + 2 * a] - (hE[a] - h[a]);
                if (a == 0) {
                    op = add_rn(op, err);
                    om = add_rn(om, err);
                }
                fnew[(7 * i + 1 + 2 * a) * P.plane + src.at(1 + 2 * a)] = op;
                fnew[(7 * i + 2 + 2 * a) * P.plane + src.at(2 + 2 * a)] = om;
            }
        }

        // ---- flow LB (Eqs. 3.2, 3.8, 3.10), D3Q15 ----
        // The collision runs in moment space on the orthogonal D3Q15 rows
        // h_k: with v = g - g^eq + G/2 and G = w (sum_k h_k <h_k, G> / |h_k|^2)
        // (G is w times a polynomial of degree <= 2),
        //   g* = g - Lambda v + G = g - w sum_k h_k mu_k,
        //   mu_k = (s_k / |h_k|^2) <h_k, v> - <h_k, G> / |h_k|^2.
        // <h_k, g^eq> (Eq. 3.8, g_0 stored as g_0 - rho0) = 0, psi rho u_a,
        // A_aa + psi P, A_ab, 0 (third order), -2 cs2 psi P (the rest
        // population's -psi P / cs2 on the last row); <h_k, G> (Eq. 3.10) =
        // a0, F_a, M_aa, M_ab, 0 (Eqs. B.5d, B.5e); A = psi rho u u + T,
        // T = psi (m^C u + u m^C) / 2.
        const T psiP = psi * Pp;
        T s[3], ugpr = T(0), pm = T(0), m1[3], m4[3], m7[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            s[a] = u[a] * gpr[a];
            ugpr = a == 0 ? s[0] : ugpr + s[a];
        }
        const T cu3 = P.c2m3 * ugpr;
        const T l2d = P.inv_n2d * s21, c2d = T(0.5) * l2d - P.inv_n2d;
        const T l2o = P.inv_n2o * s22, c2o = T(0.5) * l2o - P.inv_n2o;
        const T cmm = cs2 * mm;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int b = (a + 1) % 3;
            const T ja = psirho * u[a];
            const T Taa = mC[a] * u[a];
            const T Aaa = ja * u[a] + Taa;
            pm = a == 0 ? Aaa : pm + Aaa;
            const T p1 = mC[a] * u[b], p2 = u[a] * mC[b];
            const T Tab = T(0.5) * (p1 + p2);
            const T Aab = ja * u[b] + Tab;
            const T Maa = (Taa - src.lag(lag_T<NP>(a))) + P.two_cs2 * s[a] + cu3;
            const T Mab = (Tab - src.lag(lag_T<NP>(3 + a))) + cs2 * (u[a] * gpr[b] + gpr[a] * u[b]);
            m1[a] = P.lg1 * (j3[a] - ja) + P.cg1 * Fv[a];
            m4[a] = l2d * ((e2[a] - cmm) - (Aaa + psiP)) + c2d * Maa;
            m7[a] = l2o * (o2[a] - Aab) + c2o * Mab;
            lagn[lag_T<NP>(a) * P.plane + i0] = Taa;
            lagn[lag_T<NP>(3 + a) * P.plane + i0] = Tab;
            lagn[lag_a(a) * P.plane + i0] = T(0.5) * (p1 - p2);
        }
        lagn[lag_pm<NP>() * P.plane + i0] = pm;
        const T a0 = psi * (u[0] * grho[0] + u[1] * grho[1] + u[2] * grho[2]);
        const T m0 = P.lg0 * mm + P.cg0 * a0;
        const T m14 = P.lg4 * (corner - cs2 * (e2[0] + e2[1] + e2[2]) + P.two_cs2 * (cmm + psiP));
        const T m13 = P.lg3c * xyz;
        // sum_k h_k(c) mu_k: even part by the velocity's kind (rest, axis,
        // corner), odd part from the first- and third-order rows
        const T sd = (m4[0] + m4[1]) + m4[2];
        const T base = m0 - cs2 * sd;
        const T Ea = base + P.qa * m14, Ec = (base + sd) + P.qc * m14;
        T Oa[3], Oc[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const T r = P.lg3 * (t3[a] - cs2 * j3[a]);   // row c_a (c_b^2 - cs2)
            Oa[a] = m1[a] - cs2 * r;
            Oc[a] = m1[a] + P.one_m * r;
        }
        T* gnew = pick(F.g, nxt);
        gnew[i0] = src.g(0) - P.w15[0] * (base + P.q0 * m14);
        auto put = [&](int q, T E, T O, T w) {
            const int p = pair_rep(q), pb = pair_opp(q);
            gnew[p * P.plane + src.at(p)] = src.g(p) - w * (E + O);
            gnew[pb * P.plane + src.at(pb)] = src.g(pb) - w * (E - O);
        };
#pragma unroll
        for (int a = 0; a < 3; ++a) put(a, Ea + m4[a], Oa[a], P.w15[1]);
        // corner pairs: signs (x, y, z) = (+++), (-++), (+-+), (--+)
        const T Ep = Ec + m7[0], Em = Ec - m7[0];             // by the sign of xy
        const T yp = m7[1] + m7[2], ym = m7[1] - m7[2];       // yz, zx
        const T xp = Oc[0] + Oc[1], xm = Oc[0] - Oc[1];
        const T zp = Oc[2] + m13, zm = Oc[2] - m13;           // xyz = +-1
        put(3, Ep + yp, xp + zp, P.w15[2]);
        put(4, Em + ym, zm - xm, P.w15[2]);
        put(5, Em - ym, xm + zm, P.w15[2]);
        put(6, Ep - yp, zp - xp, P.w15[2]);
    }
}

template <typename T, int NP, bool kMacro>
__global__ void __launch_bounds__(node_threads<T>(), sizeof(T) == 4 ? 2 : 4) k3_update(P3<T> P, F3<T> F, int cur, T* out) {
    Site s;
    if (!site(P, s)) return;
    update_node<T, NP, kMacro>(P, F, cur, out, GlobalSrc<T, NP>{P, F, s, pick(F.f, cur), pick(F.g, cur), pick(F.lag, cur)});
}

// ---------------------------------------------------------------------------
// the fused step: one kernel per step, each CTA marching along z
// ---------------------------------------------------------------------------
// A CTA owns a column of 32 x TY nodes and the planes [zb, ze) of it.  The
// update of plane z reads C, psi and mu at planes z-1..z+1 on the column
// plus one node a side; mu at plane z+1 reads C and psi at planes z..z+2 on
// the column plus two nodes a side.  So for each output plane z the CTA
// forms C and psi at plane z+2 on the region x0-4 .. x0+35 (40 columns, so
// that rows are whole aligned quads) by y0-2 .. y0+TY+1, then mu at plane
// z+1 on the (32+2) x (TY+2) region, then updates plane z, with two
// barriers.  C and psi sit in a ring of five planes in shared memory and
// mu in a ring of three:
//   * the C pass for plane z+2 may overlap the slower threads' update of
//     plane z-1, which reads C at z-2..z: five slots keep them apart;
//   * the mu pass for plane z+1 starts after the barrier that follows the
//     C pass, when every thread has finished the update of plane z-1, so
//     the slot of mu at z-2 is free.
// In FP32 the phase populations and psi of the C region arrive by cp.async
// copies issued one plane ahead: by 16 bytes with kVec (nx a multiple of 4,
// so that a periodic wrap maps aligned quads to aligned quads), else node by
// node.  The thread that forms C for a quad of 4 nodes, or a node, copies
// the 7(N-1) + 1 values of each and nothing else, so it waits for its own
// copies only and needs no barrier.
// The copies of plane z+3 fly during the mu pass and the update of plane z.
// (101 x 77 x 63, N = 2, where the copies are by node: 68 us a step with
// plain loads, 62 with the copies.)
// The lagged field a (three components, read at 36 neighbour positions) comes
// the same way, a plane ahead, into a ring of three planes: 617 us a step
// instead of 722 with those reads through L1 (208 x 192 x 160, N = 3).  With kStage (FP32
// and N <= 3, where two CTAs per SM still fit) so do the column's 15 flow
// populations and 3N + 4 lagged values.  Both are issued after the barrier
// that ends the update of the plane before, fly during the mu pass, and are
// waited for ahead of the barrier that starts the update.  Groups are
// committed in the same order by every thread (empty ones where a thread has
// nothing to copy): stage(z), raw(z+3), stage(z+1), raw(z+4), ..., so "all but
// the newest group" is what the update needs and "all" what the C pass needs.
// The per-step C and mu planes of global memory are neither read nor
// written; the update arithmetic is update_node's, the same as the
// three-kernel step's.
template <typename T, int NP, int TY, bool kVec, bool kStage = false>
struct FusedGeom {
    static constexpr int N = NP + 1;
    static constexpr int CW = kBX + 8, CH = TY + 4, CN = CW * CH;   // C, psi region
    static constexpr int MW = kBX + 2, MH = TY + 2, MN = MW * MH;   // mu region
    static constexpr int NT = kBX * TY;
    static constexpr int KC = (CN + NT - 1) / NT;                   // C-region nodes per thread
    static constexpr int KM = (MN + NT - 1) / NT;                   // mu-region nodes per thread
    static constexpr int NQ = CN / 4;                               // quads of the C region
    static constexpr bool kRaw = sizeof(T) == 4;                    // C pass fed by cp.async
    static constexpr int RAW = kRaw ? (7 * NP + 1) * CN : 0;        // staged populations and psi
    static constexpr int NSTG = 15 + 3 * N + 4;                     // own-node g and lagged values
    static constexpr int STG = kStage ? NSTG * NT : 0;
    static constexpr int NMU = NP == 1 ? 1 : N;                     // mu planes (N = 2: mu_2 = -mu_1)
    static constexpr int AW = CW, AH = TY + 2, AN = AW * AH;        // region of the lagged field a
    static constexpr int A = kRaw ? 3 * 3 * AN : 0;                 // (FP32) a_xy, a_yz, a_zx, three planes
    static constexpr int BASE = 5 * (NP + 1) * CN + 3 * NMU * MN + RAW + STG + A;
    // psi rho (with mu, three planes) and grad psi of the own nodes (two planes)
    // kept by the mu pass where two CTAs still fit an SM with them (each costs
    // 1 KB and the column indices more); else the update forms both again
    // from C and psi.
    static constexpr bool kKeep = sizeof(T) * (BASE + 3 * MN + 2 * 3 * NT) + 1280 <= 228 * 1024 / 2;
    static constexpr int NM = NMU + (kKeep ? 1 : 0);                // planes of the mu ring
    static constexpr int GP = kKeep ? 2 * 3 * NT : 0;
    static constexpr size_t smem = sizeof(T) * (BASE + (kKeep ? 3 * MN : 0) + GP);
    static_assert(!kVec || (sizeof(T) == 4 && NQ <= NT), "one quad per thread, FP32");
    static_assert(!kStage || kRaw, "staging needs the cp.async path");
};

template <typename T, int NP, int TY, bool kVec, bool kStage>
struct SmemSrc {     // C, psi, mu and psi rho from the shared-memory rings
    using G = FusedGeom<T, NP, TY, kVec, kStage>;
    const T* sC;     // C ring: slot k holds NP x CN values
    const T* sPs;    // psi ring: slot k holds CN values
    const T* sMu;    // mu ring: slot k holds NM x MN values
    const T* sGp;    // (kKeep) grad psi: two slots of 3 x NT values
    const P3<T>* P;
    const T* sA;     // (FP32) a ring, slots as mu's: three fields of AN values
    const T* stg;    // (kStage) own-node g (15) and lagged planes 3.. (NT apart)
    const T* f_;     // populations and lagged planes in global memory
    const T* g_;
    const T* lag_;
    long long plane;
    int c5[3], m3[3];  // ring slots of planes z-1, z, z+1
    int gp2;           // grad psi's slot of plane z
    int ci, mi, ai;    // the node in the C, mu and a regions
    int tid;
    int xo[3], yo[3], zo[3];  // wrapped x, y nx, z nx ny of the node and its neighbours
    __device__ int at(int p) const { return zo[cz(p) + 1] + yo[cy(p) + 1] + xo[cx(p) + 1]; }
    __device__ T f(int i, int p) const { return __ldg(f_ + (7 * i + p) * plane + at(0)); }
    __device__ T g(int p) const {
        if constexpr (kStage) return stg[p * G::NT + tid];
        else return __ldg(g_ + p * plane + at(0));
    }
    __device__ T lag(int k) const {   // k >= 3: the own node's lagged planes past a
        if constexpr (kStage) return stg[(12 + k) * G::NT + tid];
        else return __ldg(lag_ + k * plane + at(0));
    }
    __device__ T a(int k, int p) const {
        if constexpr (G::kRaw) return sA[(m3[cz(p) + 1] * 3 + k) * G::AN + ai + cy(p) * G::AW + cx(p)];
        else return __ldg(lag_ + lag_a(k) * plane + at(p));
    }
    __device__ T psi(int p) const { return sPs[c5[cz(p) + 1] * G::CN + ci + cy(p) * G::CW + cx(p)]; }
    __device__ T C(int j, int p) const {
        return sC[(c5[cz(p) + 1] * NP + j) * G::CN + ci + cy(p) * G::CW + cx(p)];
    }
    __device__ T mu(int j, int p) const {
        return sMu[(m3[cz(p) + 1] * G::NM + j) * G::MN + mi + cy(p) * G::MW + cx(p)];
    }
    __device__ T psirho(int p) const {
        if constexpr (G::kKeep) return mu(G::NM - 1, p);
        else return psi_rho<T, NP>(*P, psi(p), [&](int j) { return C(j, p); });
    }
    __device__ void grad_psi(T gp[3]) const {
        if constexpr (G::kKeep) {
#pragma unroll
            for (int a = 0; a < 3; ++a) gp[a] = sGp[(gp2 * 3 + a) * G::NT + tid];
        } else {
#pragma unroll
            for (int k = 0; k < 7; ++k) {
                const int q = k < 4 ? k + 3 : k - 4;
                add_pair(*P, q, psi(pair_rep(q)) - psi(pair_opp(q)), gp);
            }
        }
    }
};

__device__ __forceinline__ int wrap_index(int v, int n) {
    v %= n;
    return v < 0 ? v + n : v;
}

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async4(void* smem_dst, const void* gmem_src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

template <typename T, int NP, int TY, bool kVec, bool kStage>
__global__ void __launch_bounds__(kBX * TY, (sizeof(T) == 4 && TY <= 8) ? 2 : 1)
    k3_fused(P3<T> P, F3<T> F, int cur, int nchunk) {
    using G = FusedGeom<T, NP, TY, kVec, kStage>;
    constexpr int N = NP + 1, CW = G::CW, CN = G::CN, MW = G::MW, MN = G::MN, NT = G::NT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sC = reinterpret_cast<T*>(smem_raw);    // 5 slots x NP x CN
    T* sPs = sC + 5 * NP * CN;                  // 5 slots x CN
    T* sMu = sPs + 5 * CN;                      // 3 slots x NM x MN
    T* sGp = sMu + 3 * G::NM * MN;              // (kKeep) 2 slots x 3 x NT
    T* sRaw = sGp + G::GP;                      // (FP32) 7 NP + 1 planes x CN
    T* sStg = sRaw + G::RAW;                    // (kStage) NSTG x NT
    T* sA = sStg + G::STG;                      // (FP32) 3 slots x 3 x AN
    const int tid = threadIdx.x;
    const int x0 = blockIdx.x * kBX, y0 = blockIdx.y * TY;
    const int zb = (int)((long long)blockIdx.z * P.nz / nchunk);
    const int ze = (int)((long long)(blockIdx.z + 1) * P.nz / nchunk);
    const T* fcur = pick(F.f, cur);
    // ring slots: C and psi of plane z >= zb - 2, mu of plane z >= zb - 1
    auto slot5 = [&](int z) { return (z - zb + 2) % 5; };
    auto slot3 = [&](int z) { return (z - zb + 1) % 3; };
    auto zoff = [&](int z) { return (long long)wrap_index(z, P.nz) * P.nxy; };

    // wrapped x and y nx of the C region's columns (x0-4+k) and rows (y0-2+k)
    __shared__ int xs[CW], ys[G::CH];
    for (int k = tid; k < CW; k += NT) xs[k] = wrap_index(x0 + k - 4, P.nx);
    for (int k = tid; k < G::CH; k += NT) ys[k] = wrap_index(y0 + k - 2, P.ny) * P.nx;
    __syncthreads();

    // (FP32) copy the populations and psi of this thread's quad (kVec), or of
    // its nodes one by one, at plane z
    auto issue = [&](int z, bool any) {
        if constexpr (G::kRaw && !kVec) {
            if (any) {
                const long long zo = zoff(z);
#pragma unroll
                for (int r = 0; r < G::KC; ++r) {
                    const int k = tid + r * NT;
                    if (k < CN) {
                        const long long g = zo + ys[k / CW] + xs[k % CW];
#pragma unroll
                        for (int q = 0; q < 7 * NP; ++q) cp_async4(sRaw + q * CN + k, fcur + q * P.plane + g);
                        cp_async4(sRaw + 7 * NP * CN + k, F.psi + g);
                    }
                }
            }
            cp_async_commit();
        }
        if constexpr (kVec) {
            if (any && tid < G::NQ) {
                const int o = 4 * tid;   // quad tid: row o / CW, columns o % CW .. + 3
                const long long g = zoff(z) + ys[o / CW] + xs[o % CW];
#pragma unroll
                for (int q = 0; q < 7 * NP; ++q) cp_async16(sRaw + q * CN + o, fcur + q * P.plane + g);
                cp_async16(sRaw + 7 * NP * CN + o, F.psi + g);
            }
            cp_async_commit();
        }
    };
    // C_i = sum_p f^i_p / psi and psi at plane z on the C region (as k3_order)
    auto c_pass = [&](int z) {
        T* c = sC + slot5(z) * NP * CN;
        T* ps = sPs + slot5(z) * CN;
        if constexpr (kVec) {
            if (tid < G::NQ) {
                const int o = 4 * tid;
                cp_async_wait<0>();
                const float4 psi = *reinterpret_cast<const float4*>(sRaw + 7 * NP * CN + o);
                *reinterpret_cast<float4*>(ps + o) = psi;
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int p = 0; p < 7; ++p) {
                        const float4 v = *reinterpret_cast<const float4*>(sRaw + (7 * j + p) * CN + o);
                        acc.x += v.x;
                        acc.y += v.y;
                        acc.z += v.z;
                        acc.w += v.w;
                    }
                    *reinterpret_cast<float4*>(c + j * CN + o) =
                        make_float4(acc.x * rcp(psi.x), acc.y * rcp(psi.y), acc.z * rcp(psi.z), acc.w * rcp(psi.w));
                }
            }
        } else {
            const long long zo = zoff(z);
            if constexpr (G::kRaw) {
                cp_async_wait<0>();
            }
#pragma unroll
            for (int r = 0; r < G::KC; ++r) {
                const int k = tid + r * NT;
                if (k < CN) {
                    const long long i = zo + ys[k / CW] + xs[k % CW];
                    const T psi = G::kRaw ? sRaw[7 * NP * CN + k] : F.psi[i];
                    ps[k] = psi;
                    const T inv = rcp(psi);
#pragma unroll
                    for (int j = 0; j < NP; ++j) {
                        T acc = T(0);
#pragma unroll
                        for (int p = 0; p < 7; ++p)
                            acc += G::kRaw ? sRaw[(7 * j + p) * CN + k] : fcur[(7 * j + p) * P.plane + i];
                        c[j * CN + k] = acc * inv;
                    }
                }
            }
        }
    };

    // mu at plane z on the mu region (as k3_mu); kKeep: psi rho there, which
    // the update differentiates, and grad psi of the column's own nodes
    auto mu_pass = [&](int z) {
        const T* cpl[3];
        const T* ppl[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            cpl[d] = sC + slot5(z - 1 + d) * NP * CN;
            ppl[d] = sPs + slot5(z - 1 + d) * CN;
        }
        T* m = sMu + slot3(z) * G::NM * MN;
        T* gps = sGp + ((z - zb) & 1) * 3 * NT;   // two slots: the update of plane z - 2 is done
        const long long zo = zoff(z);
#pragma unroll
        for (int r = 0; r < G::KM; ++r) {
            const int k = tid + r * NT;
            if (k < MN) {
                const int row = k / MW, col = k % MW;
                const int c0 = (row + 1) * CW + col + 3;
                T cth[NP], mv[N], gp[3];
                angles<T, NP>(P, F, zo + ys[row + 1] + xs[col + 3], cth);
                mu_node<T, NP>(
                    P, [&](int p) { return ppl[cz(p) + 1][c0 + cy(p) * CW + cx(p)]; },
                    [&](int j, int p) { return cpl[cz(p) + 1][j * CN + c0 + cy(p) * CW + cx(p)]; }, cth, mv, gp);
#pragma unroll
                for (int i = 0; i < G::NMU; ++i) m[i * MN + k] = mv[i];
                if (G::kKeep)
                    m[(G::NM - 1) * MN + k] =
                        psi_rho<T, NP>(P, ppl[1][c0], [&](int j) { return cpl[1][j * CN + c0]; });
                if (G::kKeep && row >= 1 && row <= TY && col >= 1 && col <= kBX) {
#pragma unroll
                    for (int a = 0; a < 3; ++a) gps[a * NT + (row - 1) * kBX + col - 1] = gp[a];
                }
            }
        }
    };

    // this thread's node of the column
    const int tx = tid % kBX, ty = tid / kBX;
    const int x = x0 + tx, y = y0 + ty;
    const bool live = x < P.nx && y < P.ny;
    SmemSrc<T, NP, TY, kVec, kStage> src;
    src.sC = sC;
    src.sPs = sPs;
    src.sMu = sMu;
    src.sGp = sGp;
    src.P = &P;
    src.stg = sStg;
    src.f_ = fcur;
    src.g_ = pick(F.g, cur);
    src.lag_ = pick(F.lag, cur);
    src.plane = P.plane;
    src.tid = tid;
    src.ci = (ty + 2) * CW + tx + 4;
    src.mi = (ty + 1) * MW + tx + 1;
    src.ai = (ty + 1) * G::AW + tx + 4;
    src.sA = sA;
    src.xo[0] = wrap_index(x - 1, P.nx);
    src.xo[1] = x;
    src.xo[2] = wrap_index(x + 1, P.nx);
    src.yo[0] = wrap_index(y - 1, P.ny) * P.nx;
    src.yo[1] = y * P.nx;
    src.yo[2] = wrap_index(y + 1, P.ny) * P.nx;
    const int nxy = (int)P.nxy;   // nx ny nz < 2^31
    // (FP32) copy the lagged field a of plane z on the column and one node
    // around it: quads of rows x0-4 .. x0+35 with kVec, else node by node
    auto copy_a = [&](int z) {
        if constexpr (G::kRaw) {
            const int zo = wrap_index(z, P.nz) * nxy;
            T* d = sA + slot3(z) * 3 * G::AN;
            if constexpr (kVec) {
                if (tid < G::AN / 4) {
                    const int row = tid / (G::AW / 4), col = 4 * (tid % (G::AW / 4));
                    const int i = zo + ys[row + 1] + xs[col];
#pragma unroll
                    for (int k = 0; k < 3; ++k) cp_async16(d + k * G::AN + 4 * tid, src.lag_ + lag_a(k) * P.plane + i);
                }
            } else {
#pragma unroll
                for (int r = 0; r < G::KM; ++r) {
                    const int n = tid + r * NT;
                    if (n < MN) {
                        const int row = n / MW, col = n % MW + 3;
                        const int i = zo + ys[row + 1] + xs[col];
#pragma unroll
                        for (int k = 0; k < 3; ++k)
                            cp_async4(d + k * G::AN + row * G::AW + col, src.lag_ + lag_a(k) * P.plane + i);
                    }
                }
            }
        }
    };
    // (FP32) the group of copies that the update of plane z waits for: field a
    // of plane z+1 and (kStage) the column's g and lagged values of plane z,
    // by quads of a row with kVec (thread t: row t / 8 % TY, quad t % 8 of plane
    // t / 64 and every fourth from there), else each thread its own node's
    auto stage = [&](int z) {
        copy_a(z + 1);
        if constexpr (kStage) {
            const int zo = wrap_index(z, P.nz) * nxy;
            if constexpr (kVec) {
                constexpr int kPer = TY * kBX / 4;   // quads of a plane's column
                const int row = tid / (kBX / 4) % TY, x4 = x0 + 4 * (tid % (kBX / 4));
                if (x4 < P.nx && y0 + row < P.ny) {
                    const int i = zo + (y0 + row) * P.nx + x4, o = row * kBX + 4 * (tid % (kBX / 4));
#pragma unroll
                    for (int r = 0; r < (G::NSTG * kPer + NT - 1) / NT; ++r) {
                        const int q = tid / kPer + r * (NT / kPer);
                        if (q < G::NSTG)
                            cp_async16(sStg + q * NT + o,
                                       (q < 15 ? src.g_ + q * P.plane : src.lag_ + (q - 12) * P.plane) + i);
                    }
                }
            } else if (live) {
                const int i = zo + src.yo[1] + src.xo[1];
#pragma unroll
                for (int p = 0; p < 15; ++p) cp_async4(sStg + p * NT + tid, src.g_ + p * P.plane + i);
#pragma unroll
                for (int k = 3; k < n_lag(N); ++k) cp_async4(sStg + (12 + k) * NT + tid, src.lag_ + k * P.plane + i);
            }
        }
        if constexpr (G::kRaw) cp_async_commit();
    };

    for (int z = zb - 2; z <= zb + 1; ++z) {
        issue(z, true);
        c_pass(z);
    }
    copy_a(zb - 1);
    copy_a(zb);
    issue(zb + 2, true);
    __syncthreads();
    mu_pass(zb - 1);
    mu_pass(zb);
    for (int z = zb; z < ze; ++z) {
        c_pass(z + 2);
        __syncthreads();   // C of plane z + 2 is formed, the update of plane z - 1 done
        stage(z);
        issue(z + 3, z + 1 < ze);
        mu_pass(z + 1);
        if constexpr (G::kRaw) cp_async_wait<1>();   // raw(z + 3) may still fly
        __syncthreads();
        if (live) {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                src.zo[d] = wrap_index(z - 1 + d, P.nz) * nxy;
                src.c5[d] = slot5(z - 1 + d);
                src.m3[d] = slot3(z - 1 + d);
            }
            src.gp2 = (z - zb) & 1;
            update_node<T, NP, false>(P, F, cur, nullptr, src);
        }
    }
}

// ---------------------------------------------------------------------------
// initial state, staging, read-out, reduction
// ---------------------------------------------------------------------------
template <typename T, int NP>
__global__ void __launch_bounds__(node_threads<T>()) k3_init(P3<T> P, F3<T> F) {
    Site s;
    if (!site(P, s)) return;
    const long long i0 = s.self();
    const T psi = F.psi[i0];
    T* f = F.f[0];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        const T epm = P.eta[i] * psi * F.mu[i * P.plane + i0];
        const T psiC = psi * F.C[i * P.plane + i0];
        f[(7 * i) * P.plane + i0] = (P.w7_0 - T(1)) * epm + psiC;
#pragma unroll
        for (int p = 1; p < 7; ++p) f[(7 * i + p) * P.plane + i0] = P.w7_1 * epm;
    }
    // g = g^eq(P = 0, u = 0): zero with g_0 stored as g_0 - rho0
#pragma unroll
    for (int p = 0; p < 15; ++p) F.g[0][p * P.plane + i0] = T(0);
}

template <typename T>
__global__ void k3_from_double(const double* __restrict__ src, T* __restrict__ dst, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = (T)src[i];
}

template <typename T>
__global__ void k3_to_double(const T* __restrict__ src, double* __restrict__ dst, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = (double)src[i];
}

template <typename T, int NP>
__global__ void k3_derived_C(P3<T> P, F3<T> F, double* out) {
    const long long n = P.nxy * P.nz;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        T sum = T(0);
#pragma unroll
        for (int j = 0; j < NP; ++j) sum += F.C[j * P.plane + i];
        out[i] = (double)(T(1) - sum);
    }
}

template <typename T, int NP>
__global__ void __launch_bounds__(256) k3_mass_partial(P3<T> P, F3<T> F, int cur) {
    __shared__ double red[256][NP];
    const long long n = P.nxy * P.nz;
    const long long chunk = (n + kMassBlocks - 1) / kMassBlocks;
    const long long lo = blockIdx.x * chunk;
    const long long hi = lo + chunk < n ? lo + chunk : n;
    double acc[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) acc[i] = 0.0;
    const T* f = pick(F.f, cur);
    for (long long k = lo + threadIdx.x; k < hi; k += 256) {
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            double s = 0.0;
#pragma unroll
            for (int p = 0; p < 7; ++p) s += (double)f[(7 * i + p) * P.plane + k];
            acc[i] += s;
        }
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) red[threadIdx.x][i] = acc[i];
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
#pragma unroll
            for (int i = 0; i < NP; ++i) red[threadIdx.x][i] += red[threadIdx.x + w][i];
        __syncthreads();
    }
    if (threadIdx.x == 0)
#pragma unroll
        for (int i = 0; i < NP; ++i) F.partial[blockIdx.x * kMaxN + i] = red[0][i];
}

// one warp: every lane sums every 32nd partial, then the lanes in a fixed order
__global__ void k3_mass_final(const double* partial, int np, double* out, int* flag) {
    int bad = 0;
    for (int i = 0; i < np; ++i) {
        double s = 0.0;
        for (int b = threadIdx.x; b < kMassBlocks; b += 32) s += partial[b * kMaxN + i];
        for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
        if (threadIdx.x == 0) {
            out[i] = s;
            if (!isfinite(s)) bad = 1;
        }
    }
    if (threadIdx.x == 0) *flag = bad;
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
size_t round256(size_t b) { return (b + 255) & ~size_t(255); }

// Every value in (0, 1] (NaN fails).  Branch-free within blocks so that the
// compiler can vectorise the scan of a whole box.
bool all_in_unit(const double* v, long long n) {
    constexpr long long kB = 4096;
    for (long long i0 = 0; i0 < n; i0 += kB) {
        const long long i1 = i0 + kB < n ? i0 + kB : n;
        int bad = 0;
        for (long long i = i0; i < i1; ++i) bad |= (int)!(v[i] > 0.0) | (int)!(v[i] <= 1.0);
        if (bad) return false;
    }
    return true;
}

bool valid(const ddcc3d_params* p) {
    if (!p) return false;
    if (p->nx < 3 || p->ny < 3 || p->nz < 3) return false;
    if ((long long)p->nx * p->ny * p->nz > (1LL << 31) - 1) return false;
    // launch grid (nx/32, ny/4, nz/2): y and z block counts are limited to 65535
    if ((long long)p->ny > 65535LL * kBY || (long long)p->nz > 65535LL * kBZ) return false;
    if (p->nphase < 2 || p->nphase > kMaxN) return false;
    if (p->precision != DDCC_FP64 && p->precision != DDCC_FP32) return false;
    if (p->reserved != 0 || (p->flags & ~(uint32_t)(DDCC3D_FLAG_SPLIT | DDCC3D_FLAG_FUSED)) != 0) return false;
    if ((p->flags & DDCC3D_FLAG_SPLIT) && (p->flags & DDCC3D_FLAG_FUSED)) return false;
    if (!(p->d0 > 0.0 && p->d0 < 0.5)) return false;     // D3Q15 rest weight (1-d0)(1-2d0) > 0
    if (!(p->width > 0.0) || !(p->eps0 > 0.0) || !(p->m0 > 0.0)) return false;
    const int N = p->nphase;
    for (int i = 0; i < N; ++i) {
        if (!(p->rho[i] > 0.0) || !(p->nu[i] > 0.0)) return false;
        for (int j = 0; j < N; ++j) {
            if (p->sigma[i][j] != p->sigma[j][i]) return false;
            if (i == j ? p->sigma[i][j] != 0.0 : !(p->sigma[i][j] > 0.0)) return false;
        }
    }
    for (int i = 0; i < N - 1; ++i)
        if (!(p->eta[i] > 0.0)) return false;
    for (double s : p->s_f)
        if (!(s > 0.0 && s < 2.0)) return false;
    for (double s : p->s_g)
        if (!(s > 0.0 && s < 2.0)) return false;
    return true;
}

struct Layout {
    size_t plane_bytes, planes, stage, partial, flag, total;
};

Layout layout(const ddcc3d_params* p) {
    Layout L{};
    const size_t e = p->precision == DDCC_FP64 ? 8 : 4;
    const size_t n = (size_t)p->nx * p->ny * p->nz;
    const int N = p->nphase;
    L.plane_bytes = round256(n * e);
    L.planes = 2 * (7 * (N - 1) + 15) + 2 * n_lag(N) + 1 + (N - 1) + (N - 1) + N;
    if (p->precision == DDCC_FP64) L.planes += 1 + kStatic;
    L.stage = round256(n * 8);
    L.partial = round256((kMassBlocks + 1) * kMaxN * 8);   // + the N-1 totals
    L.flag = 256;
    L.total = L.planes * L.plane_bytes + L.stage + L.partial + L.flag;
    return L;
}

template <typename T>
void make_params(const ddcc3d_params* p, P3<T>& K) {
    std::memset(&K, 0, sizeof(K));
    const double d0 = p->d0, cs2 = d0;
    K.nx = p->nx;
    K.ny = p->ny;
    K.nz = p->nz;
    K.N = p->nphase;
    K.nxy = (long long)p->nx * p->ny;
    const size_t e = sizeof(T);
    K.plane = (long long)(round256((size_t)K.nxy * p->nz * e) / e);
    K.cs2 = (T)cs2;
    const double wa = (d0 - d0 * d0) / 2.0, wc = d0 * d0 / 8.0, w0 = 1.0 - 3.0 * d0 + 2.0 * d0 * d0;
    K.inv_cs2 = (T)(1.0 / cs2);
    K.ga = (T)(wa / cs2);
    K.gc = (T)(wc / cs2);
    K.la = (T)(0.75 * p->width * wa / cs2);
    K.lc = (T)(0.75 * p->width * wc / cs2);
    K.w7_0 = (T)(1.0 - 3.0 * d0);
    K.w7_1 = (T)(d0 / 2.0);
    K.w15[0] = (T)w0;
    K.w15[1] = (T)wa;
    K.w15[2] = (T)wc;
    const int N = p->nphase;
    for (int i = 0; i < N; ++i) {
        K.rho[i] = (T)p->rho[i];
        K.nu[i] = (T)p->nu[i];
        K.drho[i] = (T)(p->rho[i] - p->rho[N - 1]);
        K.dnu[i] = (T)(p->nu[i] - p->nu[N - 1]);
        double b2 = 0.0;
        K.sigN[i] = (T)p->sigma[i][N - 1];
        for (int j = 0; j < N; ++j) {
            const double s = p->sigma[i][j];
            K.beta2[i][j] = (T)(6.0 * s / p->width);
            b2 += 6.0 * s / p->width;
            K.sig[i][j] = (T)s;
            K.invsig[i][j] = (T)(i == j ? 0.0 : 1.0 / s);
        }
        K.beta2s[i] = (T)b2;
    }
    for (int i = 0; i < N - 1; ++i) {
        K.eta[i] = (T)p->eta[i];
        // Eq. 17: m0 = (1/s1 - 1/2) eta_i cs2
        const double s1 = 1.0 / (p->m0 / (p->eta[i] * cs2) + 0.5);
        K.ceta[i] = (T)(cs2 * p->eta[i]);
        K.h1f[i] = (T)(0.5 * s1);
        K.h2f[i] = (T)(0.25 * s1 - 0.5);
    }
    K.m0 = (T)p->m0;
    K.hs21f = (T)(0.5 * p->s_f[1]);
    // D3Q15 row norms under the weights: 1, d0, d0(1-d0), d0^2,
    // d0^2(1-d0), d0^2 (cx cy cz), d0^2 w0 (last row)
    const double n2d = d0 * (1.0 - d0), n2o = d0 * d0, n3 = d0 * d0 * (1.0 - d0), n4 = d0 * d0 * w0;
    K.lg0 = (T)p->s_g[0];
    K.lg1 = (T)(p->s_g[1] / d0);
    K.cg0 = (T)(0.5 * p->s_g[0] - 1.0);
    K.cg1 = (T)(0.5 * p->s_g[1] / d0 - 1.0 / d0);
    K.lg3 = (T)(p->s_g[2] / n3);
    K.lg3c = (T)(p->s_g[2] / (d0 * d0));
    K.lg4 = (T)(p->s_g[3] / n4);
    K.inv_n2d = (T)(1.0 / n2d);
    K.inv_n2o = (T)(1.0 / n2o);
    // Eq. 16: nu = (1/s21 - 1/2)(1 - cs2)/2 = (1/s22 - 1/2) cs2
    K.nu_to_s21 = (T)(2.0 / (1.0 - cs2));
    K.inv_cs2_nu = (T)(1.0 / cs2);
    K.damp = (T)(1.0 / (p->eps0 * p->eps0 * p->eps0));
    // Eq. 19 with the 3D constants K = 1 - 2 d0, H = K (3 - 7 d0)(s21 - 2)/2
    const double Kc = 1.0 - 2.0 * d0;
    K.K = (T)Kc;
    K.Hfac = (T)(Kc * (3.0 - 7.0 * d0) / 2.0);
    const double sg0 = p->s_g[0];
    K.A_P = (T)(0.5 + Kc * (1.0 - d0) * (2.0 - sg0) / (2.0 * sg0));
    K.cP = (T)(cs2 / (1.0 - w0));
    K.kk = (T)(Kc / 2.0 - w0 / (1.0 - cs2));
    K.c2m3 = (T)(1.0 - 3.0 * cs2);
    K.half_K = (T)(0.5 * Kc);
    K.two_cs2 = (T)(2.0 * cs2);
    K.one_m = (T)(1.0 - cs2);
    K.q0 = (T)(2.0 * cs2 * cs2);
    K.qa = (T)(2.0 * cs2 * cs2 - cs2);
    K.qc = (T)(1.0 - 3.0 * cs2 + 2.0 * cs2 * cs2);
    for (int a = 0; a < 3; ++a) K.body[a] = (T)p->body_force[a];
}

template <typename T>
void carve(const ddcc3d_params* p, char* ws, F3<T>& F) {
    const Layout L = layout(p);
    const int N = p->nphase;
    char* c = ws;
    auto take = [&](size_t planes) { T* r = (T*)c; c += planes * L.plane_bytes; return r; };
    for (int b = 0; b < 2; ++b) F.f[b] = take(7 * (N - 1));
    for (int b = 0; b < 2; ++b) F.g[b] = take(15);
    for (int b = 0; b < 2; ++b) F.lag[b] = take(n_lag(N));
    F.psi = take(1);
    F.cosf = take(N - 1);
    F.C = take(N - 1);
    F.mu = take(N);
    if (sizeof(T) == 8) {
        F.chi = take(1);
        F.st = take(kStatic);
    }
    F.stage = (double*)c;
    c += L.stage;
    F.partial = (double*)c;
    c += L.partial;
    F.flag = (int*)c;
}

}  // namespace

struct ddcc3d_handle {
    ddcc3d_params prm;
    cudaStream_t stream;
    char* ws;
    int cur;
    int64_t steps;
    int has_cos_field;
    P3<double> kd;
    P3<float> kf;
    F3<double> fd;
    F3<float> ff;
    double* dev_mass;
    int fused;        // one k3_fused launch per step (else the three kernels)
    int cmu_valid;    // F.C and F.mu hold the current state's C and mu (cleared by a step)
    int macro_valid;  // the other copy's g planes 0..4 hold its rho, u and P (cleared by a step)
    int nchunk;       // z chunks of the fused step's grid
    int profiling;
    std::vector<cudaEvent_t> events;
    std::vector<int> rec_kind;
};

namespace {

int prof_begin(ddcc3d_handle* h, int kind) {
    if (!h->profiling) return DDCC_OK;
    const size_t i = h->rec_kind.size();
    while (h->events.size() < 2 * (i + 1)) {
        cudaEvent_t e;
        if (cudaEventCreate(&e) != cudaSuccess) return DDCC_ERR_CUDA;
        h->events.push_back(e);
    }
    h->rec_kind.push_back(kind);
    return cudaEventRecord(h->events[2 * i], h->stream) == cudaSuccess ? DDCC_OK : DDCC_ERR_CUDA;
}

int prof_end(ddcc3d_handle* h) {
    if (!h->profiling) return DDCC_OK;
    const size_t i = h->rec_kind.size() - 1;
    return cudaEventRecord(h->events[2 * i + 1], h->stream) == cudaSuccess ? DDCC_OK : DDCC_ERR_CUDA;
}

template <typename T>
dim3 grid3(const ddcc3d_params& p) {
    if (sizeof(T) == 8) {
        const long long n = (long long)p.nx * p.ny * p.nz;
        return dim3((unsigned)((n + kLinear - 1) / kLinear));
    }
    return dim3((p.nx + kBX - 1) / kBX, (p.ny + kBY - 1) / kBY, (p.nz + kBZ - 1) / kBZ);
}
template <typename T>
dim3 block3() { return sizeof(T) == 8 ? dim3(kLinear) : dim3(kBX, kBY, kBZ); }

int launched() { return cudaGetLastError() == cudaSuccess ? DDCC_OK : DDCC_ERR_CUDA; }

template <typename T, int NP>
int order_mu(ddcc3d_handle* h, const P3<T>& K, const F3<T>& F, bool order) {
    const dim3 grid = grid3<T>(h->prm), block = block3<T>();
    int rc;
    if (order) {
        if ((rc = prof_begin(h, 0))) return rc;
        k3_order<T, NP><<<grid, block, 0, h->stream>>>(K, F, h->cur);
        if ((rc = launched()) || (rc = prof_end(h))) return rc;
    }
    if ((rc = prof_begin(h, 1))) return rc;
    if constexpr (sizeof(T) == 4) {
        if (K.nx % 4 == 0) {
            const dim3 grid4((K.nx / 4 + kBX4 - 1) / kBX4, grid.y, grid.z), block4(kBX4, kBY, kBZ);
            k3_mu4<NP><<<grid4, block4, 0, h->stream>>>(K, F);
        } else {
            k3_mu<T, NP><<<grid, block, 0, h->stream>>>(K, F);
        }
    } else {
        k3_mu<T, NP><<<grid, block, 0, h->stream>>>(K, F);
    }
    if ((rc = launched()) || (rc = prof_end(h))) return rc;
    return DDCC_OK;
}

// Whether FP32 takes the fused step where the caller leaves the choice: for
// rows of whole quads, for N = 2, and for boxes of one column in x, where a
// small step's three launches weigh most.  With other rows every population is
// copied by itself (and a C is formed node by node), which from N = 3 costs
// more than the fields' way through memory that the fused step saves (us a
// step, fused and three kernels; N = 3: 33 x 32 x 32 19.8 and 16.6, 101 x 77 x
// 63 101 and 88, 131 x 97 x 100 255 and 199, 255 x 256 x 200 1829 and 1616; N =
// 4: 26.7 and 18.5, 140 and 111, 350 and 260, 2553 and 2117; N = 2 within 13%
// either way, 1043 and 1101 at the largest; 25 x 31 x 31, N = 3, 12.4 and 15.0).
bool fused_pays(const ddcc3d_params* p) { return p->nx % 4 == 0 || p->nphase == 2 || p->nx <= kBX; }

// Shared memory of the fused step and its z chunks: the count of chunks n
// minimises (waves of CTAs) x (planes a CTA forms C for), i.e.
// ceil(columns n / resident CTAs) x (ceil(nz / n) + 3).
template <typename T, int NP>
constexpr bool fused_stage() { return sizeof(T) == 4 && NP <= 2; }

template <typename T, int NP, bool kVec>
int fused_setup_v(ddcc3d_handle* h) {
    constexpr bool kS = fused_stage<T, NP>();
    using G = FusedGeom<T, NP, kFusedTY, kVec, kS>;
    if (cudaFuncSetAttribute(k3_fused<T, NP, kFusedTY, kVec, kS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)G::smem) != cudaSuccess)
        return DDCC_ERR_CUDA;
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k3_fused<T, NP, kFusedTY, kVec, kS>, G::NT, G::smem) !=
            cudaSuccess)
        return DDCC_ERR_CUDA;
    if (per_sm < 1) return DDCC_ERR_CUDA;
    const long long cols = (long long)((h->prm.nx + kBX - 1) / kBX) * ((h->prm.ny + kFusedTY - 1) / kFusedTY);
    const long long resident = (long long)sms * per_sm;
    const int nz = h->prm.nz;
    long long best = -1;
    for (int n = 1; n <= nz && n <= 65535; ++n) {
        const long long cost = ((cols * n + resident - 1) / resident) * ((nz + n - 1) / n + 3);
        if (best < 0 || cost < best) {
            best = cost;
            h->nchunk = n;
        }
    }
    return DDCC_OK;
}

// FP32 stages the C pass by cp.async: by 16 bytes where nx is a multiple of 4
// (rows are whole aligned quads), else node by node.
template <typename T>
bool fused_vec(const ddcc3d_handle* h) { return sizeof(T) == 4 && h->prm.nx % 4 == 0; }

template <typename T, int NP>
int fused_setup(ddcc3d_handle* h) {
    if constexpr (sizeof(T) == 4) {
        if (fused_vec<T>(h)) return fused_setup_v<T, NP, true>(h);
    }
    return fused_setup_v<T, NP, false>(h);
}

template <typename T, int NP, bool kVec>
int fused_launch(ddcc3d_handle* h, const P3<T>& K, const F3<T>& F) {
    constexpr bool kS = fused_stage<T, NP>();
    using G = FusedGeom<T, NP, kFusedTY, kVec, kS>;
    const dim3 gf((h->prm.nx + kBX - 1) / kBX, (h->prm.ny + kFusedTY - 1) / kFusedTY, h->nchunk);
    k3_fused<T, NP, kFusedTY, kVec, kS><<<gf, G::NT, G::smem, h->stream>>>(K, F, h->cur, h->nchunk);
    return launched();
}

template <typename T, int NP>
int step_n(ddcc3d_handle* h, const P3<T>& K, const F3<T>& F, int64_t n) {
    const dim3 grid = grid3<T>(h->prm), block = block3<T>();
    if (h->fused) {
        for (int64_t s = 0; s < n; ++s) {
            int rc;
            if ((rc = prof_begin(h, 3))) return rc;
            if constexpr (sizeof(T) == 4) {
                rc = fused_vec<T>(h) ? fused_launch<T, NP, true>(h, K, F) : fused_launch<T, NP, false>(h, K, F);
            } else {
                rc = fused_launch<T, NP, false>(h, K, F);
            }
            if (rc || (rc = prof_end(h))) return rc;
            h->cur ^= 1;
            ++h->steps;
        }
        return DDCC_OK;
    }
    for (int64_t s = 0; s < n; ++s) {
        int rc = order_mu<T, NP>(h, K, F, true);
        if (rc) return rc;
        if ((rc = prof_begin(h, 2))) return rc;
        k3_update<T, NP, false><<<grid, block, 0, h->stream>>>(K, F, h->cur, nullptr);
        if ((rc = launched()) || (rc = prof_end(h))) return rc;
        h->cur ^= 1;
        ++h->steps;
    }
    return DDCC_OK;
}

template <typename T, int NP>
int init_n(ddcc3d_handle* h, const P3<T>& K, const F3<T>& F) {
    const dim3 grid = grid3<T>(h->prm), block = block3<T>();
    int rc;
    if constexpr (sizeof(T) == 8) {
        k3_static<T><<<grid, block, 0, h->stream>>>(K, F);
        if ((rc = launched())) return rc;
    }
    if ((rc = order_mu<T, NP>(h, K, F, false))) return rc;
    k3_init<T, NP><<<grid, block, 0, h->stream>>>(K, F);
    return launched();
}

template <typename T, int NP>
int read_n(ddcc3d_handle* h, const P3<T>& K, const F3<T>& F, int field, double* host_out) {
    const dim3 grid = grid3<T>(h->prm), block = block3<T>();
    const int N = NP + 1;
    const long long n = K.nxy * K.nz;
    int rc;
    if (!h->cmu_valid) {
        if ((rc = order_mu<T, NP>(h, K, F, true))) return rc;
        h->cmu_valid = 1;
    }
    const int cb = 2 * 152 * 4, ct = 256;
    if (field >= DDCC_FIELD_C && field < DDCC_FIELD_C + N) {
        const int i = field - DDCC_FIELD_C;
        if (i < NP) k3_to_double<T><<<cb, ct, 0, h->stream>>>(F.C + i * K.plane, F.stage, n);
        else k3_derived_C<T, NP><<<cb, ct, 0, h->stream>>>(K, F, F.stage);
    } else if (field >= DDCC_FIELD_MU && field < DDCC_FIELD_MU + N) {
        k3_to_double<T><<<cb, ct, 0, h->stream>>>(F.mu + (field - DDCC_FIELD_MU) * K.plane, F.stage, n);
    } else if (field == DDCC_FIELD_PSI) {
        k3_to_double<T><<<cb, ct, 0, h->stream>>>(F.psi, F.stage, n);
    } else if (field == DDCC_FIELD_RHO || field == DDCC_FIELD_UX || field == DDCC_FIELD_UY ||
               field == DDCC_FIELD_UZ || field == DDCC_FIELD_P) {
        // rho, u and P of a state are formed together on the first read, in
        // planes of the other population copy, which the next step overwrites
        T* out = F.g[h->cur ^ 1];
        if (!h->macro_valid) {
            k3_update<T, NP, true><<<grid, block, 0, h->stream>>>(K, F, h->cur, out);
            if ((rc = launched())) return rc;
            h->macro_valid = 1;
        }
        const int k = field == DDCC_FIELD_RHO ? 0 : field == DDCC_FIELD_UX ? 1 : field == DDCC_FIELD_UY ? 2
                      : field == DDCC_FIELD_UZ ? 3 : 4;
        k3_to_double<T><<<cb, ct, 0, h->stream>>>(out + k * K.plane, F.stage, n);
    } else {
        return DDCC_ERR_PARAM;
    }
    if ((rc = launched())) return rc;
    if (cudaMemcpyAsync(host_out, F.stage, n * sizeof(double), cudaMemcpyDeviceToHost, h->stream) != cudaSuccess)
        return DDCC_ERR_CUDA;
    return cudaStreamSynchronize(h->stream) == cudaSuccess ? DDCC_OK : DDCC_ERR_CUDA;
}

template <typename T, int NP>
int mass_n(ddcc3d_handle* h, const P3<T>& K, const F3<T>& F, double* host_out) {
    k3_mass_partial<T, NP><<<kMassBlocks, 256, 0, h->stream>>>(K, F, h->cur);
    k3_mass_final<<<1, 32, 0, h->stream>>>(F.partial, NP, h->dev_mass, F.flag);
    if (launched()) return DDCC_ERR_CUDA;
    double out[kMaxN + 1];
    int flag = 0;
    if (cudaMemcpyAsync(out, h->dev_mass, NP * sizeof(double), cudaMemcpyDeviceToHost, h->stream) != cudaSuccess ||
        cudaMemcpyAsync(&flag, F.flag, sizeof(int), cudaMemcpyDeviceToHost, h->stream) != cudaSuccess ||
        cudaStreamSynchronize(h->stream) != cudaSuccess)
        return DDCC_ERR_CUDA;
    std::memcpy(host_out, out, NP * sizeof(double));
    return flag ? DDCC_ERR_NONFINITE : DDCC_OK;
}

// Host double array -> device plane of T through the double staging plane.
template <typename T>
int upload_plane(ddcc3d_handle* h, double* stage, const double* src, T* dst, long long n) {
    if (cudaMemcpyAsync(stage, src, n * sizeof(double), cudaMemcpyHostToDevice, h->stream) != cudaSuccess)
        return DDCC_ERR_CUDA;
    k3_from_double<T><<<2 * 152 * 4, 256, 0, h->stream>>>(stage, dst, n);
    if (launched()) return DDCC_ERR_CUDA;
    // the staging plane is reused by the next upload: order the copies
    return cudaStreamSynchronize(h->stream) == cudaSuccess ? DDCC_OK : DDCC_ERR_CUDA;
}

template <typename T>
int create_t(ddcc3d_handle* h, const P3<T>& K, const F3<T>& F, const double* psi, const double* cosf,
             const double* C0) {
    const long long n = K.nxy * K.nz;
    const int N = h->prm.nphase;
    int rc = upload_plane<T>(h, F.stage, psi, F.psi, n);
    if (rc) return rc;
    if (cosf)
        for (int i = 0; i < N - 1; ++i)
            if ((rc = upload_plane<T>(h, F.stage, cosf + i * n, F.cosf + i * K.plane, n))) return rc;
    for (int i = 0; i < N - 1; ++i)
        if ((rc = upload_plane<T>(h, F.stage, C0 + i * n, F.C + i * K.plane, n))) return rc;
    const Layout L = layout(&h->prm);
    for (int b = 0; b < 2; ++b)
        if (cudaMemsetAsync(F.lag[b], 0, n_lag(N) * L.plane_bytes, h->stream) != cudaSuccess) return DDCC_ERR_CUDA;
    switch (N - 1) {
        case 1: rc = init_n<T, 1>(h, K, F); break;
        case 2: rc = init_n<T, 2>(h, K, F); break;
        default: rc = init_n<T, 3>(h, K, F); break;
    }
    if (rc) return rc;
    if (h->fused) {
        switch (N - 1) {
            case 1: rc = fused_setup<T, 1>(h); break;
            case 2: rc = fused_setup<T, 2>(h); break;
            default: rc = fused_setup<T, 3>(h); break;
        }
        if (rc) return rc;
    }
    return cudaStreamSynchronize(h->stream) == cudaSuccess ? DDCC_OK : DDCC_ERR_CUDA;
}

}  // namespace

extern "C" {

size_t ddcc3d_workspace_bytes(const ddcc3d_params* params) {
    if (!valid(params)) return 0;
    return layout(params).total;
}

int ddcc3d_create(const ddcc3d_params* params, void* dev_workspace, size_t bytes, void* cuda_stream,
                  const double* psi, const double* cos_theta_field, const double* cos_theta_uniform,
                  const double* C0, ddcc3d_handle** out) {
    if (!out) return DDCC_ERR_PARAM;
    *out = nullptr;
    if (!valid(params) || !psi || !C0 || (!cos_theta_field && !cos_theta_uniform)) return DDCC_ERR_PARAM;
    const long long n = (long long)params->nx * params->ny * params->nz;
    if (!all_in_unit(psi, n)) return DDCC_ERR_PARAM;
    if (!dev_workspace || ((uintptr_t)dev_workspace & 255) || bytes < layout(params).total) return DDCC_ERR_WORKSPACE;
    ddcc3d_handle* h = new (std::nothrow) ddcc3d_handle();
    if (!h) return DDCC_ERR_NOMEM;
    h->prm = *params;
    h->stream = (cudaStream_t)cuda_stream;
    h->ws = (char*)dev_workspace;
    h->cur = 0;
    h->steps = 0;
    h->has_cos_field = cos_theta_field != nullptr;
    h->profiling = 0;
    // FP32 steps fused by default; FP64 with the three kernels (its fused
    // kernel recomputes mu on the column halos and is bound by the FP64 pipe)
    h->fused = (params->flags & DDCC3D_FLAG_FUSED) ||
               (!(params->flags & DDCC3D_FLAG_SPLIT) && params->precision == DDCC_FP32 && fused_pays(params));
    h->nchunk = 1;
    int rc;
    if (params->precision == DDCC_FP64) {
        make_params(params, h->kd);
        carve(params, h->ws, h->fd);
        h->kd.has_cos_field = h->has_cos_field;
        if (!h->has_cos_field)
            for (int i = 0; i < params->nphase - 1; ++i) h->kd.cos_uni[i] = cos_theta_uniform[i];
        h->dev_mass = h->fd.partial + kMassBlocks * kMaxN;
        rc = create_t<double>(h, h->kd, h->fd, psi, cos_theta_field, C0);
    } else {
        make_params(params, h->kf);
        carve(params, h->ws, h->ff);
        h->kf.has_cos_field = h->has_cos_field;
        if (!h->has_cos_field)
            for (int i = 0; i < params->nphase - 1; ++i) h->kf.cos_uni[i] = (float)cos_theta_uniform[i];
        h->dev_mass = h->ff.partial + kMassBlocks * kMaxN;
        rc = create_t<float>(h, h->kf, h->ff, psi, cos_theta_field, C0);
    }
    if (rc) {
        delete h;
        return rc;
    }
    *out = h;
    return DDCC_OK;
}

int ddcc3d_step(ddcc3d_handle* h, int64_t nsteps) {
    if (!h || nsteps < 0) return DDCC_ERR_PARAM;
    h->cmu_valid = 0;
    h->macro_valid = 0;
    const int np = h->prm.nphase - 1;
    if (h->prm.precision == DDCC_FP64) {
        if (np == 1) return step_n<double, 1>(h, h->kd, h->fd, nsteps);
        if (np == 2) return step_n<double, 2>(h, h->kd, h->fd, nsteps);
        return step_n<double, 3>(h, h->kd, h->fd, nsteps);
    }
    if (np == 1) return step_n<float, 1>(h, h->kf, h->ff, nsteps);
    if (np == 2) return step_n<float, 2>(h, h->kf, h->ff, nsteps);
    return step_n<float, 3>(h, h->kf, h->ff, nsteps);
}

int ddcc3d_read(ddcc3d_handle* h, int field, double* host_out) {
    if (!h || !host_out) return DDCC_ERR_PARAM;
    const int np = h->prm.nphase - 1;
    int rc;
    if (h->prm.precision == DDCC_FP64) {
        rc = np == 1   ? read_n<double, 1>(h, h->kd, h->fd, field, host_out)
             : np == 2 ? read_n<double, 2>(h, h->kd, h->fd, field, host_out)
                       : read_n<double, 3>(h, h->kd, h->fd, field, host_out);
    } else {
        rc = np == 1   ? read_n<float, 1>(h, h->kf, h->ff, field, host_out)
             : np == 2 ? read_n<float, 2>(h, h->kf, h->ff, field, host_out)
                       : read_n<float, 3>(h, h->kf, h->ff, field, host_out);
    }
    if (rc) {
        // the planes may not have been formed, and the error is not the next call's
        h->cmu_valid = h->macro_valid = 0;
        cudaGetLastError();
    }
    return rc;
}

int ddcc3d_mass(ddcc3d_handle* h, double* host_out) {
    if (!h || !host_out) return DDCC_ERR_PARAM;
    const int np = h->prm.nphase - 1;
    if (h->prm.precision == DDCC_FP64) {
        if (np == 1) return mass_n<double, 1>(h, h->kd, h->fd, host_out);
        if (np == 2) return mass_n<double, 2>(h, h->kd, h->fd, host_out);
        return mass_n<double, 3>(h, h->kd, h->fd, host_out);
    }
    if (np == 1) return mass_n<float, 1>(h, h->kf, h->ff, host_out);
    if (np == 2) return mass_n<float, 2>(h, h->kf, h->ff, host_out);
    return mass_n<float, 3>(h, h->kf, h->ff, host_out);
}

int64_t ddcc3d_step_count(const ddcc3d_handle* h) { return h ? h->steps : -1; }

int ddcc3d_profile(ddcc3d_handle* h, int enable) {
    if (!h) return DDCC_ERR_PARAM;
    h->profiling = enable != 0;
    return DDCC_OK;
}

int ddcc3d_kernel_times(ddcc3d_handle* h, double* ms_out, int64_t* launches_out, int max_kinds) {
    if (!h || max_kinds < 0) return DDCC_ERR_PARAM;
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) return DDCC_ERR_CUDA;
    double ms[kKinds] = {0.0, 0.0, 0.0, 0.0};
    int64_t cnt[kKinds] = {0, 0, 0, 0};
    for (size_t i = 0; i < h->rec_kind.size(); ++i) {
        float t = 0.f;
        if (cudaEventElapsedTime(&t, h->events[2 * i], h->events[2 * i + 1]) != cudaSuccess) return DDCC_ERR_CUDA;
        ms[h->rec_kind[i]] += t;
        ++cnt[h->rec_kind[i]];
    }
    h->rec_kind.clear();
    for (int k = 0; k < kKinds && k < max_kinds; ++k) {
        if (ms_out) ms_out[k] = ms[k];
        if (launches_out) launches_out[k] = cnt[k];
    }
    return kKinds;
}

void ddcc3d_destroy(ddcc3d_handle* h) {
    if (!h) return;
    cudaStreamSynchronize(h->stream);
    for (cudaEvent_t e : h->events) cudaEventDestroy(e);
    delete h;
}

}  // extern "C"
