// Tile kernels of the DD-CCLB step (arXiv 2311.10314, Sec. 3) and the
// small utility kernels (initial state, read-out, reductions, uploads).
//
// Tile step (two launches):
//   k_order_param  psi C_i = sum_p f^i_p, C_i = psi C_i / psi -> C scratch;
//   k_step         per 32 x 8 tile: C and psi with a 2-node halo and the
//                  lagged field a with a 1-node halo are staged in shared
//                  memory, mu_i (Eq. 2.14) is evaluated on the tile plus a
//                  1-node halo, then every node runs dev::node_update and
//                  pushes its post-collision populations to its neighbours.
// These run the FP32 step; ddcc_fp64.cu has the FP64 one.
// k_step_tma is the same tile step with every input staged by TMA tensor
// copies (halo boxes of C, psi, cos(theta) and a first, then the tile's
// populations and lagged planes, which land while mu is evaluated); it is
// the collide kernel of the tile path whenever the planes are wide enough
// for its boxes.  k_step with plain loads covers tiny grids, the read-out
// and the initial state.
#include <algorithm>
#include "ddcc_device.cuh"
#include "ddcc_tma.cuh"

namespace ddcc {
namespace {

using dev::map_index;

constexpr int BX = kTileX;
constexpr int BY = kTileY;
constexpr int NT = BX * BY;
constexpr int H2W = BX + 4, H2H = BY + 4;   // tile + 2-node halo
constexpr int H1W = BX + 2, H1H = BY + 2;   // tile + 1-node halo

// D2Q9 velocities (Sec. 3): 0 rest, 1-4 axis, 5-8 diagonal.
__constant__ int kCx[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
__constant__ int kCy[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};

template <typename T, int NP>
struct Smem {
    T C[NP - 1][H2H][H2W];
    T psi[H2H][H2W];
    T mu[NP][H1H][H1W];
    T a[H1H][H1W];
    T cth[NP - 1][H1H][H1W];
};

// Stage C (N-1 planes) and psi with a 2-node halo, a and cos(theta_iN)
// with a 1-node halo (periodic wrap or mirror ghosts).
template <typename T, int NP>
__device__ void load_tile(const KParams<T>& P, Smem<T, NP>& sm, const T* __restrict__ C,
                          const T* __restrict__ psi, const T* __restrict__ cosf,
                          const T* __restrict__ a_in, int x0, int y0, int tid) {
    for (int k = tid; k < H2H * H2W; k += NT) {
        const int ly = k / H2W, lx = k - ly * H2W;
        const int gx = map_index(x0 + lx - 2, P.nx, P.px);
        const int gy = map_index(y0 + ly - 2, P.ny, P.py);
        const long long o = P.org + (long long)gy * P.pitch + gx;
        sm.psi[ly][lx] = psi[o];
#pragma unroll
        for (int i = 0; i < NP - 1; ++i) sm.C[i][ly][lx] = C[i * P.plane + o];
    }
    for (int k = tid; k < H1H * H1W; k += NT) {
        const int ly = k / H1W, lx = k - ly * H1W;
        const int gx = map_index(x0 + lx - 1, P.nx, P.px);
        const int gy = map_index(y0 + ly - 1, P.ny, P.py);
        const long long o = P.org + (long long)gy * P.pitch + gx;
        sm.a[ly][lx] = a_in ? a_in[o] : T(0);
#pragma unroll
        for (int i = 0; i < NP - 1; ++i)
            sm.cth[i][ly][lx] = P.has_cos_field ? cosf[i * P.plane + o] : P.cos_uni[i];
    }
}

// mu on the tile + 1-node halo.
template <typename T, int NP>
__device__ void compute_mu_tile(const KParams<T>& P, Smem<T, NP>& sm, int tid) {
    for (int k = tid; k < H1H * H1W; k += NT) {
        const int ly = k / H1W, lx = k - ly * H1W;
        const int cy = ly + 1, cx = lx + 1;
        T cth[NP];
#pragma unroll
        for (int i = 0; i < NP - 1; ++i) cth[i] = sm.cth[i][ly][lx];
        T mu[NP];
        dev::chem_pot<T, NP>(
            P, [&](int j, int dy, int dx) { return sm.C[j][cy + dy][cx + dx]; },
            [&](int dy, int dx) { return sm.psi[cy + dy][cx + dx]; }, cth, mu);
#pragma unroll
        for (int i = 0; i < NP; ++i) sm.mu[i][ly][lx] = mu[i];
    }
}

template <typename T, int NP>
struct TileAcc {
    const KParams<T>& P;
    const Smem<T, NP>& sm;
    int cy, cx, hy, hx;
    long long o, plane;
    const T* __restrict__ lag_in;
    const T* __restrict__ fin;
    const T* __restrict__ gin;
    __device__ T C(int j, int dy, int dx) const { return sm.C[j][cy + dy][cx + dx]; }
    __device__ T psi(int dy, int dx) const { return sm.psi[cy + dy][cx + dx]; }
    __device__ void grad_psi(const KParams<T>& Q, T& gx, T& gy) const {
        dev::grad9(Q, [&](int dy, int dx) { return psi(dy, dx); }, gx, gy);
    }
    __device__ T psi_rho(int dy, int dx) const {
        return dev::psi_rho<T, NP>(P, psi(dy, dx), [&](int j) { return C(j, dy, dx); });
    }
    __device__ T mu(int j, int dy, int dx) const { return sm.mu[j][hy + dy][hx + dx]; }
    __device__ T a(int dy, int dx) const { return sm.a[hy + dy][hx + dx]; }
    __device__ T lag(int k) const { return lag_in[k * plane + o]; }
    __device__ T f(int i, int p) const { return fin[(i * 9 + p) * plane + o]; }
    __device__ T g(int p) const { return gin[p * plane + o]; }
};

// Push to x + c_p (periodic wrap), or back into the node's opposite
// direction where x + c_p lies beyond an outer wall (halfway bounce-back).
template <typename T, int NP>
struct TileSink {
    long long tgt[9];
    int tdir[9];
    long long o, plane;
    T* __restrict__ fout;
    T* __restrict__ gout;
    T* __restrict__ lout;
    T* __restrict__ macro_out;
    __device__ void f_out(int i, int p, T v) { fout[(i * 9 + tdir[p]) * plane + tgt[p]] = v; }
    __device__ void g_out(int p, T v) { gout[tdir[p] * plane + tgt[p]] = v; }
    __device__ void lag_out(int k, T v) { lout[k * plane + o] = v; }
    __device__ void macro(const T* Cv, T rho, T ux, T uy, T Pr, const T* mu) {
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            macro_out[j * plane + o] = Cv[j];
            macro_out[(NP + 4 + j) * plane + o] = mu[j];
        }
        macro_out[NP * plane + o] = rho;
        macro_out[(NP + 1) * plane + o] = ux;
        macro_out[(NP + 2) * plane + o] = uy;
        macro_out[(NP + 3) * plane + o] = Pr;
    }
};

// The sink of k_step: its state's readers take the one-node ghost ring of the
// lagged plane a from the state (the reverse step, and a load into a handle of
// another path), so the plane is written with its images.
template <typename T, int NP>
struct PlainSink : TileSink<T, NP> {
    long long ax, ay;   // offsets of a's images (0: none)
    __device__ void lag_out(int k, T v) {
        T* q = this->lout + k * this->plane + this->o;
        *q = v;
        if (k == 0) {
            if (ax) q[ax] = v;
            if (ay) q[ay] = v;
            if (ax && ay) q[ax + ay] = v;
        }
    }
};

// D2Q9 velocity components as compile-time functions of p (after unrolling
// they fold into the addresses).
__host__ __device__ constexpr int cxp(int p) { return (p == 1 || p == 5 || p == 8) ? 1 : (p == 3 || p == 6 || p == 7) ? -1 : 0; }
__host__ __device__ constexpr int cyp(int p) { return (p == 2 || p == 5 || p == 6) ? 1 : (p == 4 || p == 7 || p == 8) ? -1 : 0; }

// Push sink of a tile whose pushes all land inside the domain (no periodic
// wrap, no wall): every target is the node's own address plus a fixed
// offset, taken in 32-bit element offsets from the node (the launcher checks
// that the population and lagged buffers fit them).
template <typename T, int NP>
struct InnerSink {
    T* __restrict__ pop;   // output populations at this node
    T* __restrict__ lag;   // output lagged planes at this node
    int plane, pitch;
    __device__ void f_out(int i, int p, T v) { pop[(9 * i + p) * plane + cyp(p) * pitch + cxp(p)] = v; }
    __device__ void g_out(int p, T v) { pop[(9 * (NP - 1) + p) * plane + cyp(p) * pitch + cxp(p)] = v; }
    __device__ void lag_out(int k, T v) { lag[k * plane] = v; }
    __device__ void macro(const T*, T, T, T, T, const T*) {}
};

__device__ __forceinline__ int opposite(int p) {
    return p == 0 ? 0 : (p <= 4 ? ((p + 1) & 3) + 1 : ((p - 3) & 3) + 5);
}

// Push targets of node (x, y) at offset o.
template <typename T, int NP>
__device__ __forceinline__ void tile_targets(const KParams<T>& P, int x, int y, long long o, TileSink<T, NP>& sink) {
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        int tx = x + kCx[p], ty = y + kCy[p];
        bool bounce = false;
        if (tx < 0 || tx >= P.nx) {
            if (P.px) tx = tx < 0 ? tx + P.nx : tx - P.nx;
            else bounce = true;
        }
        if (ty < 0 || ty >= P.ny) {
            if (P.py) ty = ty < 0 ? ty + P.ny : ty - P.ny;
            else bounce = true;
        }
        sink.tgt[p] = bounce ? o : P.org + (long long)ty * P.pitch + tx;
        sink.tdir[p] = bounce ? opposite(p) : p;
    }
}

// Step from coordinate v to its copy in the 2-node ghost ring (0: none):
// periodic v -> v +- n, mirror -1 - v or 2 n - 1 - v.  One copy at most along
// an axis of four nodes or more.
__device__ __forceinline__ int ring2_step(int v, int n, int periodic) {
    if (v < 2) return periodic ? n : -1 - 2 * v;
    if (v >= n - 2) return periodic ? -n : 2 * (n - v) - 1;
    return 0;
}

// Push sink of the edge tiles of the fused kernel's 32 x 8 form: wrap and
// bounce-back as TileSink, and every phase population and the lagged plane a
// are also written to the copies of their node in the 2-node ghost ring that
// the next step's halo boxes read.  It takes a launch off a small grid's step
// (256 x 256, N = 3: 10.3 -> 9.1 us); the 64 x 4 form, for states over 128 MB,
// keeps the launch (4096 x 4096, N = 4: 1177 us a step with it, 1196 with
// this sink, whose registers also weigh on the inner tiles).
template <typename T, int NP>
struct EdgeSink {
    long long tgt[9];              // target, plane of the direction included
    unsigned bounced;              // bit p: population p comes back
    int dx[3], dy[3];              // ring steps of columns x-1, x, x+1 (rows: y) after wrapping
    long long o, plane;
    int pitch;
    T* __restrict__ pop;
    T* __restrict__ lag;
    __device__ void copies(T* q, int sx, int sy, T v) const {
        const long long ry = (long long)sy * pitch;
        if (sx) q[sx] = v;
        if (sy) q[ry] = v;
        if (sx && sy) q[ry + sx] = v;
    }
    __device__ void f_out(int i, int p, T v) {
        T* q = pop + (long long)(9 * i) * plane + tgt[p];
        *q = v;
        const bool b = (bounced >> p) & 1;
        copies(q, b ? dx[1] : dx[cxp(p) + 1], b ? dy[1] : dy[cyp(p) + 1], v);
    }
    __device__ void g_out(int p, T v) { pop[(long long)(9 * (NP - 1)) * plane + tgt[p]] = v; }
    __device__ void lag_out(int k, T v) {
        T* q = lag + k * plane + o;
        *q = v;
        if (k == 0) copies(q, dx[1], dy[1], v);
    }
    __device__ void macro(const T*, T, T, T, T, const T*) {}
};

// MODE 0: full step (collide + push-stream + lagged fields).
// MODE 1: macroscopic read-out of the current state (no state change).
template <typename T, int NP, int MODE>
__global__ void __launch_bounds__(NT) k_step(KParams<T> P, Fields<T> F, int cur) {
    __shared__ Smem<T, NP> sm;
    const int tid = threadIdx.x + BX * threadIdx.y;
    const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY;
    // select ping-pong copies without indexing the parameter struct at run
    // time (that would copy it to local memory)
    const T* __restrict__ lag_in = cur ? F.lag[1] : F.lag[0];
    T* __restrict__ lag_out = cur ? F.lag[0] : F.lag[1];
    const T* __restrict__ fin = cur ? F.f[1] : F.f[0];
    T* __restrict__ fout = cur ? F.f[0] : F.f[1];
    const T* __restrict__ gin = cur ? F.g[1] : F.g[0];
    T* __restrict__ gout = cur ? F.g[0] : F.g[1];
    load_tile<T, NP>(P, sm, F.C, F.psi, F.cosf, lag_in, x0, y0, tid);
    __syncthreads();
    compute_mu_tile<T, NP>(P, sm, tid);
    __syncthreads();

    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    const long long o = P.org + (long long)y * P.pitch + x;
    TileAcc<T, NP> acc{P, sm, (int)threadIdx.y + 2, (int)threadIdx.x + 2, (int)threadIdx.y + 1,
                       (int)threadIdx.x + 1, o, P.plane, lag_in, fin, gin};
    PlainSink<T, NP> sink;
    sink.o = o;
    sink.plane = P.plane;
    sink.fout = fout;
    sink.gout = gout;
    sink.lout = lag_out;
    sink.macro_out = F.macro;
    if (MODE == 0) {
        tile_targets<T, NP>(P, x, y, o, sink);
        sink.ax = dev::ring_step(x, P.nx, P.px);
        sink.ay = (long long)dev::ring_step(y, P.ny, P.py) * P.pitch;
    }
    dev::node_update<T, NP, MODE>(P, acc, sink);
}

// ---- TMA-staged tile step -------------------------------------------------

template <typename T, int NP, bool TF>
struct TLay {
    static constexpr int NPOP = 9 * NP;
    static constexpr int NLAG = 2 * NP + 3;
    static constexpr int NST = TF ? NP : 1;
    static constexpr int HX = kTileHaloW;                  // halo box columns x0-4 .. x0+35
    static constexpr int pad(int e) { return (e * (int)sizeof(T) + 127) / 128 * 128 / (int)sizeof(T); }
    static constexpr int POP_BOX = NPOP * BY * BX;
    static constexpr int LAG_BOX = NLAG * BY * BX;
    static constexpr int C_BOX = (NP - 1) * (BY + 4) * HX;   // rows y0-2 .. y0+9
    static constexpr int ST_BOX = NST * (BY + 4) * HX;
    static constexpr int A_BOX = (BY + 2) * HX;               // rows y0-1 .. y0+8
    static constexpr int MU = NP * (BY + 2) * (BX + 2);
    static constexpr size_t pop_off = 0;
    static constexpr size_t lag_off = pop_off + pad(POP_BOX);
    static constexpr size_t c_off = lag_off + pad(LAG_BOX);
    static constexpr size_t st_off = c_off + pad(C_BOX);
    static constexpr size_t a_off = st_off + pad(ST_BOX);
    static constexpr size_t mu_off = a_off + pad(A_BOX);
    static constexpr size_t end = mu_off + MU;
    static constexpr size_t bar_byte_off = (end * sizeof(T) + 127) / 128 * 128;
    static constexpr size_t bytes = bar_byte_off + 64;
    static constexpr unsigned tx_halo = (unsigned)((C_BOX + ST_BOX + A_BOX) * sizeof(T));
    static constexpr unsigned tx_tile = (unsigned)((POP_BOX + LAG_BOX) * sizeof(T));
};

template <typename T, int NP, bool TF>
struct TmaAcc {
    using L = TLay<T, NP, TF>;
    const KParams<T>& P;
    const T* sm;
    int tx, ty;
    __device__ T C(int j, int dy, int dx) const {
        return sm[L::c_off + ((size_t)j * (BY + 4) + ty + 2 + dy) * L::HX + tx + 4 + dx];
    }
    __device__ T psi(int dy, int dx) const { return sm[L::st_off + (size_t)(ty + 2 + dy) * L::HX + tx + 4 + dx]; }
    __device__ void grad_psi(const KParams<T>& Q, T& gx, T& gy) const {
        dev::grad9(Q, [&](int dy, int dx) { return psi(dy, dx); }, gx, gy);
    }
    __device__ T psi_rho(int dy, int dx) const {
        return dev::psi_rho<T, NP>(P, psi(dy, dx), [&](int j) { return C(j, dy, dx); });
    }
    __device__ T mu(int j, int dy, int dx) const {
        return sm[L::mu_off + ((size_t)j * (BY + 2) + ty + 1 + dy) * (BX + 2) + tx + 1 + dx];
    }
    __device__ T a(int dy, int dx) const { return sm[L::a_off + (size_t)(ty + 1 + dy) * L::HX + tx + 4 + dx]; }
    __device__ T lag(int k) const { return sm[L::lag_off + ((size_t)k * BY + ty) * BX + tx]; }
    __device__ T f(int i, int p) const { return sm[L::pop_off + ((size_t)(9 * i + p) * BY + ty) * BX + tx]; }
    __device__ T g(int p) const { return sm[L::pop_off + ((size_t)(9 * (NP - 1) + p) * BY + ty) * BX + tx]; }
};

// Two CTAs per SM (128 registers, ~69 KB of shared memory each).
template <typename T, int NP, bool TF>
__global__ void __launch_bounds__(NT, 2)
    k_step_tma(const __grid_constant__ CUtensorMap tm_pop, const __grid_constant__ CUtensorMap tm_lag,
               const __grid_constant__ CUtensorMap tm_c, const __grid_constant__ CUtensorMap tm_st,
               const __grid_constant__ CUtensorMap tm_a, KParams<T> P, T* __restrict__ pop_out,
               T* __restrict__ lag_out, int* __restrict__ err) {
    using L = TLay<T, NP, TF>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem_raw + L::bar_byte_off);
    const int tid = threadIdx.x + BX * threadIdx.y;
    const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY;
    if (tid == 0) {
        tma::mbar_init(&bars[0], 1);
        tma::mbar_init(&bars[1], 1);
        tma::mbar_init_fence();
    }
    __syncthreads();
    // padded coordinates: column x0 - 4 is x0 (kGX = 4), row y is y + kGY
    if (tid == 0) {
        tma::mbar_expect_tx(&bars[0], L::tx_halo);
        tma::load_3d(sm + L::c_off, &tm_c, x0, y0 - 2 + kGY, 0, &bars[0]);
        tma::load_3d(sm + L::st_off, &tm_st, x0, y0 - 2 + kGY, 0, &bars[0]);
        tma::load_3d(sm + L::a_off, &tm_a, x0, y0 - 1 + kGY, 0, &bars[0]);
        tma::mbar_expect_tx(&bars[1], L::tx_tile);
        tma::load_3d(sm + L::pop_off, &tm_pop, x0 + kGX, y0 + kGY, 0, &bars[1]);
        tma::load_3d(sm + L::lag_off, &tm_lag, x0 + kGX, y0 + kGY, 0, &bars[1]);
    }
    bool ok = tma::mbar_wait_bounded(&bars[0], 0);
    if (!__syncthreads_and(ok)) {
        // a copy has not landed within the bounded wait: record it, and give
        // every copy still in flight a second bounded wait before the CTA and
        // its shared memory go
        if (tid == 0) {
            atomicOr(err, 1);
            tma::mbar_wait_bounded(&bars[0], 0);
            tma::mbar_wait_bounded(&bars[1], 0);
        }
        return;
    }
    // mu on the tile + 1-node halo while the tile's populations land
    for (int k = tid; k < (BY + 2) * (BX + 2); k += NT) {
        const int ly = k / (BX + 2), lx = k - ly * (BX + 2);
        const T* cb = sm + L::c_off + (size_t)(ly + 1) * L::HX + lx + 3;
        const T* sb = sm + L::st_off + (size_t)(ly + 1) * L::HX + lx + 3;
        T cth[NP];
#pragma unroll
        for (int i = 0; i < NP - 1; ++i)
            cth[i] = TF ? sb[(size_t)(1 + i) * (BY + 4) * L::HX] : P.cos_uni[i];
        T mu[NP];
        dev::chem_pot<T, NP>(
            P, [&](int j, int dy, int dx) { return cb[((size_t)j * (BY + 4) + dy) * L::HX + dx]; },
            [&](int dy, int dx) { return sb[dy * L::HX + dx]; }, cth, mu);
#pragma unroll
        for (int i = 0; i < NP; ++i) sm[L::mu_off + ((size_t)i * (BY + 2) + ly) * (BX + 2) + lx] = mu[i];
    }
    ok = tma::mbar_wait_bounded(&bars[1], 0);
    if (!__syncthreads_and(ok)) {
        if (tid == 0) {
            atomicOr(err, 1);
            tma::mbar_wait_bounded(&bars[1], 0);
        }
        return;
    }
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    const long long o = P.org + (long long)y * P.pitch + x;
    TmaAcc<T, NP, TF> acc{P, sm, (int)threadIdx.x, (int)threadIdx.y};
    TileSink<T, NP> sink;
    sink.o = o;
    sink.plane = P.plane;
    sink.fout = pop_out;
    sink.gout = pop_out + (long long)9 * (NP - 1) * P.plane;
    sink.lout = lag_out;
    sink.macro_out = nullptr;
    tile_targets(P, x, y, o, sink);
    dev::node_update<T, NP, 0>(P, acc, sink);
}

// ---- TMA-staged tile step that also forms the order parameters -------------
//
// The phase populations arrive with a 2-node halo (40 x 12 box), so C_i =
// sum_p f^i_p / psi is formed in shared memory for the tile and its halo and
// never goes through HBM; the flow populations and lagged planes arrive for
// the tile only.  At outer walls the f ghost nodes hold mirror copies, so
// the C they give is the mirror image the stencils expect.

// L2 prefetch distance of the fused tile kernel, in quarter waves of
// resident CTAs.
constexpr int kPrefetchQuarterWaves = 3;

template <int NP, bool TF, int TX, int TY>
struct FLay {
    using T = float;   // FP32 alone (the C pass goes by quads)
    static constexpr int NF = 9 * (NP - 1);
    static constexpr int NLAG = 2 * NP + 3;
    static constexpr int NST = TF ? NP : 1;
    static constexpr int HX = TX + 8;                        // halo box columns x0-4 .. x0+TX+3
    static constexpr int HY = TY + 4;
    static constexpr int pad(int e) { return (e * (int)sizeof(T) + 127) / 128 * 128 / (int)sizeof(T); }
    static constexpr int FH_BOX = NF * HY * HX;              // rows y0-2 .. y0+TY+1
    static constexpr int G_BOX = 9 * TY * TX;
    static constexpr int LAG_BOX = NLAG * TY * TX;
    static constexpr int ST_BOX = NST * HY * HX;
    static constexpr int A_BOX = (TY + 2) * HX;
    static constexpr int C_ARR = (NP - 1) * HY * HX;
    static constexpr int MU = NP * (TY + 2) * (TX + 2);
    static constexpr size_t fh_off = 0;
    static constexpr size_t g_off = fh_off + pad(FH_BOX);
    static constexpr size_t lag_off = g_off + pad(G_BOX);
    static constexpr size_t st_off = lag_off + pad(LAG_BOX);
    static constexpr size_t a_off = st_off + pad(ST_BOX);
    static constexpr size_t c_off = a_off + pad(A_BOX);
    static constexpr size_t mu_off = c_off + C_ARR;
    static constexpr size_t end = mu_off + MU;
    static constexpr size_t bar_byte_off = (end * sizeof(T) + 127) / 128 * 128;
    static constexpr size_t bytes = bar_byte_off + 64;
    static constexpr unsigned tx_halo = (unsigned)((FH_BOX + ST_BOX + A_BOX) * sizeof(T));
    static constexpr unsigned tx_tile = (unsigned)((G_BOX + LAG_BOX) * sizeof(T));
};

template <int NP, bool TF, int TX, int TY>
struct FusedAcc {
    using T = float;
    using L = FLay<NP, TF, TX, TY>;
    const KParams<T>& P;
    const T* sm;
    int tx, ty;
    __device__ T C(int j, int dy, int dx) const {
        return sm[L::c_off + ((size_t)j * L::HY + ty + 2 + dy) * L::HX + tx + 4 + dx];
    }
    __device__ T psi(int dy, int dx) const { return sm[L::st_off + (size_t)(ty + 2 + dy) * L::HX + tx + 4 + dx]; }
    __device__ void grad_psi(const KParams<T>& Q, T& gx, T& gy) const {
        dev::grad9(Q, [&](int dy, int dx) { return psi(dy, dx); }, gx, gy);
    }
    __device__ T psi_rho(int dy, int dx) const {
        return dev::psi_rho<T, NP>(P, psi(dy, dx), [&](int j) { return C(j, dy, dx); });
    }
    __device__ T mu(int j, int dy, int dx) const {
        return sm[L::mu_off + ((size_t)j * (TY + 2) + ty + 1 + dy) * (TX + 2) + tx + 1 + dx];
    }
    __device__ T a(int dy, int dx) const { return sm[L::a_off + (size_t)(ty + 1 + dy) * L::HX + tx + 4 + dx]; }
    __device__ T lag(int k) const { return sm[L::lag_off + ((size_t)k * TY + ty) * TX + tx]; }
    __device__ T f(int i, int p) const {
        return sm[L::fh_off + ((size_t)(9 * i + p) * L::HY + ty + 2) * L::HX + tx + 4];
    }
    __device__ T g(int p) const { return sm[L::g_off + ((size_t)p * TY + ty) * TX + tx]; }
};

template <int NP, bool TF, int TX, int TY>
__global__ void __launch_bounds__(TX * TY, 2)
    k_step_fused(const __grid_constant__ CUtensorMap tm_fh, const __grid_constant__ CUtensorMap tm_g,
                 const __grid_constant__ CUtensorMap tm_lag, const __grid_constant__ CUtensorMap tm_st,
                 const __grid_constant__ CUtensorMap tm_a, KParams<float> P, float* __restrict__ pop_out,
                 float* __restrict__ lag_out, int* __restrict__ err, int pf_dist, int off32) {
    using T = float;
    using L = FLay<NP, TF, TX, TY>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem_raw + L::bar_byte_off);
    const int tid = threadIdx.x + TX * threadIdx.y;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    if (tid == 0) {
        tma::mbar_init(&bars[0], 1);
        tma::mbar_init(&bars[1], 1);
        tma::mbar_init_fence();
    }
    __syncthreads();
    // padded coordinates: column x0 - 4 is x0 (kGX = 4), row y is y + kGY
    if (tid == 0) {
        tma::mbar_expect_tx(&bars[0], L::tx_halo);
        tma::load_3d(sm + L::st_off, &tm_st, x0, y0 - 2 + kGY, 0, &bars[0]);   // static planes
    }
    wait_for_previous();
    if (tid == 0) {
        tma::load_3d(sm + L::fh_off, &tm_fh, x0, y0 - 2 + kGY, 0, &bars[0]);
        tma::load_3d(sm + L::a_off, &tm_a, x0, y0 - 1 + kGY, 0, &bars[0]);
        tma::mbar_expect_tx(&bars[1], L::tx_tile);
        tma::load_3d(sm + L::g_off, &tm_g, x0 + kGX, y0 + kGY, 0, &bars[1]);
        tma::load_3d(sm + L::lag_off, &tm_lag, x0 + kGX, y0 + kGY, 0, &bars[1]);
        // the tile pf_dist blocks later in launch order (roughly the CTA that
        // starts a wave of resident CTAs from now) is pulled into L2, so DRAM
        // keeps streaming while the resident CTAs compute
        const int nb = gridDim.x * gridDim.y, b = blockIdx.y * gridDim.x + blockIdx.x + pf_dist;
        if (pf_dist > 0 && b < nb) {
            const int px0 = (b % gridDim.x) * TX, py0 = (b / gridDim.x) * TY;
            tma::prefetch_3d(&tm_fh, px0, py0 - 2 + kGY, 0);
            tma::prefetch_3d(&tm_st, px0, py0 - 2 + kGY, 0);
            tma::prefetch_3d(&tm_g, px0 + kGX, py0 + kGY, 0);
            tma::prefetch_3d(&tm_lag, px0 + kGX, py0 + kGY, 0);
        }
    }
    bool ok = tma::mbar_wait_bounded(&bars[0], 0);
    if (!__syncthreads_and(ok)) {
        // a copy has not landed within the bounded wait: record it, and give
        // every copy still in flight a second bounded wait before the CTA and
        // its shared memory go
        if (tid == 0) {
            atomicOr(err, 1);
            tma::mbar_wait_bounded(&bars[0], 0);
            tma::mbar_wait_bounded(&bars[1], 0);
        }
        return;
    }
    // C_i = sum_p f^i_p / psi on the tile + 2-node halo: four columns of one
    // phase per item as 16-byte accesses over whole box rows, so a warp reads
    // consecutive quads (node by node over the columns needed, every warp
    // spanned two rows and met two-way bank conflicts: 256 x 256, N = 3, 11.0
    // -> 10.3 us a step).
    constexpr int NQ = L::HY * L::HX / 4, PL = L::HY * L::HX;
#pragma unroll
    for (int r = 0; r < ((NP - 1) * NQ + (TX * TY) - 1) / (TX * TY); ++r) {
        const int k = tid + r * (TX * TY);
        if (k < (NP - 1) * NQ) {
            const int i = k / NQ, o = 4 * (k - i * NQ);
            const T* fb = sm + L::fh_off + (size_t)(9 * i) * PL + o;
            float4 c = *reinterpret_cast<const float4*>(fb);
#pragma unroll
            for (int p = 1; p < 9; ++p) {
                const float4 v = *reinterpret_cast<const float4*>(fb + (size_t)p * PL);
                c.x += v.x;
                c.y += v.y;
                c.z += v.z;
                c.w += v.w;
            }
            const float4 ps = *reinterpret_cast<const float4*>(sm + L::st_off + o);
            *reinterpret_cast<float4*>(sm + L::c_off + (size_t)i * PL + o) =
                make_float4(c.x * dev::rcp(ps.x), c.y * dev::rcp(ps.y), c.z * dev::rcp(ps.z),
                            c.w * dev::rcp(ps.w));
        }
    }
    __syncthreads();
    // mu on the tile + 1-node halo
    for (int k = tid; k < (TY + 2) * (TX + 2); k += (TX * TY)) {
        const int ly = k / (TX + 2), lx = k - ly * (TX + 2);
        const T* cb = sm + L::c_off + (size_t)(ly + 1) * L::HX + lx + 3;
        const T* sb = sm + L::st_off + (size_t)(ly + 1) * L::HX + lx + 3;
        T cth[NP];
#pragma unroll
        for (int i = 0; i < NP - 1; ++i)
            cth[i] = TF ? sb[(size_t)(1 + i) * L::HY * L::HX] : P.cos_uni[i];
        T mu[NP];
        dev::chem_pot<T, NP>(
            P, [&](int j, int dy, int dx) { return cb[((size_t)j * L::HY + dy) * L::HX + dx]; },
            [&](int dy, int dx) { return sb[dy * L::HX + dx]; }, cth, mu);
#pragma unroll
        for (int i = 0; i < NP; ++i) sm[L::mu_off + ((size_t)i * (TY + 2) + ly) * (TX + 2) + lx] = mu[i];
    }
    ok = tma::mbar_wait_bounded(&bars[1], 0);
    if (!__syncthreads_and(ok)) {
        if (tid == 0) {
            atomicOr(err, 1);
            tma::mbar_wait_bounded(&bars[1], 0);
        }
        return;
    }
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    const long long o = P.org + (long long)y * P.pitch + x;
    if (fused_writes_rings(TX)) dependents_may_start();
    FusedAcc<NP, TF, TX, TY> acc{P, sm, (int)threadIdx.x, (int)threadIdx.y};
    // most tiles push only into the domain's interior, and (kRings) only to
    // nodes without a copy in the 2-node ghost ring: fixed neighbour offsets,
    // no wrap or bounce-back, 32-bit offsets (a block-uniform branch)
    constexpr bool kRings = fused_writes_rings(TX);
    constexpr int kIn = kRings ? 3 : 1;
    if (off32 && x0 >= kIn && y0 >= kIn && x0 + TX + kIn <= P.nx && y0 + TY + kIn <= P.ny) {
        InnerSink<T, NP> in{pop_out + o, lag_out + o, (int)P.plane, P.pitch};
        dev::node_update<T, NP, 0>(P, acc, in);
        return;
    }
    if constexpr (!kRings) {
        TileSink<T, NP> sink;
        sink.o = o;
        sink.plane = P.plane;
        sink.fout = pop_out;
        sink.gout = pop_out + (long long)9 * (NP - 1) * P.plane;
        sink.lout = lag_out;
        sink.macro_out = nullptr;
        tile_targets(P, x, y, o, sink);
        dev::node_update<T, NP, 0>(P, acc, sink);
        return;
    }
    EdgeSink<T, NP> sink;
    sink.o = o;
    sink.plane = P.plane;
    sink.pitch = P.pitch;
    sink.pop = pop_out;
    sink.lag = lag_out;
    sink.bounced = 0;
    int tx[3], ty[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        tx[d] = x + d - 1;
        ty[d] = y + d - 1;
        if (P.px) tx[d] = tx[d] < 0 ? tx[d] + P.nx : tx[d] >= P.nx ? tx[d] - P.nx : tx[d];
        if (P.py) ty[d] = ty[d] < 0 ? ty[d] + P.ny : ty[d] >= P.ny ? ty[d] - P.ny : ty[d];
        sink.dx[d] = ring2_step(tx[d], P.nx, P.px);
        sink.dy[d] = ring2_step(ty[d], P.ny, P.py);
    }
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        const int X = tx[cxp(p) + 1], Y = ty[cyp(p) + 1];
        const bool bounce = X < 0 || X >= P.nx || Y < 0 || Y >= P.ny;
        sink.bounced |= (unsigned)bounce << p;
        sink.tgt[p] = bounce ? opposite(p) * P.plane + o
                             : p * P.plane + P.org + (long long)Y * P.pitch + X;
    }
    dev::node_update<T, NP, 0>(P, acc, sink);
}

template <int NP, bool TF, int TX, int TY>
cudaError_t collide_fused_n(const TileTmaArgs<float>& a, cudaStream_t s) {
    using L = FLay<NP, TF, TX, TY>;
    const cudaError_t e = cudaFuncSetAttribute(k_step_fused<NP, TF, TX, TY>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::bytes);
    if (e != cudaSuccess) return e;
    const KParams<float>& kp = *a.kp;
    int sms = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        sms = 0;   // no prefetch
    // a wave of resident CTAs (two per SM) ahead
    const int pf_dist = kPrefetchQuarterWaves * sms * 2 / 4;
    // the inner tiles' 32-bit offsets reach every population and lagged plane
    const int off32 = (long long)(9 * NP) * kp.plane < (1LL << 31) ? 1 : 0;
    // the next step may start early where the whole step is short: 256 x 256, N =
    // 3, 8.1 us a step without, 7.4 with (4096 x 4096, N = 4: 1179 and 1185)
    return launch_dependent(fused_writes_rings(TX), k_step_fused<NP, TF, TX, TY>, dim3((kp.nx + TX - 1) / TX, (kp.ny + TY - 1) / TY),
                            dim3(TX, TY), L::bytes, s, *a.tm_pop, *a.tm_g, *a.tm_lag, *a.tm_st, *a.tm_a, kp, a.pop_out,
                            a.lag_out, a.err, pf_dist, off32);
}

template <typename T, int NP, bool TF>
cudaError_t collide_tma_n(const TileTmaArgs<T>& a, cudaStream_t s) {
    using L = TLay<T, NP, TF>;
    const cudaError_t e = cudaFuncSetAttribute(k_step_tma<T, NP, TF>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::bytes);
    if (e != cudaSuccess) return e;
    const KParams<T>& kp = *a.kp;
    k_step_tma<T, NP, TF><<<dim3((kp.nx + BX - 1) / BX, (kp.ny + BY - 1) / BY), dim3(BX, BY), L::bytes, s>>>(
        *a.tm_pop, *a.tm_lag, *a.tm_c, *a.tm_st, *a.tm_a, kp, a.pop_out, a.lag_out, a.err);
    return cudaGetLastError();
}

// Initial state (reading of the paper's set-ups): f = f^eq(C0, mu(C0), u = 0)
// by Eq. 3.5, g = g^eq(P = 0, u = 0) by Eq. 3.8 (g_0 - rho0 = 0), lagged
// fields zero.  F.C holds C0.
template <typename T, int NP>
__global__ void __launch_bounds__(NT) k_init(KParams<T> P, Fields<T> F, int cur) {
    __shared__ Smem<T, NP> sm;
    const int tid = threadIdx.x + BX * threadIdx.y;
    const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY;
    load_tile<T, NP>(P, sm, F.C, F.psi, F.cosf, nullptr, x0, y0, tid);
    __syncthreads();
    compute_mu_tile<T, NP>(P, sm, tid);
    __syncthreads();
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    const long long o = P.org + (long long)y * P.pitch + x;
    const T psi = sm.psi[threadIdx.y + 2][threadIdx.x + 2];
    T* f = cur ? F.f[1] : F.f[0];
    const T w0 = P.w1d[1] * P.w1d[1];
#pragma unroll
    for (int i = 0; i < NP - 1; ++i) {
        const T psiC = psi * sm.C[i][threadIdx.y + 2][threadIdx.x + 2];
        const T emu = P.eta[i] * psi * sm.mu[i][threadIdx.y + 1][threadIdx.x + 1];
#pragma unroll
        for (int p = 0; p < 9; ++p) {
            const T wp = P.w1d[kCx[p] + 1] * P.w1d[kCy[p] + 1];
            f[(i * 9 + p) * P.plane + o] = p == 0 ? (w0 - T(1)) * emu + psiC : wp * emu;
        }
    }
    T* g = cur ? F.g[1] : F.g[0];
#pragma unroll
    for (int p = 0; p < 9; ++p) g[p * P.plane + o] = T(0);
    T* lag = cur ? F.lag[1] : F.lag[0];
    for (int q = 0; q < 2 * NP + 3; ++q) lag[q * P.plane + o] = T(0);
}

// psi C_i = sum_p f^i_p and C_i = psi C_i / psi (Sec. 3).
template <typename T, int NP>
__global__ void __launch_bounds__(256) k_order_param(KParams<T> P, const T* __restrict__ f,
                                                     const T* __restrict__ psi, T* __restrict__ C) {
    const long long n = (long long)P.nx * P.ny;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int y = (int)(idx / P.nx), x = (int)(idx - (long long)y * P.nx);
        const long long o = P.org + (long long)y * P.pitch + x;
        const T inv = dev::rcp(psi[o]);
#pragma unroll
        for (int i = 0; i < NP - 1; ++i) {
            T s = T(0);
#pragma unroll
            for (int p = 0; p < 9; ++p) s += f[(i * 9 + p) * P.plane + o];
            C[i * P.plane + o] = s * inv;
        }
    }
}

// Per-phase sum over nodes of sum_p f^i_p in double, fixed order:
// pass 1 writes one partial per block, pass 2 sums them.
template <typename T, int NP>
__global__ void __launch_bounds__(256) k_mass_partial(KParams<T> P, const T* __restrict__ f,
                                                      double* __restrict__ partial) {
    __shared__ double red[NP - 1][256];
    const long long n = (long long)P.nx * P.ny;
    double acc[NP - 1];
#pragma unroll
    for (int i = 0; i < NP - 1; ++i) acc[i] = 0.0;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int y = (int)(idx / P.nx), x = (int)(idx - (long long)y * P.nx);
        const long long o = P.org + (long long)y * P.pitch + x;
#pragma unroll
        for (int i = 0; i < NP - 1; ++i) {
            double s = 0.0;
#pragma unroll
            for (int p = 0; p < 9; ++p) s += (double)f[(i * 9 + p) * P.plane + o];
            acc[i] += s;
        }
    }
#pragma unroll
    for (int i = 0; i < NP - 1; ++i) red[i][threadIdx.x] = acc[i];
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) {
#pragma unroll
            for (int i = 0; i < NP - 1; ++i) red[i][threadIdx.x] += red[i][threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
#pragma unroll
        for (int i = 0; i < NP - 1; ++i) partial[blockIdx.x * kMaxPhases + i] = red[i][0];
    }
}

// One warp per phase: each lane sums every 32nd partial, then the lanes are
// summed in a fixed order (one thread per phase adding all 304 took 26 us).
__global__ void k_mass_final(const double* __restrict__ partial, int nblocks, int nph,
                             double* __restrict__ out) {
    const int lane = threadIdx.x % 32, ph = threadIdx.x / 32;
    if (ph >= nph) return;
    double s = 0.0;
    for (int b = lane; b < nblocks; b += 32) s += partial[b * kMaxPhases + ph];
    for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
    if (lane == 0) out[ph] = s;
}

template <typename T>
__global__ void k_convert(const double* __restrict__ src, T* __restrict__ dst, KParams<T> P,
                          int planes) {
    const long long n = (long long)P.nx * P.ny;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n * planes;
         idx += (long long)gridDim.x * blockDim.x) {
        const long long q = idx / n, r = idx - q * n;
        const int y = (int)(r / P.nx), x = (int)(r - (long long)y * P.nx);
        dst[q * P.plane + P.org + (long long)y * P.pitch + x] = (T)src[idx];
    }
}

// `planes` consecutive planes to dense doubles, plane after plane (grid y).
template <typename T>
__global__ void k_export(const T* __restrict__ src, double* __restrict__ dst, KParams<T> P) {
    const long long n = (long long)P.nx * P.ny;
    src += blockIdx.y * P.plane;
    dst += blockIdx.y * n;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int y = (int)(idx / P.nx), x = (int)(idx - (long long)y * P.nx);
        dst[idx] = (double)src[P.org + (long long)y * P.pitch + x];
    }
}

// Ghost frame: every cell of [-kGX, nx + kGX) x [-kGY, ny + kGY) outside
// the domain takes the value of its periodic image or wall mirror.  The
// cells are enumerated as 2 kGY full-width ghost rows, then 2 kGX ghost
// columns of the ny domain rows.
template <typename T>
__global__ void k_fill_ghosts(GhostRing<T> g0, GhostRing<T> g1, KParams<T> P) {
    // one ghost cell per thread, plane blockIdx.y of ring g0 and then of
    // ring g1: first the 2 gy full rows (corners included), then the 2 gx
    // side columns of the ny interior rows, grouped by row so that a row's
    // side cells are neighbours in a warp.  Every source is an interior
    // node, so the cells are independent.
    const bool second = (int)blockIdx.y >= g0.planes;
    const int gx = second ? g1.gx : g0.gx, gy = second ? g1.gy : g0.gy;
    const int W = P.nx + 2 * gx;
    const int nrow = 2 * gy * W, ncol = 2 * gx * P.ny;
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nrow + ncol) return;
    int X, Y;
    if (r < nrow) {
        const int k = r / W;
        X = r - k * W - gx;
        Y = k < gy ? k - gy : P.ny + (k - gy);
    } else {
        const int c = r - nrow;
        Y = c / (2 * gx);
        const int k = c - Y * (2 * gx);
        X = k < gx ? k - gx : P.nx + (k - gx);
    }
    const int sx = map_index(X, P.nx, P.px), sy = map_index(Y, P.ny, P.py);
    T* pl = second ? g1.base + (long long)((int)blockIdx.y - g0.planes) * P.plane
                   : g0.base + (long long)blockIdx.y * P.plane;
    pl[P.org + (long long)Y * P.pitch + X] = pl[P.org + (long long)sy * P.pitch + sx];
}

// Open x ends: equilibrium at (u_in(y), 0) with mu = 0 and m^C = 0 (Eqs. 3.5,
// 3.8); C = C_in at the inlet, the neighbour column's at the outlet; psi P
// from the neighbour column by Eq. 19 without its velocity terms.  A thread
// has one population set (phase i, or the flow and the remaining lagged
// planes) of one end node, in blocks of one warp: the launch is a chain of
// dependent loads and is bound by their latency.  Phase populations and plane
// a go to the node's copies in the 2-node ghost ring too.
constexpr int kOpenThreads = 32;
template <typename T, int NP>
__global__ void __launch_bounds__(kOpenThreads) k_open_bc(KParams<T> P, T* pop, T* lag,
                                                          const T* __restrict__ psi, const T* __restrict__ inflow) {
    dependents_may_start();
    wait_for_previous();
    const int idx = blockIdx.x * kOpenThreads + threadIdx.x;
    const int end = idx % (2 * P.ny), set = idx / (2 * P.ny);
    if (set >= NP) return;
    const int side = end / P.ny, y = end - side * P.ny;
    const int xb = side ? P.nx - 1 : 0, xn = side ? P.nx - 2 : 1;
    const long long pl = P.plane;
    const long long ob = P.org + (long long)y * P.pitch + xb, on = P.org + (long long)y * P.pitch + xn;
    const int sx = ring2_step(xb, P.nx, 0);
    const long long sy = (long long)ring2_step(y, P.ny, P.py) * P.pitch;
    auto put = [&](T* q, T v) {
        q[ob] = v;
        q[ob + sx] = v;
        if (sy) {
            q[ob + sy] = v;
            q[ob + sy + sx] = v;
        }
    };
    const T psib = psi[ob], psin = psi[on];
    const T u = inflow[y];
    const T cs2 = P.cs2;
    auto fraction = [&](int j) {
        if (side == 0) return inflow[(1 + j) * P.ny + y];
        T v[9], sf = T(0);
#pragma unroll
        for (int p = 0; p < 9; ++p) v[p] = pop[(9 * j + p) * pl + on];
#pragma unroll
        for (int p = 0; p < 9; ++p) sf += v[p];
        return sf / psin;
    };
    if (set < NP - 1) {
        // phase: f_0 = psi C, f_p = w_p psi C c_p.u / cs2
        const T psiC = psib * fraction(set);
        const T fa = P.w9[1] * psiC * u / cs2, fd = P.w9[2] * psiC * u / cs2;
#pragma unroll
        for (int p = 0; p < 9; ++p) {
            const T m = p <= 4 ? fa : fd;
            put(pop + (9 * set + p) * pl, p == 0 ? psiC : cxp(p) > 0 ? m : cxp(p) < 0 ? -m : T(0));
        }
        lag[(1 + 2 * set) * pl + ob] = psiC * u;
        lag[(2 + 2 * set) * pl + ob] = T(0);
        return;
    }
    T* g = pop + (long long)9 * (NP - 1) * pl;
    T gn[9], sum_g = T(0);
#pragma unroll
    for (int p = 1; p < 9; ++p) gn[p] = g[p * pl + on];
    const T pmn = lag[(2 * NP + 2) * pl + on];
    T rho = T(0), sC = T(0);
#pragma unroll
    for (int j = 0; j < NP - 1; ++j) {
        const T c = fraction(j);
        sC += c;
        rho += c * P.rho[j];
    }
    rho += (T(1) - sC) * P.rho[NP - 1];
#pragma unroll
    for (int p = 1; p < 9; ++p) sum_g += gn[p];
    const T psiP = psib * (P.cP * (sum_g - P.Kh * pmn) / psin);
    // flow: g_p = w_p psi P / cs2 + s_p (g_0 stored less rho0), s_p of the
    // resting-solid-free equilibrium with m^C = 0
    const T Axx = psib * rho * u * u;
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        const T wp = P.w9[p == 0 ? 0 : p <= 4 ? 1 : 2];
        const T cx = T(cxp(p));
        const T sp = wp * (cx * psib * rho * u / cs2 + Axx * (cx * cx - cs2) / (cs2 - cs2 * cs2));
        g[p * pl + ob] = (p == 0 ? (wp - T(1)) : wp) * psiP / cs2 + sp;
    }
    put(lag, T(0));
    lag[(2 * NP - 1) * pl + ob] = T(0);
    lag[(2 * NP) * pl + ob] = T(0);
    lag[(2 * NP + 1) * pl + ob] = T(0);
    lag[(2 * NP + 2) * pl + ob] = psib * rho * u * u;
}

template <typename T>
__global__ void k_walls_init(KParams<T> P, T* __restrict__ psi, T* __restrict__ e) {
    const long long n = (long long)P.nx * P.ny;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int y = (int)(idx / P.nx), x = (int)(idx - (long long)y * P.nx);
        const long long o = P.org + (long long)y * P.pitch + x;
        psi[o] = T(1);
        for (int j = 0; j < P.N - 1; ++j) e[j * P.plane + o] = T(0);
    }
}

// psi *= psi_k; e_j += cos(theta^k_jN) |grad psi_k| (the gradient stencil of
// the step, on psi_k with its ghost frame).
template <typename T>
__global__ void k_wall_accumulate(KParams<T> P, const T* __restrict__ stage, T* __restrict__ psi,
                                  T* __restrict__ e) {
    const long long n = (long long)P.nx * P.ny;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int y = (int)(idx / P.nx), x = (int)(idx - (long long)y * P.nx);
        const long long o = P.org + (long long)y * P.pitch + x;
        T gx, gy;
        dev::grad9(P, [&](int dy, int dx) { return stage[o + (long long)dy * P.pitch + dx]; }, gx, gy);
        const T ag = sqrt(gx * gx + gy * gy);
        psi[o] = psi[o] * stage[o];
        for (int j = 0; j < P.N - 1; ++j) e[j * P.plane + o] += stage[(1 + j) * P.plane + o] * ag;
    }
}

__global__ void k_store(long long* dst, long long v) { *dst = v; }

inline dim3 tile_grid(int nx, int ny) {
    return dim3((nx + BX - 1) / BX, (ny + BY - 1) / BY);
}

inline int flat_blocks(long long n) {
    long long b = (n + 255) / 256;
    return (int)(b < 152 * 16 ? (b < 1 ? 1 : b) : 152 * 16);
}

template <typename T, int NP>
cudaError_t order_param_n(const KParams<T>& kp, const Fields<T>& fd, int cur, cudaStream_t s) {
    k_order_param<T, NP><<<flat_blocks((long long)kp.nx * kp.ny), 256, 0, s>>>(kp, fd.f[cur], fd.psi, fd.C);
    return cudaGetLastError();
}

template <typename T, int NP>
cudaError_t collide_n(const KParams<T>& kp, const Fields<T>& fd, int cur, cudaStream_t s) {
    k_step<T, NP, 0><<<tile_grid(kp.nx, kp.ny), dim3(BX, BY), 0, s>>>(kp, fd, cur);
    return cudaGetLastError();
}

template <typename T, int NP>
cudaError_t macro_n(const KParams<T>& kp, const Fields<T>& fd, int cur, cudaStream_t s) {
    k_order_param<T, NP><<<flat_blocks((long long)kp.nx * kp.ny), 256, 0, s>>>(kp, fd.f[cur], fd.psi, fd.C);
    k_step<T, NP, 1><<<tile_grid(kp.nx, kp.ny), dim3(BX, BY), 0, s>>>(kp, fd, cur);
    return cudaGetLastError();
}

template <typename T, int NP>
cudaError_t init_n(const KParams<T>& kp, const Fields<T>& fd, int cur, cudaStream_t s) {
    k_init<T, NP><<<tile_grid(kp.nx, kp.ny), dim3(BX, BY), 0, s>>>(kp, fd, cur);
    return cudaGetLastError();
}

template <typename T, int NP>
cudaError_t mass_n(const KParams<T>& kp, const Fields<T>& fd, int cur, double* out, cudaStream_t s) {
    k_mass_partial<T, NP><<<kMassBlocks, 256, 0, s>>>(kp, fd.f[cur], fd.partial);
    k_mass_final<<<1, 32 * (NP - 1), 0, s>>>(fd.partial, kMassBlocks, NP - 1, out);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_store(long long* dst, long long v, cudaStream_t s) {
    k_store<<<1, 1, 0, s>>>(dst, v);
    return cudaGetLastError();
}

#define DDCC_DISPATCH(fn, ...)                                \
    switch (kp.N) {                                           \
        case 2: return fn<T, 2>(__VA_ARGS__);                 \
        case 3: return fn<T, 3>(__VA_ARGS__);                 \
        case 4: return fn<T, 4>(__VA_ARGS__);                 \
        default: return cudaErrorInvalidValue;                \
    }

template <typename T>
cudaError_t launch_init(const KParams<T>& kp, const Fields<T>& fd, int cur, cudaStream_t s) {
    DDCC_DISPATCH(init_n, kp, fd, cur, s);
}
template <typename T>
cudaError_t launch_order_param(const KParams<T>& kp, const Fields<T>& fd, int cur, cudaStream_t s) {
    DDCC_DISPATCH(order_param_n, kp, fd, cur, s);
}
template <typename T>
cudaError_t launch_collide(const KParams<T>& kp, const Fields<T>& fd, int cur, cudaStream_t s) {
    DDCC_DISPATCH(collide_n, kp, fd, cur, s);
}
template <typename T>
cudaError_t launch_macro(const KParams<T>& kp, const Fields<T>& fd, int cur, cudaStream_t s) {
    DDCC_DISPATCH(macro_n, kp, fd, cur, s);
}
template <typename T>
cudaError_t launch_mass(const KParams<T>& kp, const Fields<T>& fd, int cur, double* out,
                        cudaStream_t s) {
    DDCC_DISPATCH(mass_n, kp, fd, cur, out, s);
}
template <typename T>
size_t tile_tma_smem_bytes(int N, bool tf) {
    switch (N * 2 + (tf ? 1 : 0)) {
        case 4: return TLay<T, 2, false>::bytes;
        case 5: return TLay<T, 2, true>::bytes;
        case 6: return TLay<T, 3, false>::bytes;
        case 7: return TLay<T, 3, true>::bytes;
        case 8: return TLay<T, 4, false>::bytes;
        case 9: return TLay<T, 4, true>::bytes;
        default: return 0;
    }
}
// The fused kernel's tile: 32 x 8 or 64 x 4 (see fused_tile_wide).
template <int TX, int TY>
size_t fused_smem_shape(int N, bool tf) {
    switch (N * 2 + (tf ? 1 : 0)) {
        case 4: return FLay<2, false, TX, TY>::bytes;
        case 5: return FLay<2, true, TX, TY>::bytes;
        case 6: return FLay<3, false, TX, TY>::bytes;
        case 7: return FLay<3, true, TX, TY>::bytes;
        case 8: return FLay<4, false, TX, TY>::bytes;
        case 9: return FLay<4, true, TX, TY>::bytes;
        default: return 0;
    }
}
template <typename T>
size_t tile_fused_smem_bytes(int N, bool tf, bool wide) {
    return wide ? fused_smem_shape<kWideX, kWideY>(N, tf) : fused_smem_shape<BX, BY>(N, tf);
}
template <int TX, int TY>
cudaError_t fused_shape(const TileTmaArgs<float>& a, cudaStream_t s) {
    const bool tf = a.kp->has_cos_field != 0;
    switch (a.kp->N * 2 + (tf ? 1 : 0)) {
        case 4: return collide_fused_n<2, false, TX, TY>(a, s);
        case 5: return collide_fused_n<2, true, TX, TY>(a, s);
        case 6: return collide_fused_n<3, false, TX, TY>(a, s);
        case 7: return collide_fused_n<3, true, TX, TY>(a, s);
        case 8: return collide_fused_n<4, false, TX, TY>(a, s);
        case 9: return collide_fused_n<4, true, TX, TY>(a, s);
        default: return cudaErrorInvalidValue;
    }
}
template <typename T>
cudaError_t launch_collide_fused(const TileTmaArgs<T>& a, cudaStream_t s) {
    return a.wide ? fused_shape<kWideX, kWideY>(a, s) : fused_shape<BX, BY>(a, s);
}
template <typename T>
cudaError_t launch_collide_tma(const TileTmaArgs<T>& a, cudaStream_t s) {
    const bool tf = a.kp->has_cos_field != 0;
    switch (a.kp->N * 2 + (tf ? 1 : 0)) {
        case 4: return collide_tma_n<T, 2, false>(a, s);
        case 5: return collide_tma_n<T, 2, true>(a, s);
        case 6: return collide_tma_n<T, 3, false>(a, s);
        case 7: return collide_tma_n<T, 3, true>(a, s);
        case 8: return collide_tma_n<T, 4, false>(a, s);
        case 9: return collide_tma_n<T, 4, true>(a, s);
        default: return cudaErrorInvalidValue;
    }
}
template <typename T>
cudaError_t launch_convert(const double* src, T* dst, const KParams<T>& kp, int planes,
                           cudaStream_t s) {
    k_convert<T><<<flat_blocks((long long)kp.nx * kp.ny * planes), 256, 0, s>>>(src, dst, kp, planes);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_export(const T* src, double* dst, const KParams<T>& kp, int planes, cudaStream_t s) {
    k_export<T><<<dim3(flat_blocks((long long)kp.nx * kp.ny), planes), 256, 0, s>>>(src, dst, kp);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_fill_ghosts2(const GhostRing<T>& g0, const GhostRing<T>& g1, const KParams<T>& kp,
                                cudaStream_t s) {
    long long n = 0;   // cells per plane of the larger ring
    for (const GhostRing<T>* g : {&g0, &g1}) {
        if (g->planes < 0 || g->gx < 0 || g->gx > kGX || g->gy < 0 || g->gy > kGY) return cudaErrorInvalidValue;
        if (g->planes > 0) {
            if (!g->base) return cudaErrorInvalidValue;
            n = std::max(n, 2LL * g->gy * (kp.nx + 2 * g->gx) + 2LL * g->gx * kp.ny);
        }
    }
    const long long planes = (long long)g0.planes + g1.planes;
    if (n == 0 || planes == 0) return cudaSuccess;
    if (planes > 65535 || n > (1LL << 31) - 256) return cudaErrorInvalidValue;
    k_fill_ghosts<T><<<dim3((unsigned)((n + 255) / 256), (unsigned)planes), 256, 0, s>>>(g0, g1, kp);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_fill_ghosts(T* base, int planes, const KParams<T>& kp, cudaStream_t s, int gx, int gy) {
    return launch_fill_ghosts2<T>(GhostRing<T>{base, planes, gx, gy}, GhostRing<T>{nullptr, 0, 0, 0}, kp, s);
}

template <typename T, int NP>
cudaError_t open_bc_n(const KParams<T>& kp, T* pop, T* lag, const T* psi, const T* inflow, cudaStream_t s) {
    return launch_dependent(sizeof(T) == 4, k_open_bc<T, NP>, dim3((2 * kp.ny * NP + kOpenThreads - 1) / kOpenThreads), dim3(kOpenThreads),
                            0, s, kp, pop, lag, psi, inflow);
}
template <typename T>
cudaError_t launch_open_bc(const KParams<T>& kp, T* pop, T* lag, const T* psi, const T* inflow,
                           cudaStream_t s) {
    DDCC_DISPATCH(open_bc_n, kp, pop, lag, psi, inflow, s);
}

template <typename T>
cudaError_t launch_walls_init(const KParams<T>& kp, T* psi, T* e, cudaStream_t s) {
    k_walls_init<T><<<flat_blocks((long long)kp.nx * kp.ny), 256, 0, s>>>(kp, psi, e);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_wall_accumulate(const KParams<T>& kp, const T* stage, T* psi, T* e, cudaStream_t s) {
    k_wall_accumulate<T><<<flat_blocks((long long)kp.nx * kp.ny), 256, 0, s>>>(kp, stage, psi, e);
    return cudaGetLastError();
}

#define DDCC_INSTANTIATE(T)                                                                      \
    template cudaError_t launch_init<T>(const KParams<T>&, const Fields<T>&, int, cudaStream_t);  \
    template cudaError_t launch_mass<T>(const KParams<T>&, const Fields<T>&, int, double*,        \
                                        cudaStream_t);                                           \
    template cudaError_t launch_convert<T>(const double*, T*, const KParams<T>&, int, cudaStream_t); \
    template cudaError_t launch_export<T>(const T*, double*, const KParams<T>&, int, cudaStream_t); \
    template cudaError_t launch_fill_ghosts<T>(T*, int, const KParams<T>&, cudaStream_t, int, int);         \
    template cudaError_t launch_walls_init<T>(const KParams<T>&, T*, T*, cudaStream_t);          \
    template cudaError_t launch_open_bc<T>(const KParams<T>&, T*, T*, const T*, const T*, cudaStream_t); \
    template cudaError_t launch_wall_accumulate<T>(const KParams<T>&, const T*, T*, T*, cudaStream_t);

DDCC_INSTANTIATE(double)
DDCC_INSTANTIATE(float)

// the tile step and its read-out run in FP32; FP64 has its own (ddcc_fp64.cu)
template cudaError_t launch_order_param<float>(const KParams<float>&, const Fields<float>&, int, cudaStream_t);
template cudaError_t launch_collide<float>(const KParams<float>&, const Fields<float>&, int, cudaStream_t);
template cudaError_t launch_macro<float>(const KParams<float>&, const Fields<float>&, int, cudaStream_t);
template cudaError_t launch_fill_ghosts2<float>(const GhostRing<float>&, const GhostRing<float>&, const KParams<float>&,
                                                cudaStream_t);
template size_t tile_tma_smem_bytes<float>(int, bool);
template size_t tile_fused_smem_bytes<float>(int, bool, bool);
template cudaError_t launch_collide_fused<float>(const TileTmaArgs<float>&, cudaStream_t);
template cudaError_t launch_collide_tma<float>(const TileTmaArgs<float>&, cudaStream_t);

}  // namespace ddcc
