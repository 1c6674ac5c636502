// The FP64 step of the 2D path, as two kernels over plain loads:
//   k_fields64  C_i = sum_p f^i_p / psi, psi rho and mu_i (Eq. 2.14) -> planes
//   k_update64  the node update (dev::node_update) from those planes, and the
//               macroscopic read-out in its MODE 1
// GB300 takes 64 cycles per sub-partition for an FP64 warp instruction (add,
// multiply and fused multiply-add alike, also for a warp with one active
// lane), so the step is bound by the number of FP64 warp instructions and
// by how evenly the warps cover the 608 sub-partitions; memory is idle (the
// step moves under a tenth of the bandwidth).  Hence:
//  * C, psi rho and mu are formed once per node and go through memory (L2 for
//    the smaller grids); the one-kernel tile formed C on 1.7 and mu on 1.3
//    nodes per node of its 32 x 8 tile;
//  * what depends on psi alone (1 / psi, grad psi, 3 |grad psi|) is formed once
//    at create and kept as planes;
//  * k_update64 numbers the nodes row by row and gives each thread one, in
//    blocks of two warps: no lane is spent on tile padding, no shared memory
//    limits the blocks per SM, and a small grid still reaches every SM (64 x 64
//    nodes are 64 blocks; as 32 x 8 tiles they were 16, on 16 SMs);
//  * neighbours are addressed by wrapped or mirrored indices (integer work is
//    free beside the FP64 pipe), so no ghost frame is read; the one-node
//    ghost ring of the lagged plane a, which the reverse step reads, is
//    written along with the plane.
// A 32 x 8 tile in one kernel took 511 us a step at 512 x 512, N = 4, and 40 at
// 64 x 64, N = 2, this pair 440 and 20, and with one rate for the phases'
// higher moments (relax_one_rate) 396 and 16.  With one rate a node of four
// phases takes 763 FP64 instructions (by the transforms 28 a phase more), and
// at 1024 x 1024 the two kernels run them at the rate that independent chains
// of multiply-adds reach (ddcc_measure_fp64_peak): 1.51 ms a step.
#include "ddcc_device.cuh"

namespace ddcc {
namespace {

using dev::map_index;
using dev::ring_step;
using Real = double;

constexpr int FX = 32, FY = 4, FT = FX * FY;   // threads (and nodes) of k_fields64
constexpr int UT = 64;                         // threads of k_update64

// static planes, one after the other
enum { kInvPsi, kGradX, kGradY, kAgp3, kStaticPlanes };

__device__ constexpr int vx(int p) { return (p == 1 || p == 5 || p == 8) ? 1 : (p == 3 || p == 6 || p == 7) ? -1 : 0; }
__device__ constexpr int vy(int p) { return (p == 2 || p == 5 || p == 6) ? 1 : (p == 4 || p == 7 || p == 8) ? -1 : 0; }
__device__ constexpr int vopp(int p) { return p == 0 ? 0 : (p <= 4 ? ((p + 1) & 3) + 1 : ((p - 3) & 3) + 5); }

// psi with its ghost frame filled
__global__ void k_static64(KParams<Real> P, const Real* __restrict__ psi, Real* __restrict__ st) {
    const long long n = (long long)P.nx * P.ny;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int y = (int)(i / P.nx), x = (int)(i - (long long)y * P.nx);
        const long long o = P.org + (long long)y * P.pitch + x;
        Real gx, gy;
        dev::grad9(P, [&](int dy, int dx) { return psi[o + (long long)dy * P.pitch + dx]; }, gx, gy);
        st[kInvPsi * P.plane + o] = 1.0 / psi[o];
        st[kGradX * P.plane + o] = gx;
        st[kGradY * P.plane + o] = gy;
        // with several solids the angle planes already carry |grad psi_k|
        st[kAgp3 * P.plane + o] = P.wet_field ? 3.0 : 3.0 * sqrt(gx * gx + gy * gy);
    }
}

// C on the block's 32 x 4 nodes and one node around them in shared memory,
// mu on the nodes.
template <int NP>
__global__ void __launch_bounds__(FT) k_fields64(KParams<Real> P, const Real* __restrict__ f,
                                                 const Real* __restrict__ psi, const Real* __restrict__ st,
                                                 const Real* __restrict__ cosf, Real* __restrict__ C,
                                                 Real* __restrict__ chi, Real* __restrict__ mu, int tiles_x) {
    constexpr int W = FX + 2, H = FY + 2;
    __shared__ Real sC[NP - 1][H][W], sP[H][W];
    const int tid = threadIdx.x;
    const int x0 = (blockIdx.x % tiles_x) * FX, y0 = (blockIdx.x / tiles_x) * FY;
    // all the loads of a thread before the first use of one, so that they are
    // in flight together (beyond the last ring node they repeat it)
    constexpr int R = (H * W + FT - 1) / FT, NF = 9 * (NP - 1);
    Real v[R][NF], inv[R], ps[R];
    long long o_[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int k = min(tid + r * FT, H * W - 1), ly = k / W, lx = k - ly * W;
        const int X = min(x0 + lx - 1, P.nx), Y = min(y0 + ly - 1, P.ny);
        const long long o = o_[r] = P.org + (long long)map_index(Y, P.ny, P.py) * P.pitch + map_index(X, P.nx, P.px);
        inv[r] = st[kInvPsi * P.plane + o];
        ps[r] = psi[o];
#pragma unroll
        for (int q = 0; q < NF; ++q) v[r][q] = f[q * P.plane + o];
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int k = min(tid + r * FT, H * W - 1), ly = k / W, lx = k - ly * W;
        Real c[NP - 1];
#pragma unroll
        for (int i = 0; i < NP - 1; ++i) {
            Real s = v[r][9 * i];
#pragma unroll
            for (int p = 1; p < 9; ++p) s += v[r][9 * i + p];
            sC[i][ly][lx] = c[i] = s * inv[r];
        }
        sP[ly][lx] = ps[r];
        if (lx >= 1 && lx <= FX && ly >= 1 && ly <= FY && x0 + lx - 1 < P.nx && y0 + ly - 1 < P.ny) {
#pragma unroll
            for (int i = 0; i < NP - 1; ++i) C[i * P.plane + o_[r]] = c[i];
            chi[o_[r]] = dev::psi_rho<Real, NP>(P, ps[r], [&](int j) { return c[j]; });
        }
    }
    __syncthreads();
    const int tx = tid % FX, ty = tid / FX, x = x0 + tx, y = y0 + ty;
    if (x >= P.nx || y >= P.ny) return;
    const long long o = P.org + (long long)y * P.pitch + x;
    Real cth[NP], m[NP];
#pragma unroll
    for (int i = 0; i < NP - 1; ++i) cth[i] = P.has_cos_field ? cosf[i * P.plane + o] : P.cos_uni[i];
    dev::chem_pot_with<Real, NP>(
        P, [&](int j, int dy, int dx) { return sC[j][ty + 1 + dy][tx + 1 + dx]; },
        [&](int dy, int dx) { return sP[ty + 1 + dy][tx + 1 + dx]; }, cth, st[kAgp3 * P.plane + o],
        st[kInvPsi * P.plane + o], m);
#pragma unroll
    for (int i = 0; i < (NP == 2 ? 1 : NP); ++i) mu[i * P.plane + o] = m[i];   // N = 2: mu_2 = -mu_1
}

template <int NP>
struct Acc64 {
    const Real *C_, *chi_, *mu_, *psi_, *st_, *pop_, *lag_;
    long long plane, o;
    long long row[3];   // offsets of rows y-1, y, y+1
    int col[3];         // columns x-1, x, x+1
    __device__ long long at(int dy, int dx) const { return row[dy + 1] + col[dx + 1]; }
    __device__ Real C(int j, int dy, int dx) const { return __ldg(C_ + j * plane + at(dy, dx)); }
    __device__ Real psi(int, int) const { return __ldg(psi_ + o); }   // the node's own only
    __device__ Real psi_rho(int dy, int dx) const { return __ldg(chi_ + at(dy, dx)); }
    __device__ void grad_psi(const KParams<Real>&, Real& gx, Real& gy) const {
        gx = __ldg(st_ + kGradX * plane + o);
        gy = __ldg(st_ + kGradY * plane + o);
    }
    __device__ Real mu(int j, int dy, int dx) const { return __ldg(mu_ + j * plane + at(dy, dx)); }
    __device__ Real a(int dy, int dx) const { return __ldg(lag_ + at(dy, dx)); }
    __device__ Real lag(int k) const { return __ldg(lag_ + k * plane + o); }
    __device__ Real f(int i, int p) const { return __ldg(pop_ + (9 * i + p) * plane + o); }
    __device__ Real g(int p) const { return __ldg(pop_ + (9 * (NP - 1) + p) * plane + o); }
};

// Push to x + c_p (periodic wrap), or back into the node's opposite direction
// off an outer wall (halfway bounce-back); plane a with its ghost images.
template <int NP>
struct Sink64 {
    long long tgt[9];   // target offset, plane of the direction included
    long long o, plane, ax, ay;   // offsets of a's ghost images (0: none)
    Real *pop, *lagp, *mac;
    __device__ void f_out(int i, int p, Real v) { pop[9 * i * plane + tgt[p]] = v; }
    __device__ void g_out(int p, Real v) { pop[9 * (NP - 1) * plane + tgt[p]] = v; }
    __device__ void lag_out(int k, Real v) {
        lagp[k * plane + o] = v;
        if (k == 0) {
            if (ax) lagp[o + ax] = v;
            if (ay) lagp[o + ay] = v;
            if (ax && ay) lagp[o + ax + ay] = v;
        }
    }
    __device__ void macro(const Real* Cv, Real rho, Real ux, Real uy, Real Pr, const Real* m) {
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            mac[j * plane + o] = Cv[j];
            mac[(NP + 4 + j) * plane + o] = m[j];
        }
        mac[NP * plane + o] = rho;
        mac[(NP + 1) * plane + o] = ux;
        mac[(NP + 2) * plane + o] = uy;
        mac[(NP + 3) * plane + o] = Pr;
    }
};

template <int NP, int MODE, bool kOneRate>
__global__ void __launch_bounds__(UT, 5) k_update64(KParams<Real> P, Step64Args F) {
    const unsigned idx = blockIdx.x * (unsigned)UT + threadIdx.x;
    if (idx >= (unsigned)P.nx * (unsigned)P.ny) return;
    const int y = (int)(idx / (unsigned)P.nx), x = (int)(idx - (unsigned)y * (unsigned)P.nx);
    Acc64<NP> acc{F.C, F.chi, F.mu, F.psi, F.st, F.pop_in, F.lag_in, P.plane};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        acc.row[d] = P.org + (long long)map_index(y - 1 + d, P.ny, P.py) * P.pitch;
        acc.col[d] = map_index(x - 1 + d, P.nx, P.px);
    }
    acc.o = acc.at(0, 0);
    Sink64<NP> sink;
    sink.o = acc.o;
    sink.plane = P.plane;
    sink.pop = F.pop_out;
    sink.lagp = F.lag_out;
    sink.mac = F.macro;
    if (MODE == 0) {
        sink.ax = ring_step(x, P.nx, P.px);
        sink.ay = (long long)ring_step(y, P.ny, P.py) * P.pitch;
        const bool wx[3] = {!P.px && x == 0, false, !P.px && x == P.nx - 1};
        const bool wy[3] = {!P.py && y == 0, false, !P.py && y == P.ny - 1};
#pragma unroll
        for (int p = 0; p < 9; ++p) {
            const bool bounce = wx[vx(p) + 1] || wy[vy(p) + 1];
            sink.tgt[p] = bounce ? vopp(p) * P.plane + acc.o : p * P.plane + acc.at(vy(p), vx(p));
        }
    }
    dev::node_update<Real, NP, MODE, kOneRate>(P, acc, sink);
}

template <int NP>
cudaError_t fields_n(const KParams<Real>& kp, const Step64Args& a, cudaStream_t s) {
    const int tx = (kp.nx + FX - 1) / FX, ty = (kp.ny + FY - 1) / FY;
    k_fields64<NP><<<(unsigned)((long long)tx * ty), FT, 0, s>>>(kp, a.pop_in, a.psi, a.st, a.cosf, a.C, a.chi, a.mu, tx);
    return cudaGetLastError();
}

template <int NP, int MODE>
cudaError_t update_n(const KParams<Real>& kp, const Step64Args& a, cudaStream_t s) {
    const long long n = (long long)kp.nx * kp.ny;
    const unsigned blocks = (unsigned)((n + UT - 1) / UT);
    // 512 x 512, N = 4: 327 us a launch by the transforms, 285 with one rate
    if (MODE == 0 && kp.one_rate) k_update64<NP, MODE, MODE == 0><<<blocks, UT, 0, s>>>(kp, a);
    else k_update64<NP, MODE, false><<<blocks, UT, 0, s>>>(kp, a);
    return cudaGetLastError();
}

}  // namespace

int static64_planes() { return kStaticPlanes; }

cudaError_t launch_static64(const KParams<double>& kp, const double* psi, double* st, cudaStream_t s) {
    const long long n = (long long)kp.nx * kp.ny, b = (n + 255) / 256;
    k_static64<<<(unsigned)(b < 152 * 16 ? b : 152 * 16), 256, 0, s>>>(kp, psi, st);
    return cudaGetLastError();
}

cudaError_t launch_fields64(const KParams<double>& kp, const Step64Args& a, cudaStream_t s) {
    switch (kp.N) {
        case 2: return fields_n<2>(kp, a, s);
        case 3: return fields_n<3>(kp, a, s);
        case 4: return fields_n<4>(kp, a, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_update64(const KParams<double>& kp, const Step64Args& a, cudaStream_t s) {
    switch (kp.N * 2 + (a.macro ? 1 : 0)) {
        case 4: return update_n<2, 0>(kp, a, s);
        case 5: return update_n<2, 1>(kp, a, s);
        case 6: return update_n<3, 0>(kp, a, s);
        case 7: return update_n<3, 1>(kp, a, s);
        case 8: return update_n<4, 0>(kp, a, s);
        case 9: return update_n<4, 1>(kp, a, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace ddcc
