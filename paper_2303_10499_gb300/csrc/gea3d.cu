// gea3d.cu -- the time step of the GEA pressure-based Euler solver
// (Girfoglio, Quaini & Rozza, arXiv 2303.10499, Section 3) on a uniform
// Cartesian x-y-z grid, FP64, and the C ABI of include/gea3d.h.
//
// Blocks of 32 x 8 threads: one thread per cell of a layer, or per column of a
// few layers in the kernels with a reduction and the finest prolongation
// (columns_of); the solve's kernels take one pair of cells of a row per thread.
// Neighbour values are read through the read-only cache with the one-layer
// wall ghosts applied on the fly (wall-normal velocity odd, tangential and
// scalars even, h with dh/dz = -g). The transport operator
// T(X) = (rho1/dt) X + C(X) - nu L(X) (fourth-order face values) is assembled
// once a step as a 13-point cross stencil. The
// pressure equation is solved by CG on the black half of a red-black colouring,
// preconditioned with a V-cycle (piecewise-constant transfer over 2 x 2 x 2
// cells, red-black smoothing), the loops as conditional WHILE nodes of a CUDA
// graph ended by a one-thread control kernel. Reductions are deterministic (block partials
// summed in a fixed order by the last block).
//
// Layout: every array (cells and faces) is indexed (k (ny+1) + j) P + i with
// P = nx + 1 rounded up to 32: x-face i lies between cells i-1 and i,
// y-face j between rows j-1 and j, z-face k between layers k-1 and k.
#include "gea_internal.cuh"
#include "../../include/gea3d.h"

#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <climits>
#include <type_traits>
#include <vector>

namespace g3 {

constexpr int TX = 32, TY = 8, NT = TX * TY;
static_assert(NT == gea::NTHREADS, "block_sum reduces NTHREADS values");
constexpr int kMaxLev = 12;
constexpr double kCoarsestRatio = 1.0;
constexpr double kRefT = 300.0;
enum { E3 = 0, U3 = 1, V3 = 2, W3 = 3, H3 = 4 };
enum { L_MOM = 0, L_ENTH = 1, L_CG = 2 };
enum { C_PRED = 0, C_MOM, C_ERHS, C_ENTH, C_HELM, C_RZ, C_PQ, C_UPD, C_DER, C_DIAG };

struct Geo {
    int nx, ny, nz, P;
    double dx, dy, dz;
    double idx, idy, idz, idx2, idy2, idz2, ivol;   // 1/dx, ..., 1/dx^2, ..., 1/(dx dy dz)
    double ax, ay, az;                              // face areas dy dz, dx dz, dx dy
    // products formed once on the host (in a kernel each would be an FP64
    // instruction of every thread)
    double hidx, hidy, hidz, tidx, tidy, tidz;      // 1/(2 dx), ..., 2/dx, ...
    double hax, hay, haz;                           // half the face areas
    double s12;                                     // 1/(12 dx dy dz)
};

__host__ __device__ inline int id3(const Geo &G, int i, int j, int k)
{
    return (k * (G.ny + 1) + j) * G.P + i;
}

struct Phy {
    double R, cp, g, mu, nuh, dt, idt;
    double icp, icv; // 1/cp, 1/cv
    double mux, muy, muz, mud, nud;   // mu/dx^2, ..., 2 mu (1/dx^2 + 1/dy^2 + 1/dz^2), the same with mu/Pr
    int les, pr_ne1; // les_d2 > 0; mu/Pr != mu
    double les_d2;   // (cs Delta)^2 with Delta = (dx dy dz)^(1/3); 0: constant mu
};

struct St {
    double *rho, *u, *v, *w, *T, *h, *p, *pp, *pold, *phix, *phiy, *phiz;
};

// The FP64 Helmholtz operator: (A x)_i = c_i x_i + sum_f a_f (x_i - x_N),
// d = c + sum a, wd = 1/d, a on the x-, y- and z-faces (zero on walls); r the
// residual of a solve's start.
struct Lev {
    Geo G;
    double *c, *d, *ax, *ay, *az, *r, *wd;
};

// FP32 level of the multigrid preconditioner (on the finest level the twin
// of the FP64 operator; r, e and e2 unused there): w = 1/d, r the restricted
// residual, e the smoothed correction of the down half, e2 the correction.
struct Lev32 {
    Geo G;
    float *c, *d, *ax, *ay, *az, *w, *r, *e, *e2;
    double fx, fy, fz;   // coarse-face factors 1/8 coarse_scale (k_coarsen)
};

// The operator of a solve in its own precision.
template <class R>
struct Op {
    Geo G;
    const R *d, *ax, *ay, *az, *wd;
};

// The vectors of a solve: one value per pair of cells of a row, of its black
// cell or (w) of its red one. p the direction, w the red part of A p over d
// with the sign turned, q = S p, rb the residual, xb the solution, ef = rb / d
// and z the preconditioned residual (z = ef on a hierarchy of one level).
template <class R>
struct Rb {
    R *p, *w, *q, *rb, *xb;
    float *ef, *z;
};

// The transport operator T(X) = (rho1/dt) X + C(X) - mu L(X) of the step as
// a 13-point stencil (slot 0 the cell, then x-2, x-1, x+1, x+2, y-2, ...,
// z+2), the fourth-order face interpolation and the Laplacian folded into
// the weights; set once per step from the fluxes phi^n and rho1.
constexpr int NCF = 13;
struct Cf {
    double *c[NCF];
};

struct Sc {
    double bn2[4];
    double b2, r2, rz, pq, alpha, beta;
    int done[3], trips[3], sweeps[2], cg_it, corr, cg_iters[4];
    double cg_relres[4];
    int status, bad_cells;
    long long steps_done;
    int last_sweeps[2], last_cg_iters[4];
    double last_cg_relres[4];
    int last_status;
    long long launches;
    unsigned counters[16];
    double mass, energy;   // diagnostics (k_diag3)
};

struct Args {
    Geo G;
    Phy F;
    St S, N;
    double *rho1, *dinvu, *dinvh, *bu, *bv, *bw, *ua, *va, *wa, *ub, *vb, *wb, *bh, *ha, *hb;
    double *rho2, *psi, *Dx, *Dy, *Dz, *Hx, *Hy, *Hz;
    double *dtr1;   // dt / rho1
    double *kin;    // K1 = |u1|^2 / 2
    double *mueff;  // mu + mu_t (LES only)
    const double *gzc, *gzf;   // g z of the cell centres (layer k) and of the horizontal faces (k = 0..nz)
    const double *gx2, *gy2, *gz2;   // 2 g z / dx, 2 g z / dy of the cell centres, 2 g z / dz of the horizontal faces
    Cf cf;
    Sc *sc;
    double *part;
    double jtol2, ctol2;
};

__device__ __forceinline__ double ld(const double *p) { return __ldg(p); }
__device__ __forceinline__ float ld(const float *p) { return __ldg(p); }
__device__ __forceinline__ float ldf(const float *p) { return __ldg(p); }

// Cell (i,j,k) of the thread, or false beyond the box.
__device__ __forceinline__ bool cell(const Geo &G, int &i, int &j, int &k)
{
    i = blockIdx.x * TX + threadIdx.x;
    j = blockIdx.y * TY + threadIdx.y;
    k = blockIdx.z;
    return i < G.nx && j < G.ny && k < G.nz;
}

// The kernels with a reduction and the finest prolongation walk consecutive
// cell layers of their column tile (one block reduction per column: a
// reduction of three FP64 values costs a block 36 FP64 instructions of one
// warp, 4.5 per cell at one cell a thread): (i, j) of the thread and its layer
// range [k0, k1), from the launch shape (columns_of). The layer loop stays
// rolled: unrolled, its interleaved loads took 56-79 registers a thread and the
// kernels ran 30-40 % slower at the lower occupancy.
__device__ __forceinline__ bool column(const Geo &G, int &i, int &j, int &k0, int &k1)
{
    const int layers = (G.nz + gridDim.z - 1) / gridDim.z;
    i = blockIdx.x * TX + threadIdx.x;
    j = blockIdx.y * TY + threadIdx.y;
    k0 = blockIdx.z * layers;
    k1 = min(G.nz, k0 + layers);
    return i < G.nx && j < G.ny;
}

// X at (i,j,k) with at most one index one layer outside the box: the ghost
// of wall rule BC.
template <int BC>
__device__ __forceinline__ double at(const Geo &G, const Phy &F, const double *X, int i, int j, int k)
{
    if (i < 0) { const double v = ld(&X[id3(G, 0, j, k)]); return BC == U3 ? -v : v; }
    if (i >= G.nx) { const double v = ld(&X[id3(G, G.nx - 1, j, k)]); return BC == U3 ? -v : v; }
    if (j < 0) { const double v = ld(&X[id3(G, i, 0, k)]); return BC == V3 ? -v : v; }
    if (j >= G.ny) { const double v = ld(&X[id3(G, i, G.ny - 1, k)]); return BC == V3 ? -v : v; }
    if (k < 0) {
        const double v = ld(&X[id3(G, i, j, 0)]);
        return BC == W3 ? -v : (BC == H3 ? v + F.g * G.dz : v);
    }
    if (k >= G.nz) {
        const double v = ld(&X[id3(G, i, j, G.nz - 1)]);
        return BC == W3 ? -v : (BC == H3 ? v - F.g * G.dz : v);
    }
    return ld(&X[id3(G, i, j, k)]);
}

// X at the neighbour (i+di, j+dj, k+dk) of cell q: a fixed offset from q
// when the whole stencil of the cell lies inside the box (interior), the
// ghost rule otherwise.
template <int BC>
__device__ __forceinline__ double nbr(const Geo &G, const Phy &F, const double *X, int q, bool interior,
                                      int i, int j, int k, int di, int dj, int dk)
{
    if (interior) return ld(X + q + di + dj * G.P + dk * G.P * (G.ny + 1));
    return at<BC>(G, F, X, i + di, j + dj, k + dk);
}

// Compact 7-point Laplacian through the ghosts.
template <int BC>
__device__ double lap(const Args &a, const double *X, int i, int j, int k)
{
    const Geo &G = a.G;
    const Phy &F = a.F;
    const double xc = at<BC>(G, F, X, i, j, k);
    return (at<BC>(G, F, X, i + 1, j, k) - xc + at<BC>(G, F, X, i - 1, j, k) - xc) * G.idx2 +
           (at<BC>(G, F, X, i, j + 1, k) - xc + at<BC>(G, F, X, i, j - 1, k) - xc) * G.idy2 +
           (at<BC>(G, F, X, i, j, k + 1) - xc + at<BC>(G, F, X, i, j, k - 1) - xc) * G.idz2;
}

// Deterministic grid sum of NV values per thread (3D grid of 32 x 8 blocks)
// in two levels: the last block of each group of kGroup blocks adds its
// group's block totals, the last group adds the group totals, each in a fixed
// order. True in thread 0 of the very last block, with the totals in tot.
// part holds kCntSlots doubles of group counters (zero between launches),
// then NV x blocks block totals, then NV x groups group totals. T is the
// type of the per-thread values and of the block sums (FP32 in the inner
// solves of the mixed step); block totals onward are FP64.
constexpr int kGroup = 1024;
constexpr int kCntSlots = 2048;   // 4096 group counters
template <int NV, class T = double>
__device__ bool gsum(const T (&v)[NV], double *red, double *part, unsigned *counter, double (&tot)[NV])
{
    __shared__ int flag;
    const int tid = threadIdx.x + threadIdx.y * TX;
    const int bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    const int nb = gridDim.x * gridDim.y * gridDim.z;
    const int ng = (nb + kGroup - 1) / kGroup, grp = bid / kGroup, g0 = grp * kGroup;
    const int gn = min(kGroup, nb - g0);
    unsigned *gcnt = reinterpret_cast<unsigned *>(part);
    double *p1 = part + kCntSlots, *p2 = p1 + (size_t)NV * nb;
    T bt[NV];
    gea::block_sum<NV, T>(v, reinterpret_cast<T *>(red), bt);
    if (tid == 0) {
#pragma unroll
        for (int m = 0; m < NV; ++m) p1[(size_t)m * nb + bid] = (double)bt[m];
        __threadfence();
        flag = atomicAdd(&gcnt[grp], 1u) == (unsigned)gn - 1u;
    }
    __syncthreads();
    if (!flag) return false;
    __threadfence();
    double s[NV];
#pragma unroll
    for (int m = 0; m < NV; ++m) {
        s[m] = 0.0;
        for (int bb = tid; bb < gn; bb += NT) s[m] += __ldcg(&p1[(size_t)m * nb + g0 + bb]);
    }
    double gt[NV];
    gea::block_sum<NV>(s, red, gt);
    if (tid == 0) {
        gcnt[grp] = 0u;
#pragma unroll
        for (int m = 0; m < NV; ++m) p2[(size_t)m * ng + grp] = gt[m];
        __threadfence();
        flag = atomicAdd(counter, 1u) == (unsigned)ng - 1u;
    }
    __syncthreads();
    if (!flag) return false;
    __threadfence();
#pragma unroll
    for (int m = 0; m < NV; ++m) {
        s[m] = 0.0;
        for (int bb = tid; bb < ng; bb += NT) s[m] += __ldcg(&p2[(size_t)m * ng + bb]);
    }
    gea::block_sum<NV>(s, red, tot);
    if (tid == 0) *counter = 0u;
    return tid == 0;
}

__device__ __forceinline__ bool over(const Sc *sc, int which) { return sc->status || sc->done[which]; }

}  // namespace g3

namespace g3 {

// ---- set-up from conservative fields (dense nz x ny x nx arrays) ----

__global__ void k_derive(Geo G, Phy F, const double *rho, const double *ru, const double *rv,
                         const double *rw, const double *re, const double *gzc, St S, Sc *sc)
{
    int i, j, k;
    if (!cell(G, i, j, k)) return;
    const int n = (k * G.ny + j) * G.nx + i, q = id3(G, i, j, k);
    const double gz = gzc[k];
    const double r = rho[n], ir = gea::recip(r);
    const double ru0 = ru[n], rv0 = rv[n], rw0 = rw[n], e1 = re[n];
    const double u = ru0 * ir, v = rv0 * ir, w = rw0 * ir;
    // e = re / r rounded as a division would: T and with it p = rho R T carry
    // the hydrostatic balance
    const double e0 = e1 * ir, e = fma(fma(-r, e0, e1), ir, e0);
    const double T = ((e - 0.5 * fma(u, u, fma(v, v, w * w))) - gz) * F.icv;
    if (!(r > 0.0) || !(T > 0.0)) atomicAdd(&sc->bad_cells, 1);
    S.rho[q] = r; S.u[q] = u; S.v[q] = v; S.w[q] = w; S.T[q] = T; S.h[q] = F.cp * T;
    const double p = r * F.R * T;
    S.p[q] = p; S.pp[q] = fma(r, gz, p); S.pold[q] = p;
    const int sx = 1, sy = G.nx, sz = G.nx * G.ny;
    S.phix[q] = i > 0 ? (ru[n - sx] + ru0) * G.hax : 0.0;
    S.phiy[q] = j > 0 ? (rv[n - sy] + rv0) * G.hay : 0.0;
    S.phiz[q] = k > 0 ? (rw[n - sz] + rw0) * G.haz : 0.0;
    if (i == G.nx - 1) S.phix[id3(G, G.nx, j, k)] = 0.0;
    if (j == G.ny - 1) S.phiy[id3(G, i, G.ny, k)] = 0.0;
    if (k == G.nz - 1) S.phiz[id3(G, i, j, G.nz)] = 0.0;
}

// Differences of p' and rho between two cells: p'_b - p'_a - gz (rho_b - rho_a),
// the face force times the spacing when a and b share the face of height gz.
// On a wall the cell stands for its missing neighbour, which gives zero.
__device__ __forceinline__ double fdiff(const double *pp, const double *rho, int b, int a, double gz)
{
    return fma(-gz, ld(&rho[b]) - ld(&rho[a]), ld(&pp[b]) - ld(&pp[a]));
}

// Neighbour indices of cell q at (i, j, k), the cell itself beyond a wall.
struct Nb {
    int w, e, s, n, b, t;
};
__device__ __forceinline__ Nb neighbours(const Geo &G, int q, int i, int j, int k)
{
    const int sy = G.P, sz = G.P * (G.ny + 1);
    return Nb{i > 0 ? q - 1 : q,  i + 1 < G.nx ? q + 1 : q,  j > 0 ? q - sy : q,
              j + 1 < G.ny ? q + sy : q, k > 0 ? q - sz : q, k + 1 < G.nz ? q + sz : q};
}

__device__ __forceinline__ void fin_pred(Sc *sc, const double (&t)[3])
{
    for (int m = 0; m < 3; ++m) sc->bn2[m] = t[m];
    sc->done[L_MOM] = 0;
    sc->trips[L_MOM] = 0;
    sc->sweeps[0] = 0;
}

// ---- Step 1 (eq. e1_d, eq. step2_sd first line) ----

// Smagorinsky LES: mu_eff = mu + rho^n (cs Delta)^2 |S|, |S| = sqrt(2 S_ij S_ij)
// from central differences of u^n (ghosts by the wall rules).
__global__ void k_les(Args a)
{
    if (a.sc->status) return;
    int i, j, k;
    if (!cell(a.G, i, j, k)) return;
    const Geo &G = a.G;
    const Phy &F = a.F;
    const double hx = G.hidx, hy = G.hidy, hz = G.hidz;
    const double *u = a.S.u, *v = a.S.v, *w = a.S.w;
    const int q = id3(G, i, j, k);
    const bool in = i >= 1 && i + 1 < G.nx && j >= 1 && j + 1 < G.ny && k >= 1 && k + 1 < G.nz;
    auto U = [&](int di, int dj, int dk) { return nbr<U3>(G, F, u, q, in, i, j, k, di, dj, dk); };
    auto V = [&](int di, int dj, int dk) { return nbr<V3>(G, F, v, q, in, i, j, k, di, dj, dk); };
    auto Wv = [&](int di, int dj, int dk) { return nbr<W3>(G, F, w, q, in, i, j, k, di, dj, dk); };
    const double ux = (U(1, 0, 0) - U(-1, 0, 0)) * hx;
    const double uy = (U(0, 1, 0) - U(0, -1, 0)) * hy;
    const double uz = (U(0, 0, 1) - U(0, 0, -1)) * hz;
    const double vx = (V(1, 0, 0) - V(-1, 0, 0)) * hx;
    const double vy = (V(0, 1, 0) - V(0, -1, 0)) * hy;
    const double vz = (V(0, 0, 1) - V(0, 0, -1)) * hz;
    const double wx = (Wv(1, 0, 0) - Wv(-1, 0, 0)) * hx;
    const double wy = (Wv(0, 1, 0) - Wv(0, -1, 0)) * hy;
    const double wz = (Wv(0, 0, 1) - Wv(0, 0, -1)) * hz;
    const double sxy = uy + vx, sxz = uz + wx, syz = vz + wy;
    const double S = sqrt(fma(2.0, fma(ux, ux, fma(vy, vy, wz * wz)), fma(sxy, sxy, fma(sxz, sxz, syz * syz))));
    a.mueff[q] = fma(ld(&a.S.rho[q]) * F.les_d2, S, F.mu);
}

// rho1, the Jacobi reciprocals, b = rho^n u^n / dt - G_cell, initial guesses
// u^n; acc += |b|^2 per component.
__global__ void k_pred(Args a)
{
    if (a.sc->status) return;
    __shared__ double red[3 * NT];
    double acc[3] = {0.0, 0.0, 0.0}, tot[3];
    const Geo &G = a.G;
    const Phy &F = a.F;
    int i, j, k0, k1;
    if (column(G, i, j, k0, k1))
#pragma unroll 1
        for (int k = k0; k < k1; ++k) {
            const int q = id3(G, i, j, k), sy = G.P, sz = G.P * (G.ny + 1);
            const Nb nb = neighbours(G, q, i, j, k);
            const double pw = ld(&a.S.phix[q]), pe = ld(&a.S.phix[q + 1]);
            const double ps = ld(&a.S.phiy[q]), pn = ld(&a.S.phiy[q + sy]);
            const double pb = ld(&a.S.phiz[q]), pt = ld(&a.S.phiz[q + sz]);
            const double dv = ((pe - pw) + (pn - ps) + (pt - pb)) * G.ivol, r = ld(&a.S.rho[q]);
            const double rho1 = fma(-F.dt, dv, r);
            a.rho1[q] = rho1;
            // diffusion weights per face: mu/Delta^2, or with LES the face mean of
            // mu_eff over Delta^2 (a wall face takes the cell's own, the even ghost)
            double mw, me, ms, mn, mb, mt, md;
            if (F.les) {
                const double mc = ld(&a.mueff[q]);
                // (mu_c + mu_N)/2 / Delta^2, the halves folded into the factors
                const double hx = 0.5 * G.idx2, hy = 0.5 * G.idy2, hz = 0.5 * G.idz2;
                mw = (mc + ld(&a.mueff[nb.w])) * hx; me = (mc + ld(&a.mueff[nb.e])) * hx;
                ms = (mc + ld(&a.mueff[nb.s])) * hy; mn = (mc + ld(&a.mueff[nb.n])) * hy;
                mb = (mc + ld(&a.mueff[nb.b])) * hz; mt = (mc + ld(&a.mueff[nb.t])) * hz;
                md = (mw + me) + (ms + mn) + (mb + mt);
            } else {
                mw = me = F.mux;
                ms = mn = F.muy;
                mb = mt = F.muz;
                md = F.mud;
            }
            const double c0 = fma(rho1, F.idt, (7.0 / 12.0) * dv);
            const double cu = c0 + md, icu = gea::recip(cu);
            a.dinvu[q] = icu;
            // the enthalpy diagonal: the diffusion scaled by 1/Pr (LES requires Pr = 1)
            double ich = icu;
            gea::rarely(F.pr_ne1, [&] { ich = gea::recip(c0 + F.nud); });
            a.dinvh[q] = ich;
            // T as a stencil: the outgoing flux of a face times its fourth-order
            // value (-X_m + 7 X_a + 7 X_b - X_p)/12, minus the diffusion
            const double fw = pw * G.s12, fe = pe * G.s12, fs = ps * G.s12, fn = pn * G.s12, fb = pb * G.s12, ft = pt * G.s12;
            const Cf &cf = a.cf;
            cf.c[0][q] = cu;
            cf.c[1][q] = fw;
            cf.c[2][q] = -fma(7.0, fw, fe) - mw;
            cf.c[3][q] = fma(7.0, fe, fw) - me;
            cf.c[4][q] = -fe;
            cf.c[5][q] = fs;
            cf.c[6][q] = -fma(7.0, fs, fn) - ms;
            cf.c[7][q] = fma(7.0, fn, fs) - mn;
            cf.c[8][q] = -fn;
            cf.c[9][q] = fb;
            cf.c[10][q] = -fma(7.0, fb, ft) - mb;
            cf.c[11][q] = fma(7.0, ft, fb) - mt;
            cf.c[12][q] = -ft;
            // sums of the two face forces of each direction (over the spacing); in x
            // and y both faces have the cell's height
            const double gc = ld(&a.gzc[k]);
            const double sxf = fdiff(a.S.pp, a.S.rho, nb.e, nb.w, gc), syf = fdiff(a.S.pp, a.S.rho, nb.n, nb.s, gc);
            const double szf = fdiff(a.S.pp, a.S.rho, nb.t, q, ld(&a.gzf[k + 1])) + fdiff(a.S.pp, a.S.rho, q, nb.b, ld(&a.gzf[k]));
            a.dtr1[q] = F.dt * gea::recip(rho1);
            const double u = ld(&a.S.u[q]), v = ld(&a.S.v[q]), w = ld(&a.S.w[q]), rdt = r * F.idt;
            const double bu = fma(-G.hidx, sxf, rdt * u), bv = fma(-G.hidy, syf, rdt * v), bw = fma(-G.hidz, szf, rdt * w);
            a.bu[q] = bu; a.bv[q] = bv; a.bw[q] = bw;
            a.ua[q] = u; a.va[q] = v; a.wa[q] = w;
            acc[0] = fma(bu, bu, acc[0]);
            acc[1] = fma(bv, bv, acc[1]);
            acc[2] = fma(bw, bw, acc[2]);
        }
    if (gsum<3>(acc, red, a.part, &a.sc->counters[C_PRED], tot)) fin_pred(a.sc, tot);
}

// The 13 stencil weights of a cell.
struct W13 {
    double w[NCF];
};

__device__ __forceinline__ W13 weights(const Args &a, int q)
{
    W13 c;
#pragma unroll
    for (int m = 0; m < NCF; ++m) c.w[m] = ld(&a.cf.c[m][q]);
    return c;
}

// b minus the off-centre part of T(X), the sum over the 12 neighbour slots of
// weight times value (ghosts by rule BC; slots two cells beyond a wall carry
// weight 0), as one chain of FMAs.
template <int BC>
__device__ __forceinline__ double toff(const Args &a, double b, const W13 &c, const double *X, int i, int j, int k)
{
    const Geo &G = a.G;
    const Phy &F = a.F;
    if (i >= 2 && i + 2 < G.nx && j >= 2 && j + 2 < G.ny && k >= 2 && k + 2 < G.nz) {
        // away from the walls: the neighbours at fixed offsets (same order)
        const int sy = G.P, sz = G.P * (G.ny + 1);
        const double *x = X + id3(G, i, j, k);
        double t = fma(-c.w[1], ld(x - 2), b);
        t = fma(-c.w[2], ld(x - 1), t);
        t = fma(-c.w[3], ld(x + 1), t);
        t = fma(-c.w[4], ld(x + 2), t);
        t = fma(-c.w[5], ld(x - 2 * sy), t);
        t = fma(-c.w[6], ld(x - sy), t);
        t = fma(-c.w[7], ld(x + sy), t);
        t = fma(-c.w[8], ld(x + 2 * sy), t);
        t = fma(-c.w[9], ld(x - 2 * sz), t);
        t = fma(-c.w[10], ld(x - sz), t);
        t = fma(-c.w[11], ld(x + sz), t);
        t = fma(-c.w[12], ld(x + 2 * sz), t);
        return t;
    }
    double t = fma(-c.w[1], at<BC>(G, F, X, i - 2, j, k), b);
    t = fma(-c.w[2], at<BC>(G, F, X, i - 1, j, k), t);
    t = fma(-c.w[3], at<BC>(G, F, X, i + 1, j, k), t);
    t = fma(-c.w[4], at<BC>(G, F, X, i + 2, j, k), t);
    t = fma(-c.w[5], at<BC>(G, F, X, i, j - 2, k), t);
    t = fma(-c.w[6], at<BC>(G, F, X, i, j - 1, k), t);
    t = fma(-c.w[7], at<BC>(G, F, X, i, j + 1, k), t);
    t = fma(-c.w[8], at<BC>(G, F, X, i, j + 2, k), t);
    t = fma(-c.w[9], at<BC>(G, F, X, i, j, k - 2), t);
    t = fma(-c.w[10], at<BC>(G, F, X, i, j, k - 1), t);
    t = fma(-c.w[11], at<BC>(G, F, X, i, j, k + 1), t);
    t = fma(-c.w[12], at<BC>(G, F, X, i, j, k + 2), t);
    return t;
}

__device__ __forceinline__ void copy_column(const Geo &G, const double *x, double *y)
{
    int i, j, k0, k1;
    if (column(G, i, j, k0, k1))
        for (int k = k0; k < k1; ++k) y[id3(G, i, j, k)] = ld(&x[id3(G, i, j, k)]);
}

// One Jacobi sweep of the three momentum components (pairs of sweeps; the
// second of a pair copies once the first met the tolerance). Five blocks per
// SM (48 registers, no spills) measured 3.5 % faster than four.
__global__ void __launch_bounds__(NT, 5) k_mom(Args a, const double *ui, const double *vi, const double *wi, double *uo, double *vo,
                      double *wo, int second)
{
    Sc *sc = a.sc;
    if (sc->status) return;
    if (second && sc->done[L_MOM]) {
        copy_column(a.G, ui, uo);
        copy_column(a.G, vi, vo);
        copy_column(a.G, wi, wo);
        return;
    }
    __shared__ double red[3 * NT];
    double acc[3] = {0.0, 0.0, 0.0}, tot[3];
    int i, j, k0, k1;
    if (column(a.G, i, j, k0, k1))
#pragma unroll 1
        for (int k = k0; k < k1; ++k) {
            const int q = id3(a.G, i, j, k);
            const double di = ld(&a.dinvu[q]);
            const W13 c = weights(a, q);
            // one component after the other (the empty asm keeps the compiler
            // from interleaving their loads, which would cost registers)
            const double u0 = ld(&ui[q]);
            const double ru = toff<U3>(a, fma(-c.w[0], u0, ld(&a.bu[q])), c, ui, i, j, k);
            uo[q] = fma(ru, di, u0);
            acc[0] = fma(ru, ru, acc[0]);
            asm volatile("" ::: "memory");
            const double v0 = ld(&vi[q]);
            const double rv = toff<V3>(a, fma(-c.w[0], v0, ld(&a.bv[q])), c, vi, i, j, k);
            vo[q] = fma(rv, di, v0);
            acc[1] = fma(rv, rv, acc[1]);
            asm volatile("" ::: "memory");
            const double w0 = ld(&wi[q]);
            const double rw = toff<W3>(a, fma(-c.w[0], w0, ld(&a.bw[q])), c, wi, i, j, k);
            wo[q] = fma(rw, di, w0);
            acc[2] = fma(rw, rw, acc[2]);
        }
    if (gsum<3>(acc, red, a.part, &sc->counters[C_MOM], tot)) {
        sc->sweeps[0] += 1;
        if (!isfinite(tot[0]) || !isfinite(tot[1]) || !isfinite(tot[2])) sc->status = GEA_ERR_NONFINITE;
        else if (tot[0] <= a.jtol2 * sc->bn2[0] && tot[1] <= a.jtol2 * sc->bn2[1] && tot[2] <= a.jtol2 * sc->bn2[2])
            sc->done[L_MOM] = 1;
    }
}

// ---- Step 2 (eq. step3_sd) ----

// K1 = |u1|^2/2 per cell (eq. step1_3sd); its wall ghosts are the mirrored
// cells' values (the squares of odd and even ghosts agree).
__global__ void k_kin(Args a, const double *u1, const double *v1, const double *w1)
{
    if (a.sc->status) return;
    int i, j, k;
    if (!cell(a.G, i, j, k)) return;
    const int q = id3(a.G, i, j, k);
    const double u = ld(&u1[q]), v = ld(&v1[q]), w = ld(&w1[q]);
    a.kin[q] = 0.5 * fma(u, u, fma(v, v, w * w));
}

// Right-hand side of the enthalpy equation and its initial guess h^n:
// (rho h + rho K - p^{n-1})/dt - rho1 K1/dt - C(K1) + p^n/dt - rho1 g w1.
__global__ void k_enth_rhs(Args a, const double *w1)
{
    if (a.sc->status) return;
    __shared__ double red[NT];
    double acc[1] = {0.0}, tot[1];
    const Geo &G = a.G;
    const Phy &F = a.F;
    int i, j, k0, k1;
    if (column(G, i, j, k0, k1))
#pragma unroll 1
        for (int k = k0; k < k1; ++k) {
            const int q = id3(G, i, j, k);
            // C(K1), fourth-order face values of K1 with even ghosts; the 1/12 of
            // the face values is applied once to the sum: 12 X_f = 7 (X_a + X_b) - (X_m + X_p)
            double s = 0.0;
            const double Kc = ld(&a.kin[q]);
            const bool in = i >= 2 && i + 2 < G.nx && j >= 2 && j + 2 < G.ny && k >= 2 && k + 2 < G.nz;
            auto K = [&](int ii, int jj, int kk) {
                return nbr<E3>(G, F, a.kin, q, in, i, j, k, ii - i, jj - j, kk - k);
            };
            auto f12 = [](double xm, double xa, double xb, double xp) { return fma(7.0, xa + xb, -(xm + xp)); };
            if (i + 1 < G.nx) s = fma(ld(&a.S.phix[id3(G, i + 1, j, k)]), f12(K(i - 1, j, k), Kc, K(i + 1, j, k), K(i + 2, j, k)), s);
            if (i > 0) s = fma(-ld(&a.S.phix[q]), f12(K(i - 2, j, k), K(i - 1, j, k), Kc, K(i + 1, j, k)), s);
            if (j + 1 < G.ny) s = fma(ld(&a.S.phiy[id3(G, i, j + 1, k)]), f12(K(i, j - 1, k), Kc, K(i, j + 1, k), K(i, j + 2, k)), s);
            if (j > 0) s = fma(-ld(&a.S.phiy[q]), f12(K(i, j - 2, k), K(i, j - 1, k), Kc, K(i, j + 1, k)), s);
            if (k + 1 < G.nz) s = fma(ld(&a.S.phiz[id3(G, i, j, k + 1)]), f12(K(i, j, k - 1), Kc, K(i, j, k + 1), K(i, j, k + 2)), s);
            if (k > 0) s = fma(-ld(&a.S.phiz[q]), f12(K(i, j, k - 2), K(i, j, k - 1), Kc, K(i, j, k + 1)), s);
            const double r = ld(&a.S.rho[q]), u = ld(&a.S.u[q]), v = ld(&a.S.v[q]), w = ld(&a.S.w[q]);
            const double h = ld(&a.S.h[q]), rho1 = ld(&a.rho1[q]);
            const double Kn = 0.5 * fma(u, u, fma(v, v, w * w));
            const double te = fma(r, h + Kn, -ld(&a.S.pold[q])) + ld(&a.S.p[q]);
            const double bh = fma(-rho1 * F.g, ld(&w1[q]), fma(F.idt, fma(-rho1, Kc, te), -(G.s12 * s)));
            a.bh[q] = bh;
            a.ha[q] = h;
            acc[0] = fma(bh, bh, acc[0]);
        }
    if (gsum<1>(acc, red, a.part, &a.sc->counters[C_ERHS], tot)) {
        a.sc->bn2[3] = tot[0];
        a.sc->done[L_ENTH] = 0;
        a.sc->trips[L_ENTH] = 0;
        a.sc->sweeps[1] = 0;
    }
}

// One Jacobi sweep of h (pairs as for momentum); five blocks per SM (48
// registers) measured 8 % faster than four.
__global__ void __launch_bounds__(NT, 5) k_enth(Args a, const double *hi, double *ho, int second)
{
    Sc *sc = a.sc;
    if (sc->status) return;
    if (second && sc->done[L_ENTH]) {
        copy_column(a.G, hi, ho);
        return;
    }
    __shared__ double red[NT];
    double acc[1] = {0.0}, tot[1];
    int i, j, k0, k1;
    if (column(a.G, i, j, k0, k1))
#pragma unroll 1
        for (int k = k0; k < k1; ++k) {
            const int q = id3(a.G, i, j, k);
            const W13 c = weights(a, q);
            const double h0 = ld(&hi[q]);
            // T with nu_h = mu/Pr: the mu-stencil plus (mu - nu_h) L(h)
            double r = toff<H3>(a, fma(-c.w[0], h0, ld(&a.bh[q])), c, hi, i, j, k);
            gea::rarely(a.F.pr_ne1, [&] { r = fma(a.F.nuh - a.F.mu, lap<H3>(a, hi, i, j, k), r); });
            ho[q] = fma(r, ld(&a.dinvh[q]), h0);
            acc[0] = fma(r, r, acc[0]);
        }
    if (gsum<1>(acc, red, a.part, &sc->counters[C_ENTH], tot)) {
        sc->sweeps[1] += 1;
        if (!isfinite(tot[0])) sc->status = GEA_ERR_NONFINITE;
        else if (tot[0] <= a.jtol2 * sc->bn2[3]) sc->done[L_ENTH] = 1;
    }
}

// EOS update (eqs. step3_2sd, step3_3sd): T^{n+1} = T^n + (h^{n+1} - h^n)/cp,
// psi = 1/(R T^{n+1}), rho2 = psi p^n, and c = psi/dt of the fine level.
__global__ void k_eos(Args a, Lev L, Lev32 m, const double *h1)
{
    if (a.sc->status) return;
    int i, j, k;
    if (!cell(a.G, i, j, k)) return;
    const Phy &F = a.F;
    const int q = id3(a.G, i, j, k);
    const double hq = ld(&h1[q]);
    const double T1 = fma(hq - ld(&a.S.h[q]), F.icp, ld(&a.S.T[q]));
    const double psi = gea::recip(F.R * T1);
    a.N.T[q] = T1;
    a.N.h[q] = hq;
    a.rho2[q] = ld(&a.S.p[q]) * psi;
    a.psi[q] = psi;
    const double c = psi * F.idt;
    L.c[q] = c;
    m.c[q] = (float)c;
}

// Face coefficients of the fine level: D_f = dt rho2_f / rho1_f with face
// means of the two cells, on the cell's west, south and bottom faces (zero
// on walls; the last cells also zero the east, north and top wall faces),
// and a_f = D_f / Delta^2.
__global__ void k_faces(Args a, Lev L, Lev32 m)
{
    if (a.sc->status) return;
    int i, j, k;
    if (!cell(a.G, i, j, k)) return;
    const Geo &G = a.G;
    const int q = id3(G, i, j, k), sx = 1, sy = G.P, sz = G.P * (G.ny + 1);
    const double r2 = ld(&a.rho2[q]), r1 = ld(&a.rho1[q]), dt = a.F.dt;
    // the halves of the two face means cancel exactly
    auto D = [&](int qn) { return dt * (r2 + ld(&a.rho2[qn])) * gea::recip(r1 + ld(&a.rho1[qn])); };
    const double Dw = i > 0 ? D(q - sx) : 0.0;
    const double Ds = j > 0 ? D(q - sy) : 0.0;
    const double Db = k > 0 ? D(q - sz) : 0.0;
    a.Dx[q] = Dw; a.Dy[q] = Ds; a.Dz[q] = Db;
    const double ax = Dw * G.idx2, ay = Ds * G.idy2, az = Db * G.idz2;
    L.ax[q] = ax; L.ay[q] = ay; L.az[q] = az;
    m.ax[q] = (float)ax; m.ay[q] = (float)ay; m.az[q] = (float)az;
    if (i == G.nx - 1) { a.Dx[q + sx] = 0.0; L.ax[q + sx] = 0.0; m.ax[q + sx] = 0.0f; }
    if (j == G.ny - 1) { a.Dy[q + sy] = 0.0; L.ay[q + sy] = 0.0; m.ay[q + sy] = 0.0f; }
    if (k == G.nz - 1) { a.Dz[q + sz] = 0.0; L.az[q + sz] = 0.0; m.az[q + sz] = 0.0f; }
}

// Diagonal d = c + the six face coefficients, and 1/d (in FP64 where the solve
// is: RECIP).
template <bool RECIP>
__global__ void k_diag(Lev L, Lev32 m, Sc *sc)
{
    if (sc->status) return;
    int i, j, k;
    if (!cell(L.G, i, j, k)) return;
    const Geo &G = L.G;
    const int q = id3(G, i, j, k), sy = G.P, sz = G.P * (G.ny + 1);
    const double d = ld(&L.c[q]) + (ld(&L.ax[q]) + ld(&L.ax[q + 1])) + (ld(&L.ay[q]) + ld(&L.ay[q + sy])) +
                     (ld(&L.az[q]) + ld(&L.az[q + sz]));
    L.d[q] = d;
    if (RECIP) L.wd[q] = gea::recip(d);
    m.d[q] = (float)d;
    m.w[q] = 1.0f / (float)d;
}

}  // namespace g3

namespace g3 {

// ---- Step 3 (eq. step2_sd second line, eq. p_prime_sd, eq. step4_4sd) ----

// H(u) = rho^n u^n / dt - C(u) + mu L(u) at the newest velocity
__global__ void k_H(Args a, const double *U, const double *V, const double *W)
{
    if (a.sc->status) return;
    int i, j, k;
    if (!cell(a.G, i, j, k)) return;
    const int q = id3(a.G, i, j, k);
    const double r = ld(&a.S.rho[q]) * a.F.idt;
    // C(X) - mu L(X) = T(X) - (rho1/dt) X
    const W13 c = weights(a, q);
    const double c0 = fma(-ld(&a.rho1[q]), a.F.idt, c.w[0]);
    a.Hx[q] = toff<U3>(a, fma(-c0, ld(&U[q]), r * ld(&a.S.u[q])), c, U, i, j, k);
    a.Hy[q] = toff<V3>(a, fma(-c0, ld(&V[q]), r * ld(&a.S.v[q])), c, V, i, j, k);
    a.Hz[q] = toff<W3>(a, fma(-c0, ld(&W[q]), r * ld(&a.S.w[q])), c, W, i, j, k);
}

// ---- the pressure solve: red-black multigrid CG ----
//
// Cells are coloured by the parity of i + j + k (even: black). A couples the
// two colours only, so the red unknowns follow from the black ones and CG runs
// on the black half with S = A_bb - A_br A_rr^-1 A_rb: half the vector traffic,
// as many coefficient reads as A, and fewer iterations with the red-black
// V-cycle than with damped Jacobi on all cells. One FP64 step of
// 512 x 512 x 256 (two levels): 11 + 5 -> 10 + 5 iterations of 2.9 -> 1.95 ms,
// 139 -> 117 ms; the mixed step of 192 x 192 x 96 (one level): 4 + 4 -> 3 + 3
// iterations, 5.8 -> 5.1 ms. The products are at the FP64 rate (7.5 instructions
// a cell, 0.97 ms together), the vector steps and the cycle at memory's.
//
// The vectors hold one value per pair of cells (2 m, 2 m + 1) of a row, at
// (k (ny+1) + j) P/2 + m. With s = (j + k) & 1 the pair's black cell is 2 m + s,
// its red one 2 m + 1 - s; the black cell's red neighbours are those of the
// pairs m - 1 + s (west), m + s (east) and m of the rows beside, above and
// below, the red cell's black neighbours those of m - s, m + 1 - s and m: all
// reads are contiguous.

// Pair m of a row (j, k) and its layer range, as column().
__device__ __forceinline__ bool pair_column(const Geo &G, int &m, int &j, int &k0, int &k1)
{
    const int layers = (G.nz + gridDim.z - 1) / gridDim.z;
    m = blockIdx.x * TX + threadIdx.x;
    j = blockIdx.y * TY + threadIdx.y;
    k0 = blockIdx.z * layers;
    k1 = min(G.nz, k0 + layers);
    return 2 * m < G.nx && j < G.ny;
}

__device__ __forceinline__ int pair_id(const Geo &G, int m, int j, int k)
{
    return (k * (G.ny + 1) + j) * (G.P / 2) + m;
}

// Indices of the six neighbours of cell i of pair index c (RED: the pair's
// red cell). A neighbour beyond a wall is replaced by the opposite one: its
// coefficient is zero and the opposite cell always exists.
template <bool RED>
__device__ __forceinline__ Nb pair_neighbours(const Geo &G, int c, int i, int j, int k)
{
    const int s = (j + k) & 1, cw = c + (RED ? -s : s - 1), ce = cw + 1;
    const int cy = G.P / 2, cz = cy * (G.ny + 1);
    return Nb{i > 0 ? cw : ce,          i + 1 < G.nx ? ce : cw,     j > 0 ? c - cy : c + cy,
              j + 1 < G.ny ? c + cy : c - cy, k > 0 ? c - cz : c + cz, k + 1 < G.nz ? c + cz : c - cz};
}

// The same on a field of cells.
__device__ __forceinline__ Nb other_colour(const Geo &G, int q, int i, int j, int k)
{
    const int sy = G.P, sz = G.P * (G.ny + 1);
    return Nb{i > 0 ? q - 1 : q + 1,          i + 1 < G.nx ? q + 1 : q - 1,  j > 0 ? q - sy : q + sy,
              j + 1 < G.ny ? q + sy : q - sy, k > 0 ? q - sz : q + sz, k + 1 < G.nz ? q + sz : q - sz};
}

// t + the six face coefficients of cell q times x at its neighbours.
template <class R, class XF>
__device__ __forceinline__ R add_faces(R t, const Geo &G, const R *ax, const R *ay, const R *az, int q, const Nb &n,
                                       XF x)
{
    const int sy = G.P, sz = G.P * (G.ny + 1);
    t = fma(ld(&ax[q]), x(n.w), t);
    t = fma(ld(&ax[q + 1]), x(n.e), t);
    t = fma(ld(&ay[q]), x(n.s), t);
    t = fma(ld(&ay[q + sy]), x(n.n), t);
    t = fma(ld(&az[q]), x(n.b), t);
    return fma(ld(&az[q + sz]), x(n.t), t);
}

__device__ __forceinline__ void fin_helm(Sc *sc, const double (&t)[2], double tol2, int corr)
{
    sc->b2 = t[0];
    sc->r2 = t[1];
    sc->cg_it = 0;
    sc->corr = corr;
    sc->trips[L_CG] = 0;
    sc->rz = 0.0;
    sc->beta = 0.0;
    sc->done[L_CG] = t[1] <= tol2 * t[0];
    sc->cg_iters[corr] = 0;
    sc->cg_relres[corr] = t[0] > 0.0 ? sqrt(t[1] / t[0]) : 0.0;
    if (!isfinite(t[0]) || !isfinite(t[1])) sc->status = GEA_ERR_NONFINITE;
}

// Mixed step: the inner FP32 solve's tolerance is relative to the initial
// residual r0 = b - A p'_prev (kept in b2); nothing to solve if r0 is already
// at the FP64 tolerance relative to b.
__device__ __forceinline__ void fin_helm_mixed(Sc *sc, const double (&t)[2], double tol2, int corr)
{
    sc->b2 = t[1];
    sc->r2 = t[1];
    sc->cg_it = 0;
    sc->corr = corr;
    sc->trips[L_CG] = 0;
    sc->rz = 0.0;
    sc->beta = 0.0;
    sc->done[L_CG] = t[1] <= tol2 * t[0];
    sc->cg_iters[corr] = 0;
    sc->cg_relres[corr] = 1.0;
    if (!isfinite(t[0]) || !isfinite(t[1])) sc->status = GEA_ERR_NONFINITE;
}

// b_i = (rho^n_i + psi_i rho2_i g z_i)/dt - sum_f D_f/Delta_f [H_f . n + g z_f (rho2_N - rho2_i)/Delta_f],
// r = b - A x with x = xin, and r/d on the red cells into w; acc += (b^2, r^2).
// Mixed step (R = float): r rounded to FP32.
template <class R>
__global__ void k_helm_rhs(Args a, Lev L, const double *xin, int corr, R *rout, const R *wd, R *w)
{
    if (a.sc->status) return;
    __shared__ double red[2 * NT];
    double acc[2] = {0.0, 0.0}, tot[2];
    const Geo &G = a.G;
    const Phy &F = a.F;
    int i, j, k0, k1;
    if (column(G, i, j, k0, k1))
#pragma unroll 1
        for (int k = k0; k < k1; ++k) {
            const int q = id3(G, i, j, k), sy = G.P, sz = G.P * (G.ny + 1);
            const Nb nb = neighbours(G, q, i, j, k);
            const double r2 = ld(&a.rho2[q]);
            // twice the outgoing flux of a direction over its spacing, from
            // D_f (H_a + H_b + 2 g z_f (rho2_b - rho2_a) / Delta); D_f = 0 on walls
            auto pair = [&](const double *D, int up, const double *H, int ql, int qu, double gl, double gu) {
                const double h = ld(&H[q]);
                const double f = ld(&D[q + up]) * fma(gu, ld(&a.rho2[qu]) - r2, h + ld(&H[qu]));
                return fma(-ld(&D[q]), fma(gl, r2 - ld(&a.rho2[ql]), h + ld(&H[ql])), f);
            };
            const double gx = ld(&a.gx2[k]), gy = ld(&a.gy2[k]);
            double fl = G.hidx * pair(a.Dx, 1, a.Hx, nb.w, nb.e, gx, gx);
            fl = fma(G.hidy, pair(a.Dy, sy, a.Hy, nb.s, nb.n, gy, gy), fl);
            fl = fma(G.hidz, pair(a.Dz, sz, a.Hz, nb.b, nb.t, ld(&a.gz2[k]), ld(&a.gz2[k + 1])), fl);
            const double b = fma(fma(ld(&a.psi[q]) * r2, ld(&a.gzc[k]), ld(&a.S.rho[q])), F.idt, -fl);
            double r = fma(-ld(&L.d[q]), ld(&xin[q]), b);
            r = fma(ld(&L.ax[q]), ld(&xin[nb.w]), r);
            r = fma(ld(&L.ax[q + 1]), ld(&xin[nb.e]), r);
            r = fma(ld(&L.ay[q]), ld(&xin[nb.s]), r);
            r = fma(ld(&L.ay[q + sy]), ld(&xin[nb.n]), r);
            r = fma(ld(&L.az[q]), ld(&xin[nb.b]), r);
            r = fma(ld(&L.az[q + sz]), ld(&xin[nb.t]), r);
            rout[q] = (R)r;
            if ((i + j + k) & 1) w[pair_id(G, i >> 1, j, k)] = ld(&wd[q]) * (R)r;
            acc[0] = fma(b, b, acc[0]);
            acc[1] = fma(r, r, acc[1]);
        }
    if (gsum<2>(acc, red, a.part, &a.sc->counters[C_HELM], tot)) {
        if (sizeof(R) == sizeof(float)) fin_helm_mixed(a.sc, tot, a.ctol2, corr);
        else fin_helm(a.sc, tot, a.ctol2, corr);
    }
}

// ---- red-black V-cycle in FP32 (the preconditioner of the CG) ----
//
// The preconditioner only shapes the search directions: the CG residual and
// its stopping test keep the solve's precision, so the converged pressure is
// that of the solve's system. On the black half of the finest level the cycle
// starts with e = rb / d on black (the red residual is zero), restricts what
// that leaves on red, and ends with one black relaxation.

// Coarse level: c_C = mean of the 8 children's c, a coarse face = c.fx, c.fy or
// c.fz times the sum of its 4 fine faces (an eighth, the Galerkin value, times
// coarse_scale of its direction; a sixteenth where the spacings are equal),
// d_C = c_C + sum of its faces. One thread per coarse cell; sums in FP64,
// stored FP32.
__global__ void k_coarsen(Lev32 f, Lev32 c)
{
    int I, J, K;
    if (!cell(c.G, I, J, K)) return;
    const Geo &G = f.G, &H = c.G;
    const int Q = id3(H, I, J, K);
    double cs = 0.0, fx0 = 0.0, fx1 = 0.0, fy0 = 0.0, fy1 = 0.0, fz0 = 0.0, fz1 = 0.0;
    for (int dk = 0; dk < 2; ++dk)
        for (int dj = 0; dj < 2; ++dj)
            for (int di = 0; di < 2; ++di) {
                const int i = 2 * I + di, j = 2 * J + dj, k = 2 * K + dk;
                const int q = id3(G, i, j, k);
                cs += ldf(&f.c[q]);
                if (di == 0) fx0 += ldf(&f.ax[q]); else fx1 += ldf(&f.ax[q + 1]);
                if (dj == 0) fy0 += ldf(&f.ay[q]); else fy1 += ldf(&f.ay[q + G.P]);
                if (dk == 0) fz0 += ldf(&f.az[q]); else fz1 += ldf(&f.az[q + G.P * (G.ny + 1)]);
            }
    const double cc = 0.125 * cs;
    c.c[Q] = (float)cc;
    c.ax[Q] = (float)(c.fx * fx0); c.ay[Q] = (float)(c.fy * fy0); c.az[Q] = (float)(c.fz * fz0);
    if (I == H.nx - 1) c.ax[Q + 1] = (float)(c.fx * fx1);
    if (J == H.ny - 1) c.ay[Q + H.P] = (float)(c.fy * fy1);
    if (K == H.nz - 1) c.az[Q + H.P * (H.ny + 1)] = (float)(c.fz * fz1);
    const double d = cc + c.fx * (fx0 + fx1) + c.fy * (fy0 + fy1) + c.fz * (fz0 + fz1);
    c.d[Q] = (float)d;
    c.w[Q] = (float)(1.0 / d);
}

// Restriction of the residual sum a e_b on the red cells to the coarse level
// (mean of the 8 children; zero on black). e_b is ef pair by pair on the
// finest level (FINE), f.e on the others. One thread per coarse cell.
template <bool FINE>
__global__ void k_mg_down(Lev32 f, const float *ef, Lev32 c, Sc *sc)
{
    if (over(sc, L_CG)) return;
    int I, J, K;
    if (!cell(c.G, I, J, K)) return;
    const Geo &G = f.G;
    float t = 0.0f;
#pragma unroll
    for (int dk = 0; dk < 2; ++dk)
#pragma unroll
        for (int dj = 0; dj < 2; ++dj) {
            const int j = 2 * J + dj, k = 2 * K + dk, i = 2 * I + 1 - ((dj + dk) & 1);
            const int q = id3(G, i, j, k);
            const Nb n = FINE ? pair_neighbours<true>(G, pair_id(G, I, j, k), i, j, k) : other_colour(G, q, i, j, k);
            t = add_faces<float>(t, G, f.ax, f.ay, f.az, q, n, [&](int x) { return ldf(&ef[x]); });
        }
    c.r[id3(c.G, I, J, K)] = 0.125f * t;
}

// The cell of one colour in pair m of a row.
template <bool RED>
__device__ __forceinline__ bool coloured(const Geo &G, int &i, int &j, int &k)
{
    const int m = blockIdx.x * TX + threadIdx.x;
    j = blockIdx.y * TY + threadIdx.y;
    k = blockIdx.z;
    const int s = (j + k) & 1;
    i = 2 * m + (RED ? 1 - s : s);
    return i < G.nx && j < G.ny && k < G.nz;
}

// Black half of a red-black sweep on a level below the finest: the red cells
// hold r / d plus (up half) the coarse correction ec, and black gets
// (r + sum a e_red) / d, into out.
__global__ void k_mg_black(Lev32 f, const float *ec, Geo cg, float *out, Sc *sc)
{
    if (over(sc, L_CG)) return;
    int i, j, k;
    if (!coloured<false>(f.G, i, j, k)) return;
    const Geo &G = f.G;
    const int q = id3(G, i, j, k);
    const Nb n = other_colour(G, q, i, j, k);
    // the pair's other cell has the same coarse parent, the neighbours beyond
    // the 2 x 2 x 2 block the adjacent one
    const int Q = ec ? id3(cg, i >> 1, j >> 1, k >> 1) : 0, cy = cg.P, cz = cg.P * (cg.ny + 1);
    const int up = (n.e - q) * ((i & 1) ? 1 : 0), dn = (n.w - q) * ((i & 1) ? 0 : 1);
    auto e = [&](int x, int Qx) {
        const float v = ldf(&f.w[x]) * ldf(&f.r[x]);
        return ec ? v + ldf(&ec[Qx]) : v;
    };
    const int jn = n.n > q ? 1 : -1, js = n.s > q ? 1 : -1, kt = n.t > q ? 1 : -1, kb = n.b > q ? 1 : -1;
    float t = ldf(&f.r[q]);
    const int sy = G.P, sz = G.P * (G.ny + 1);
    t = fmaf(ldf(&f.ax[q]), e(n.w, Q + (dn < 0 ? -1 : 0)), t);
    t = fmaf(ldf(&f.ax[q + 1]), e(n.e, Q + (up > 0 ? 1 : 0)), t);
    t = fmaf(ldf(&f.ay[q]), e(n.s, Q + (((j + js) >> 1) - (j >> 1)) * cy), t);
    t = fmaf(ldf(&f.ay[q + sy]), e(n.n, Q + (((j + jn) >> 1) - (j >> 1)) * cy), t);
    t = fmaf(ldf(&f.az[q]), e(n.b, Q + (((k + kb) >> 1) - (k >> 1)) * cz), t);
    t = fmaf(ldf(&f.az[q + sz]), e(n.t, Q + (((k + kt) >> 1) - (k >> 1)) * cz), t);
    out[q] = ldf(&f.w[q]) * t;
}

// Red half of the sweep that ends a level: (r + sum a out_black) / d.
__global__ void k_mg_red(Lev32 f, float *out, Sc *sc)
{
    if (over(sc, L_CG)) return;
    int i, j, k;
    if (!coloured<true>(f.G, i, j, k)) return;
    const int q = id3(f.G, i, j, k);
    const Nb n = other_colour(f.G, q, i, j, k);
    const float t = add_faces<float>(ldf(&f.r[q]), f.G, f.ax, f.ay, f.az, q, n, [&](int x) { return out[x]; });
    out[q] = ldf(&f.w[q]) * t;
}

__device__ __forceinline__ void fin_rz(Sc *sc, double t)
{
    sc->beta = (sc->cg_it == 0 || sc->rz == 0.0) ? 0.0 : t / sc->rz;
    sc->rz = t;
}

// Up half on the finest level: z = (rb + sum a P ec) / d = ef + w sum a P ec on
// black; acc += rb z (FP64 for the FP64 CG, FP32 for the mixed step's).
template <class R>
__global__ void k_mg_up(Lev32 f, Rb<R> v, const float *ec, Geo cg, Sc *sc, double *part)
{
    if (over(sc, L_CG)) return;
    __shared__ double red[NT];
    R acc[1] = {(R)0};
    double tot[1];
    const Geo &G = f.G;
    int m, j, k0, k1;
    if (pair_column(G, m, j, k0, k1))
#pragma unroll 1
        for (int k = k0; k < k1; ++k) {
            const int s = (j + k) & 1, i = 2 * m + s;
            if (i >= G.nx) continue;
            const int q = id3(G, i, j, k), c = pair_id(G, m, j, k);
            // parents of the neighbours: of the black cell's own pair m, and the
            // pairs, rows and layers beside it
            auto parent = [&](int mm, int jj, int kk) { return id3(cg, mm, jj >> 1, kk >> 1); };
            const int mw = s ? m : max(m - 1, 0), me = s && i + 1 < G.nx ? m + 1 : m;
            const Nb n{parent(mw, j, k), parent(me, j, k), parent(m, j > 0 ? j - 1 : j, k),
                       parent(m, j + 1 < G.ny ? j + 1 : j, k), parent(m, j, k > 0 ? k - 1 : k),
                       parent(m, j, k + 1 < G.nz ? k + 1 : k)};
            const float t =
                add_faces<float>(0.0f, G, f.ax, f.ay, f.az, q, n, [&](int x) { return ldf(&ec[x]); });
            const float z = fmaf(ldf(&f.w[q]), t, ldf(&v.ef[c]));
            v.z[c] = z;
            acc[0] = fma(ld(&v.rb[c]), (R)z, acc[0]);
        }
    if (gsum<1, R>(acc, red, part, &sc->counters[C_RZ], tot)) fin_rz(sc, tot[0]);
}

// ---- CG on the black half ----

// Start of a solve: the black residual that the relaxed red cells (v.w = r/d)
// leave, rb = r + sum a w, and ef. SINGLE (one level): z = ef; acc += rb z.
template <class R, bool SINGLE>
__global__ void k_rb_start(Op<R> A, const R *r, const float *wf, Rb<R> v, Sc *sc, double *part)
{
    if (over(sc, L_CG)) return;
    __shared__ double red[NT];
    R acc[1] = {(R)0};
    double tot[1];
    const Geo &G = A.G;
    int m, j, k0, k1;
    if (pair_column(G, m, j, k0, k1))
#pragma unroll 1
        for (int k = k0; k < k1; ++k) {
            const int i = 2 * m + ((j + k) & 1);
            if (i >= G.nx) continue;
            const int q = id3(G, i, j, k), c = pair_id(G, m, j, k);
            const R g = add_faces<R>(ld(&r[q]), G, A.ax, A.ay, A.az, q, pair_neighbours<false>(G, c, i, j, k),
                                     [&](int x) { return ld(&v.w[x]); });
            const float e = ldf(&wf[q]) * (float)g;
            v.rb[c] = g;
            v.ef[c] = e;
            if (SINGLE) acc[0] = fma(g, (R)e, acc[0]);
        }
    if (SINGLE)
        if (gsum<1, R>(acc, red, part, &sc->counters[C_RZ], tot)) fin_rz(sc, tot[0]);
}

// p = z + beta p (the first direction: z), pair by pair.
template <class R>
__global__ void k_pupd(Geo G, Rb<R> v, Sc *sc)
{
    if (over(sc, L_CG)) return;
    int i, j, k;
    if (!coloured<false>(G, i, j, k)) return;
    const int c = pair_id(G, i >> 1, j, k);
    const R z = (R)ldf(&v.z[c]);
    v.p[c] = sc->cg_it == 0 ? z : fma((R)sc->beta, v.p[c], z);
}

// w = (sum a p) / d on red
template <class R>
__global__ void k_spmv_red(Op<R> A, Rb<R> v, Sc *sc)
{
    if (over(sc, L_CG)) return;
    int i, j, k;
    if (!coloured<true>(A.G, i, j, k)) return;
    const Geo &G = A.G;
    const int q = id3(G, i, j, k), c = pair_id(G, i >> 1, j, k);
    const R t = add_faces<R>((R)0, G, A.ax, A.ay, A.az, q, pair_neighbours<true>(G, c, i, j, k),
                             [&](int x) { return ld(&v.p[x]); });
    v.w[c] = ld(&A.wd[q]) * t;
}

// q = S p = d p - sum a w on black, acc += p.q; alpha = rz / p.q
template <class R>
__global__ void k_spmv_black(Op<R> A, Rb<R> v, Sc *sc, double *part)
{
    if (over(sc, L_CG)) return;
    __shared__ double red[NT];
    R acc[1] = {(R)0};
    double tot[1];
    const Geo &G = A.G;
    int m, j, k0, k1;
    if (pair_column(G, m, j, k0, k1))
#pragma unroll 1
        for (int k = k0; k < k1; ++k) {
            const int i = 2 * m + ((j + k) & 1);
            if (i >= G.nx) continue;
            const int q = id3(G, i, j, k), c = pair_id(G, m, j, k);
            const R p = ld(&v.p[c]);
            const R t = add_faces<R>(-ld(&A.d[q]) * p, G, A.ax, A.ay, A.az, q, pair_neighbours<false>(G, c, i, j, k),
                                     [&](int x) { return ld(&v.w[x]); });
            v.q[c] = -t;
            acc[0] = fma(p, -t, acc[0]);
        }
    if (gsum<1, R>(acc, red, part, &sc->counters[C_PQ], tot)) {
        sc->pq = tot[0];
        sc->alpha = tot[0] != 0.0 ? sc->rz / tot[0] : 0.0;
        if (!isfinite(tot[0])) sc->status = GEA_ERR_NONFINITE;
    }
}

// xb += alpha p, rb -= alpha q, ef = rb / d; acc += rb^2 and (SINGLE) rb z.
template <class R, bool SINGLE>
__global__ void k_update(Geo G, const float *wf, Rb<R> v, double tol2, Sc *sc, double *part)
{
    if (over(sc, L_CG)) return;
    constexpr int NV = SINGLE ? 2 : 1;
    __shared__ double red[NV * NT];
    R acc[NV] = {};
    double tot[NV];
    const R alpha = (R)sc->alpha;
    const bool first = sc->cg_it == 0;
    int m, j, k0, k1;
    if (pair_column(G, m, j, k0, k1))
#pragma unroll 1
        for (int k = k0; k < k1; ++k) {
            const int i = 2 * m + ((j + k) & 1);
            if (i >= G.nx) continue;
            const int q = id3(G, i, j, k), c = pair_id(G, m, j, k);
            v.xb[c] = fma(alpha, ld(&v.p[c]), first ? (R)0 : v.xb[c]);
            const R rn = fma(-alpha, ld(&v.q[c]), v.rb[c]);
            const float e = ldf(&wf[q]) * (float)rn;
            v.rb[c] = rn;
            v.ef[c] = e;
            acc[0] = fma(rn, rn, acc[0]);
            if (SINGLE) acc[NV - 1] = fma(rn, (R)e, acc[NV - 1]);
        }
    if (gsum<NV, R>(acc, red, part, &sc->counters[C_UPD], tot)) {
        const int n = sc->cg_it + 1;
        sc->cg_it = n;
        sc->r2 = tot[0];
        sc->cg_iters[sc->corr] = n;
        sc->cg_relres[sc->corr] = sc->b2 > 0.0 ? sqrt(tot[0] / sc->b2) : 0.0;
        if (!isfinite(tot[0])) sc->status = GEA_ERR_NONFINITE;
        else if (tot[0] <= tol2 * sc->b2) sc->done[L_CG] = 1;
        else if (SINGLE) fin_rz(sc, tot[NV - 1]);
    }
}

// The solution: xout = xin + xb on black, xin + (r + sum a xb) / d on red (xin
// alone if there was nothing to solve).
template <class R>
__global__ void k_solution(Op<R> A, const R *r, Rb<R> v, const double *xin, double *xout, const Sc *sc)
{
    if (sc->status) return;
    const Geo &G = A.G;
    const bool dx = sc->cg_it > 0;
    const int m = blockIdx.x * TX + threadIdx.x, j = blockIdx.y * TY + threadIdx.y, k = blockIdx.z;
    if (2 * m >= G.nx || j >= G.ny) return;
    const int s = (j + k) & 1, c = pair_id(G, m, j, k), q = id3(G, 2 * m, j, k);
    if (2 * m + s < G.nx) xout[q + s] = dx ? xin[q + s] + (double)ld(&v.xb[c]) : xin[q + s];
    const int i = 2 * m + 1 - s, qr = q + 1 - s;
    if (i < G.nx) {
        double x = xin[qr];
        if (dx) {
            const R t = add_faces<R>(ld(&r[qr]), G, A.ax, A.ay, A.az, qr, pair_neighbours<true>(G, c, i, j, k),
                                     [&](int y) { return ld(&v.xb[y]); });
            x += (double)(ld(&A.wd[qr]) * t);
        }
        xout[qr] = x;
    }
}

// Correction: face forces from the new p' and rho2, F_f = D_f (H_f - G_f),
// u = (dt/rho1)(H - G_cell), p = p' - rho2 g z, rho = p psi, phi = F |A|,
// p^{n-1} <- p^n. Each cell writes its west, south and bottom faces (and the
// walls beyond its east, north and top faces).
__global__ void k_correct(Args a)
{
    if (a.sc->status) return;
    int i, j, k;
    if (!cell(a.G, i, j, k)) return;
    const Geo &G = a.G;
    const int q = id3(G, i, j, k), sx = 1, sy = G.P, sz = G.P * (G.ny + 1);
    const Nb nb = neighbours(G, q, i, j, k);
    const double gc = ld(&a.gzc[k]);
    // Delta G_f of the west, south and bottom faces, and the sum over both
    // faces of each direction
    const double fw = fdiff(a.N.pp, a.rho2, q, nb.w, gc), fs = fdiff(a.N.pp, a.rho2, q, nb.s, gc);
    const double fb = fdiff(a.N.pp, a.rho2, q, nb.b, ld(&a.gzf[k]));
    const double sxf = fdiff(a.N.pp, a.rho2, nb.e, nb.w, gc), syf = fdiff(a.N.pp, a.rho2, nb.n, nb.s, gc);
    const double szf = fdiff(a.N.pp, a.rho2, nb.t, q, ld(&a.gzf[k + 1])) + fb;
    const double c1 = ld(&a.dtr1[q]);
    const double hx = ld(&a.Hx[q]), hy = ld(&a.Hy[q]), hz = ld(&a.Hz[q]);
    a.N.u[q] = c1 * fma(-G.hidx, sxf, hx);
    a.N.v[q] = c1 * fma(-G.hidy, syf, hy);
    a.N.w[q] = c1 * fma(-G.hidz, szf, hz);
    const double pn = fma(-ld(&a.rho2[q]), gc, ld(&a.N.pp[q]));
    a.N.p[q] = pn;
    a.N.rho[q] = pn * ld(&a.psi[q]);
    a.N.pold[q] = ld(&a.S.p[q]);
    // F_f |A_f| = D_f (|A_f| / 2) (H_a + H_b - 2 G_f) (D_f = 0 on walls)
    a.N.phix[q] = (ld(&a.Dx[q]) * G.hax) * fma(-G.tidx, fw, hx + ld(&a.Hx[nb.w]));
    a.N.phiy[q] = (ld(&a.Dy[q]) * G.hay) * fma(-G.tidy, fs, hy + ld(&a.Hy[nb.s]));
    a.N.phiz[q] = (ld(&a.Dz[q]) * G.haz) * fma(-G.tidz, fb, hz + ld(&a.Hz[nb.b]));
    if (i == G.nx - 1) a.N.phix[q + sx] = 0.0;
    if (j == G.ny - 1) a.N.phiy[q + sy] = 0.0;
    if (k == G.nz - 1) a.N.phiz[q + sz] = 0.0;
}

// ---- the mixed-precision step (GEA_FLAG_MIXED) ----
//
// Each implicit solve is one defect correction: an FP64 residual r0 of the
// FP64 operator at the previous value, an FP32 solve for the increment with
// FP32 copies of the operator to ||r|| <= mp_rtol ||r0||, and the FP64
// update. Increments take the homogeneous form of each wall rule (the h
// ghost offset cancels). FP32 reductions are summed in FP32 within a block
// and in FP64 across blocks.

// FP32 data of the mixed step: the stencil weights and reciprocals, the
// FP64 residuals rounded to FP32, the increments (Jacobi ping-pong), and the
// start residual of the pressure solve.
struct Mx {
    float *c[NCF];
    float *dinvu, *dinvh, *r0u, *r0v, *r0w, *r0h;
    float *du[2], *dv[2], *dw[2], *dh[2];
    float *r;            // the pressure residual
    double tol2;
};

// Increment at (i,j,k) with at most one index one layer outside the box: the
// homogeneous ghost of wall rule BC (odd for the wall-normal velocity, even
// otherwise).
template <int BC>
__device__ __forceinline__ float atf(const Geo &G, const float *X, int i, int j, int k)
{
    if (i < 0) { const float v = ldf(&X[id3(G, 0, j, k)]); return BC == U3 ? -v : v; }
    if (i >= G.nx) { const float v = ldf(&X[id3(G, G.nx - 1, j, k)]); return BC == U3 ? -v : v; }
    if (j < 0) { const float v = ldf(&X[id3(G, i, 0, k)]); return BC == V3 ? -v : v; }
    if (j >= G.ny) { const float v = ldf(&X[id3(G, i, G.ny - 1, k)]); return BC == V3 ? -v : v; }
    if (k < 0) { const float v = ldf(&X[id3(G, i, j, 0)]); return BC == W3 ? -v : v; }
    if (k >= G.nz) { const float v = ldf(&X[id3(G, i, j, G.nz - 1)]); return BC == W3 ? -v : v; }
    return ldf(&X[id3(G, i, j, k)]);
}

struct W13f {
    float w[NCF];
};

__device__ __forceinline__ W13f weightsf(const Mx &m, int q)
{
    W13f c;
#pragma unroll
    for (int s = 0; s < NCF; ++s) c.w[s] = ldf(&m.c[s][q]);
    return c;
}

// Off-centre part of the FP32 stencil applied to an increment.
template <int BC>
__device__ __forceinline__ float tofff(const Geo &G, const W13f &c, const float *X, int i, int j, int k)
{
    if (i >= 2 && i + 2 < G.nx && j >= 2 && j + 2 < G.ny && k >= 2 && k + 2 < G.nz) {
        const int sy = G.P, sz = G.P * (G.ny + 1);
        const float *x = X + id3(G, i, j, k);
        float t = c.w[1] * ldf(x - 2);
        t = fmaf(c.w[2], ldf(x - 1), t);
        t = fmaf(c.w[3], ldf(x + 1), t);
        t = fmaf(c.w[4], ldf(x + 2), t);
        t = fmaf(c.w[5], ldf(x - 2 * sy), t);
        t = fmaf(c.w[6], ldf(x - sy), t);
        t = fmaf(c.w[7], ldf(x + sy), t);
        t = fmaf(c.w[8], ldf(x + 2 * sy), t);
        t = fmaf(c.w[9], ldf(x - 2 * sz), t);
        t = fmaf(c.w[10], ldf(x - sz), t);
        t = fmaf(c.w[11], ldf(x + sz), t);
        t = fmaf(c.w[12], ldf(x + 2 * sz), t);
        return t;
    }
    float t = c.w[1] * atf<BC>(G, X, i - 2, j, k);
    t = fmaf(c.w[2], atf<BC>(G, X, i - 1, j, k), t);
    t = fmaf(c.w[3], atf<BC>(G, X, i + 1, j, k), t);
    t = fmaf(c.w[4], atf<BC>(G, X, i + 2, j, k), t);
    t = fmaf(c.w[5], atf<BC>(G, X, i, j - 2, k), t);
    t = fmaf(c.w[6], atf<BC>(G, X, i, j - 1, k), t);
    t = fmaf(c.w[7], atf<BC>(G, X, i, j + 1, k), t);
    t = fmaf(c.w[8], atf<BC>(G, X, i, j + 2, k), t);
    t = fmaf(c.w[9], atf<BC>(G, X, i, j, k - 2), t);
    t = fmaf(c.w[10], atf<BC>(G, X, i, j, k - 1), t);
    t = fmaf(c.w[11], atf<BC>(G, X, i, j, k + 1), t);
    t = fmaf(c.w[12], atf<BC>(G, X, i, j, k + 2), t);
    return t;
}

// Compact Laplacian of an increment with even ghosts (the enthalpy's Pr
// correction).
__device__ __forceinline__ float lapf(const Geo &G, const float *X, int i, int j, int k)
{
    const float xc = atf<E3>(G, X, i, j, k);
    return (atf<E3>(G, X, i + 1, j, k) - xc + atf<E3>(G, X, i - 1, j, k) - xc) * (float)G.idx2 +
           (atf<E3>(G, X, i, j + 1, k) - xc + atf<E3>(G, X, i, j - 1, k) - xc) * (float)G.idy2 +
           (atf<E3>(G, X, i, j, k + 1) - xc + atf<E3>(G, X, i, j, k - 1) - xc) * (float)G.idz2;
}

__device__ __forceinline__ void copy_cellf(const Geo &G, const float *x, float *y)
{
    int i, j, k;
    if (cell(G, i, j, k)) y[id3(G, i, j, k)] = ldf(&x[id3(G, i, j, k)]);
}

// FP64 residuals r0 = b - T(u^n) of the three momentum components, the FP32
// copies of the stencil and the reciprocals, and the first FP32 sweep from
// zero, du = r0 / T_CC; the loop's reference norms are ||r0||^2.
__global__ void k_mx_r0mom(Args a, Mx m)
{
    Sc *sc = a.sc;
    if (sc->status) return;
    __shared__ double red[3 * NT];
    double acc[3] = {0.0, 0.0, 0.0}, tot[3];
    int i, j, k0, k1;
    if (column(a.G, i, j, k0, k1))
#pragma unroll 1
        for (int k = k0; k < k1; ++k) {
            const int q = id3(a.G, i, j, k);
            const W13 c = weights(a, q);
            const double ru = toff<U3>(a, fma(-c.w[0], ld(&a.S.u[q]), ld(&a.bu[q])), c, a.S.u, i, j, k);
            asm volatile("" ::: "memory");
            const double rv = toff<V3>(a, fma(-c.w[0], ld(&a.S.v[q]), ld(&a.bv[q])), c, a.S.v, i, j, k);
            asm volatile("" ::: "memory");
            const double rw = toff<W3>(a, fma(-c.w[0], ld(&a.S.w[q]), ld(&a.bw[q])), c, a.S.w, i, j, k);
#pragma unroll
            for (int s = 0; s < NCF; ++s) m.c[s][q] = (float)c.w[s];
            const float di = (float)ld(&a.dinvu[q]);
            m.dinvu[q] = di;
            m.dinvh[q] = (float)ld(&a.dinvh[q]);
            const float fu = (float)ru, fv = (float)rv, fw = (float)rw;
            m.r0u[q] = fu; m.r0v[q] = fv; m.r0w[q] = fw;
            m.du[0][q] = fu * di; m.dv[0][q] = fv * di; m.dw[0][q] = fw * di;
            acc[0] = fma(ru, ru, acc[0]);
            acc[1] = fma(rv, rv, acc[1]);
            acc[2] = fma(rw, rw, acc[2]);
        }
    if (gsum<3>(acc, red, a.part, &sc->counters[C_MOM], tot)) {
        for (int s = 0; s < 3; ++s) sc->bn2[s] = tot[s];
        sc->done[L_MOM] = 0;
        sc->trips[L_MOM] = 0;
        sc->sweeps[0] = 0;
        if (!isfinite(tot[0]) || !isfinite(tot[1]) || !isfinite(tot[2])) sc->status = GEA_ERR_NONFINITE;
    }
}

// One FP32 Jacobi sweep of the momentum increments (pairs as in the FP64
// step: the second copies once the first met the tolerance).
__global__ void k_mx_mom(Args a, Mx m, const float *ui, const float *vi, const float *wi, float *uo, float *vo,
                         float *wo, int second)
{
    Sc *sc = a.sc;
    if (sc->status) return;
    if (second && sc->done[L_MOM]) {
        copy_cellf(a.G, ui, uo);
        copy_cellf(a.G, vi, vo);
        copy_cellf(a.G, wi, wo);
        return;
    }
    __shared__ double red[3 * NT];
    float acc[3] = {0.0f, 0.0f, 0.0f};
    double tot[3];
    int i, j, k;
    if (cell(a.G, i, j, k)) {
        const Geo &G = a.G;
        const int q = id3(G, i, j, k);
        const W13f c = weightsf(m, q);
        const float di = ldf(&m.dinvu[q]);
        const float u0 = ldf(&ui[q]), v0 = ldf(&vi[q]), w0 = ldf(&wi[q]);
        const float ru = ldf(&m.r0u[q]) - fmaf(c.w[0], u0, tofff<U3>(G, c, ui, i, j, k));
        const float rv = ldf(&m.r0v[q]) - fmaf(c.w[0], v0, tofff<V3>(G, c, vi, i, j, k));
        const float rw = ldf(&m.r0w[q]) - fmaf(c.w[0], w0, tofff<W3>(G, c, wi, i, j, k));
        uo[q] = fmaf(ru, di, u0);
        vo[q] = fmaf(rv, di, v0);
        wo[q] = fmaf(rw, di, w0);
        acc[0] = ru * ru; acc[1] = rv * rv; acc[2] = rw * rw;
    }
    if (gsum<3, float>(acc, red, a.part, &sc->counters[C_MOM], tot)) {
        sc->sweeps[0] += 1;
        if (!isfinite(tot[0]) || !isfinite(tot[1]) || !isfinite(tot[2])) sc->status = GEA_ERR_NONFINITE;
        else if (tot[0] <= m.tol2 * sc->bn2[0] && tot[1] <= m.tol2 * sc->bn2[1] && tot[2] <= m.tol2 * sc->bn2[2])
            sc->done[L_MOM] = 1;
    }
}

// u^{n+1/3} = u^n + du (FP64).
__global__ void k_mx_u1(Args a, const float *du, const float *dv, const float *dw)
{
    if (a.sc->status) return;
    int i, j, k;
    if (!cell(a.G, i, j, k)) return;
    const int q = id3(a.G, i, j, k);
    a.ua[q] = ld(&a.S.u[q]) + (double)ldf(&du[q]);
    a.va[q] = ld(&a.S.v[q]) + (double)ldf(&dv[q]);
    a.wa[q] = ld(&a.S.w[q]) + (double)ldf(&dw[q]);
}

// FP64 residual r0 = b_h - T_h(h^n) (h^n with its wall rule), rounded to FP32,
// and the first FP32 sweep dh = r0 / T_h,CC; the loop's reference ||r0||^2.
__global__ void k_mx_r0h(Args a, Mx m)
{
    Sc *sc = a.sc;
    if (sc->status) return;
    __shared__ double red[NT];
    double acc[1] = {0.0}, tot[1];
    int i, j, k0, k1;
    if (column(a.G, i, j, k0, k1))
#pragma unroll 1
        for (int k = k0; k < k1; ++k) {
            const int q = id3(a.G, i, j, k);
            const W13 c = weights(a, q);
            double r0 = toff<H3>(a, fma(-c.w[0], ld(&a.S.h[q]), ld(&a.bh[q])), c, a.S.h, i, j, k);
            gea::rarely(a.F.pr_ne1, [&] { r0 = fma(a.F.nuh - a.F.mu, lap<H3>(a, a.S.h, i, j, k), r0); });
            const float f = (float)r0;
            m.r0h[q] = f;
            m.dh[0][q] = f * ldf(&m.dinvh[q]);
            acc[0] = fma(r0, r0, acc[0]);
        }
    if (gsum<1>(acc, red, a.part, &sc->counters[C_ENTH], tot)) {
        sc->bn2[3] = tot[0];
        sc->done[L_ENTH] = 0;
        sc->trips[L_ENTH] = 0;
        sc->sweeps[1] = 0;
        if (!isfinite(tot[0])) sc->status = GEA_ERR_NONFINITE;
    }
}

// One FP32 Jacobi sweep of the enthalpy increment (even ghosts).
__global__ void k_mx_enth(Args a, Mx m, const float *hi, float *ho, int second)
{
    Sc *sc = a.sc;
    if (sc->status) return;
    if (second && sc->done[L_ENTH]) {
        copy_cellf(a.G, hi, ho);
        return;
    }
    __shared__ double red[NT];
    float acc[1] = {0.0f};
    double tot[1];
    int i, j, k;
    if (cell(a.G, i, j, k)) {
        const Geo &G = a.G;
        const int q = id3(G, i, j, k);
        const W13f c = weightsf(m, q);
        const float h0 = ldf(&hi[q]);
        float t = fmaf(c.w[0], h0, tofff<E3>(G, c, hi, i, j, k));
        gea::rarely(a.F.pr_ne1, [&] { t = fmaf((float)(a.F.mu - a.F.nuh), lapf(G, hi, i, j, k), t); });
        const float r = ldf(&m.r0h[q]) - t;
        ho[q] = fmaf(r, ldf(&m.dinvh[q]), h0);
        acc[0] = r * r;
    }
    if (gsum<1, float>(acc, red, a.part, &sc->counters[C_ENTH], tot)) {
        sc->sweeps[1] += 1;
        if (!isfinite(tot[0])) sc->status = GEA_ERR_NONFINITE;
        else if (tot[0] <= m.tol2 * sc->bn2[3]) sc->done[L_ENTH] = 1;
    }
}

// h^{n+1} = h^n + dh into ha (FP64).
__global__ void k_mx_h1(Args a, const float *dh)
{
    if (a.sc->status) return;
    int i, j, k;
    if (!cell(a.G, i, j, k)) return;
    const int q = id3(a.G, i, j, k);
    a.ha[q] = ld(&a.S.h[q]) + (double)ldf(&dh[q]);
}

// ---- loop control and step bookkeeping (one thread) ----

__global__ void k_ctl(Sc *sc, cudaGraphConditionalHandle h, int graph, int which, int maxtrips, int body)
{
    const int trips = ++sc->trips[which];
    const int done = sc->done[which];
    sc->launches += body;
    if (!done && !sc->status && trips >= maxtrips) sc->status = GEA_ERR_NOCONV;
    if (graph) cudaGraphSetConditional(h, (done || sc->status || trips >= maxtrips) ? 0u : 1u);
}

__global__ void k_begin(Sc *sc)
{
    for (int c = 0; c < 4; ++c) { sc->cg_iters[c] = 0; sc->cg_relres[c] = 0.0; }
}

__global__ void k_end(Sc *sc, int fixed)
{
    sc->launches += fixed;
    if (sc->status) {
        sc->last_status = sc->status;
        return;
    }
    sc->steps_done += 1;
    sc->last_sweeps[0] = sc->sweeps[0];
    sc->last_sweeps[1] = sc->sweeps[1];
    for (int c = 0; c < 4; ++c) {
        sc->last_cg_iters[c] = sc->cg_iters[c];
        sc->last_cg_relres[c] = sc->cg_relres[c];
    }
    sc->last_status = 0;
}

}  // namespace g3

using namespace g3;

struct gea3d_ctx {
    Geo G;
    Phy F;
    gea_constants C;
    cudaStream_t stream = nullptr, cap = nullptr, cap2 = nullptr;
    std::vector<void *> allocs;
    St S[2];
    double *rho1, *dinvu, *dinvh, *bu, *bv, *bw, *ua, *va, *wa, *ub, *vb, *wb, *bh, *ha, *hb;
    double *rho2, *psi, *Dx, *Dy, *Dz, *Hx, *Hy, *Hz;
    Rb<double> rb{};                      // the pressure solve's vectors (FP64 step)
    Rb<float> rbf{};                      // (mixed step)
    double *dtr1;                         // dt / rho1
    double *kin;                          // K1
    double *mueff = nullptr;              // LES eddy viscosity field
    double *gz = nullptr;                 // g z: nz cell centres, then nz + 1 horizontal faces
    bool mixed = false;                   // GEA_FLAG_MIXED
    Mx mx{};                              // FP32 data of the mixed step
    Cf cf;                                // transport stencil weights
    double *stage = nullptr;              // dense conservative fields (5 arrays)
    std::vector<Lev> L;                   // the FP64 fine-level operator
    std::vector<Lev32> M;                 // the FP32 multigrid hierarchy
    Sc *sc = nullptr;
    double *part = nullptr;
    cudaGraph_t graph[2] = {nullptr, nullptr};
    cudaGraphExec_t exec[2] = {nullptr, nullptr};
    bool have_state = false;
    long long steps_at_sync = 0;
    char err[256] = {0};
};

namespace {

int fail3(gea3d_ctx *c, int code, const char *fmt, ...)
{
    if (c) {
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(c->err, sizeof(c->err), fmt, ap);
        va_end(ap);
    }
    return code;
}

#define CK3(call)                                                                                   \
    do {                                                                                            \
        cudaError_t e_ = (call);                                                                    \
        if (e_ != cudaSuccess)                                                                      \
            return fail3(ctx, GEA_ERR_CUDA, "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, \
                         __LINE__);                                                                 \
    } while (0)

Geo make_geo(int nx, int ny, int nz, double lx, double ly, double lz)
{
    Geo G;
    G.nx = nx; G.ny = ny; G.nz = nz;
    G.P = (nx + 1 + 31) / 32 * 32;
    G.dx = lx / nx; G.dy = ly / ny; G.dz = lz / nz;
    G.idx = 1.0 / G.dx; G.idy = 1.0 / G.dy; G.idz = 1.0 / G.dz;
    G.idx2 = 1.0 / (G.dx * G.dx); G.idy2 = 1.0 / (G.dy * G.dy); G.idz2 = 1.0 / (G.dz * G.dz);
    G.ivol = 1.0 / (G.dx * G.dy * G.dz);
    G.ax = G.dy * G.dz; G.ay = G.dx * G.dz; G.az = G.dx * G.dy;
    G.hidx = 0.5 * G.idx; G.hidy = 0.5 * G.idy; G.hidz = 0.5 * G.idz;
    G.tidx = 2.0 * G.idx; G.tidy = 2.0 * G.idy; G.tidz = 2.0 * G.idz;
    G.hax = 0.5 * G.ax; G.hay = 0.5 * G.ay; G.haz = 0.5 * G.az;
    G.s12 = G.ivol / 12.0;
    return G;
}

// elements of one array (cells or faces) of a level
size_t elems(const Geo &G) { return (size_t)(G.nz + 1) * (G.ny + 1) * G.P; }

// Diagnostics (Remark 2) in three dimensions: theta' = T (p0/p)^(R/cp) -
// theta_bar(z) per cell into th (dense nz x ny x nx, x fastest; optional),
// mass = sum rho V and energy = sum rho (cv T + |u|^2/2 + g z) V (Section
// 2.1's total energy) into the scalars.
__global__ void k_diag3(Geo G, Phy F, double p0, St S, const double *thbar, const double *gzc, double *th, Sc *sc,
                        double *part)
{
    __shared__ double red[2 * NT];
    int i, j, k;
    double v[2] = {0.0, 0.0};
    if (cell(G, i, j, k)) {
        const int q = id3(G, i, j, k);
        const double T = ld(&S.T[q]), rho = ld(&S.rho[q]);
        if (th) th[((size_t)k * G.ny + j) * G.nx + i] = T / pow(ld(&S.p[q]) / p0, F.R / F.cp) - ld(&thbar[k]);
        const double u = ld(&S.u[q]), vv = ld(&S.v[q]), w = ld(&S.w[q]);
        const double V = G.dx * G.dy * G.dz;
        const double K = 0.5 * (u * u + vv * vv + w * w);
        v[0] = rho * V;
        v[1] = rho * ((F.cp - F.R) * T + K + ld(&gzc[k])) * V;
    }
    double tot[2];
    if (gsum<2>(v, red, part, &sc->counters[C_DIAG], tot)) {
        sc->mass = tot[0];
        sc->energy = tot[1];
    }
}

dim3 grid_of(const Geo &G) { return dim3((G.nx + TX - 1) / TX, (G.ny + TY - 1) / TY, G.nz); }
// The grid of the column kernels: up to `most` layers per block, fewer where
// that would leave less than kMinBlocks blocks, about three waves of five
// blocks on each of 152 SMs (a grid of 33 x 33 x 24 has 240 one-layer tiles in
// all). Lines measured in us a step, FP64 / mixed. kMinBlocks 1200, 2400, 4800:
// 96 x 96 x 96 2274, 2237, 2237 / 1533, 1519, 1512; 192 x 192 x 96 6632, 6670,
// 6809 / 4644, 4660, 4745; without columns 6926 / 4813. kLayersHeavy (the stencil
// kernels) 1, 2, 4, 8 at 256 x 256 x 128: 15126, 14723, 14668, 14827 / 10740,
// 10530, 10455, 10489. kLayers (the light CG kernels) 4, 8 and 16 differ by less
// than 0.2 % there.
constexpr int kLayers = 8, kLayersHeavy = 4, kMinBlocks = 2400;
dim3 columns_of(const Geo &G, const dim3 &g, int most)
{
    int layers = most;
    while (layers > 1 && (size_t)g.x * g.y * ((G.nz + layers - 1) / layers) < (size_t)kMinBlocks) layers /= 2;
    return dim3(g.x, g.y, (G.nz + layers - 1) / layers);
}
// The grids over pairs of cells: one layer a block, and columns.
dim3 grid_pairs(const Geo &G) { return dim3(((G.nx + 1) / 2 + TX - 1) / TX, (G.ny + TY - 1) / TY, G.nz); }
const dim3 kBlk(TX, TY);
size_t nblocks(const Geo &G)
{
    const dim3 g = grid_of(G);
    return (size_t)g.x * g.y * g.z;
}

Args args_of(gea3d_ctx *c, int from)
{
    Args a;
    a.G = c->G; a.F = c->F;
    a.S = c->S[from]; a.N = c->S[from ^ 1];
    a.rho1 = c->rho1; a.dinvu = c->dinvu; a.dinvh = c->dinvh;
    a.bu = c->bu; a.bv = c->bv; a.bw = c->bw;
    a.ua = c->ua; a.va = c->va; a.wa = c->wa; a.ub = c->ub; a.vb = c->vb; a.wb = c->wb;
    a.bh = c->bh; a.ha = c->ha; a.hb = c->hb;
    a.rho2 = c->rho2; a.psi = c->psi; a.Dx = c->Dx; a.Dy = c->Dy; a.Dz = c->Dz;
    a.Hx = c->Hx; a.Hy = c->Hy; a.Hz = c->Hz;
    a.cf = c->cf;
    a.dtr1 = c->dtr1;
    a.kin = c->kin;
    a.mueff = c->mueff;
    a.gzc = c->gz;
    a.gzf = c->gz + c->G.nz;
    a.gx2 = a.gzf + c->G.nz + 1;
    a.gy2 = a.gx2 + c->G.nz;
    a.gz2 = a.gy2 + c->G.nz;
    a.sc = c->sc; a.part = c->part;
    a.jtol2 = c->C.jac_rtol * c->C.jac_rtol;
    a.ctol2 = c->C.cg_rtol * c->C.cg_rtol;
    return a;
}

// WHILE node on the graph captured on s; body(stream, handle) captured into it
template <class Body>
int capture_while3(gea3d_ctx *ctx, cudaStream_t s, Body body)
{
    cudaStreamCaptureStatus cs;
    cudaGraph_t g;
    const cudaGraphNode_t *deps = nullptr;
    const cudaGraphEdgeData *edges = nullptr;
    size_t ndeps = 0;
    CK3(cudaStreamGetCaptureInfo(s, &cs, nullptr, &g, &deps, &edges, &ndeps));
    if (cs != cudaStreamCaptureStatusActive) return fail3(ctx, GEA_ERR_CUDA, "capture not active");
    cudaGraphConditionalHandle h;
    CK3(cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault));
    cudaGraphNodeParams prm = {cudaGraphNodeTypeConditional};
    prm.conditional.handle = h;
    prm.conditional.type = cudaGraphCondTypeWhile;
    prm.conditional.size = 1;
    cudaGraphNode_t node;
    CK3(cudaGraphAddNode(&node, g, deps, edges, ndeps, &prm));
    CK3(cudaStreamUpdateCaptureDependencies(s, &node, nullptr, 1, cudaStreamSetCaptureDependencies));
    CK3(cudaStreamBeginCaptureToGraph(ctx->cap2, prm.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                      cudaStreamCaptureModeThreadLocal));
    body(ctx->cap2, h);
    cudaGraph_t out = nullptr;
    CK3(cudaStreamEndCapture(ctx->cap2, &out));
    return GEA_OK;
}

// Event pairs around the launches of an eager step (per-kernel timing). A
// solver-loop kernel launched after its loop finished returns at once (a
// converged solve, or the second Jacobi sweep of a pair that copies): it is
// recorded with zero cells, the loop's flags read before the launch.
struct Trace3 {
    struct Rec {
        const char *name;
        long long cells;
        cudaEvent_t e0, e1;
    };
    std::vector<Rec> recs;
    const Sc *dsc = nullptr;
    // the loop whose finished flag makes the kernel return, or -1
    static int gate(const char *name)
    {
        static const char *cg[] = {"g3_rb_start",  "g3_mg_down",     "g3_mg_black",      "g3_mg_red",
                                   "g3_mg_up",     "g3_pupd",        "g3_spmv_red",      "g3_spmv_black",
                                   "g3_update",    "g3_mx_rb_start", "g3_mx_mg_up",      "g3_mx_pupd",
                                   "g3_mx_spmv_red", "g3_mx_spmv_black", "g3_mx_update"};
        for (const char *c : cg)
            if (!strcmp(name, c)) return L_CG;
        if (!strcmp(name, "g3_mom") || !strcmp(name, "g3_mx_mom")) return L_MOM;
        if (!strcmp(name, "g3_enth") || !strcmp(name, "g3_mx_enth")) return L_ENTH;
        return -1;
    }
    ~Trace3()
    {
        for (auto &r : recs) {
            cudaEventDestroy(r.e0);
            cudaEventDestroy(r.e1);
        }
    }
};

// Run go() (one launch on st), bracketed by an event pair when tracing.
template <class Go>
void traced(Trace3 *tr, const char *name, const Geo &G, cudaStream_t st, Go go)
{
    if (!tr) {
        go();
        return;
    }
    Trace3::Rec r{name, (long long)G.nx * G.ny * G.nz, nullptr, nullptr};
    const int g = Trace3::gate(name);
    if (g >= 0 && tr->dsc) {
        Sc h;
        if (cudaMemcpyAsync(&h, tr->dsc, sizeof(Sc), cudaMemcpyDeviceToHost, st) == cudaSuccess &&
            cudaStreamSynchronize(st) == cudaSuccess && (h.status || h.done[g]))
            r.cells = 0;
    }
    cudaEventCreate(&r.e0);
    cudaEventCreate(&r.e1);
    cudaEventRecord(r.e0, st);
    go();
    cudaEventRecord(r.e1, st);
    tr->recs.push_back(r);
}

// Run a loop body eagerly until its control kernel reports the loop over.
template <class Body>
int eager_while3(gea3d_ctx *ctx, cudaStream_t s, int which, int maxtrips, Body body)
{
    for (int t = 0; t < maxtrips + 1; ++t) {
        body(s, (cudaGraphConditionalHandle)0);
        Sc h;
        CK3(cudaMemcpyAsync(&h, ctx->sc, sizeof(Sc), cudaMemcpyDeviceToHost, s));
        CK3(cudaStreamSynchronize(s));
        if (h.done[which] || h.status || h.trips[which] >= maxtrips) break;
    }
    return GEA_OK;
}

// z = M^-1 rb (one FP32 V-cycle; nothing to do on one level); returns launches
template <class R>
int vcycle(gea3d_ctx *ctx, const Args &a, const Rb<R> &v, cudaStream_t st, Trace3 *tr)
{
    Lev32 *M = ctx->M.data();
    const int nlev = (int)ctx->M.size();
    if (nlev == 1) return 0;
    int n = 0;
    auto black = [&](const Lev32 &f, const float *ec, const Geo &cg, float *out) {
        traced(tr, "g3_mg_black", f.G, st, [&] { k_mg_black<<<grid_pairs(f.G), kBlk, 0, st>>>(f, ec, cg, out, a.sc); });
        ++n;
    };
    auto red = [&](const Lev32 &f) {
        traced(tr, "g3_mg_red", f.G, st, [&] { k_mg_red<<<grid_pairs(f.G), kBlk, 0, st>>>(f, f.e2, a.sc); });
        ++n;
    };
    traced(tr, "g3_mg_down", M[1].G, st, [&] {
        k_mg_down<true><<<grid_of(M[1].G), kBlk, 0, st>>>(M[0], v.ef, M[1], a.sc);
    });
    ++n;
    for (int l = 1; l + 1 < nlev; ++l) {
        black(M[l], nullptr, M[l].G, M[l].e);
        traced(tr, "g3_mg_down", M[l + 1].G, st, [&] {
            k_mg_down<false><<<grid_of(M[l + 1].G), kBlk, 0, st>>>(M[l], M[l].e, M[l + 1], a.sc);
        });
        ++n;
    }
    // the coarsest level: one symmetric red-black sweep
    for (int l = nlev - 1; l >= 1; --l) {
        black(M[l], l == nlev - 1 ? nullptr : M[l + 1].e2, l == nlev - 1 ? M[l].G : M[l + 1].G, M[l].e2);
        red(M[l]);
    }
    const Geo &G = ctx->G;
    traced(tr, ctx->mixed ? "g3_mx_mg_up" : "g3_mg_up", G, st, [&] {
        k_mg_up<R><<<columns_of(G, grid_pairs(G), kLayers), kBlk, 0, st>>>(M[0], v, M[1].e2, M[1].G, a.sc, a.part);
    });
    return n + 1;
}

// One pressure solve of corrector c from x = xin into N.pp: residual, CG on
// the black half to the relative residual tol2 (squared) and the solution.
// A: the operator in the solve's precision, r its start residual.
template <class R, class Loop>
int solve_pressure(gea3d_ctx *ctx, const Args &a, const Op<R> &A, R *r, const Rb<R> &v, double tol2, const double *xin,
                   int c, cudaStream_t s, bool graph, Trace3 *tr, Loop loop, int &fixed)
{
    const Geo &G = ctx->G;
    const bool mx = ctx->mixed, single = ctx->M.size() == 1;
    const float *wf = ctx->M[0].w;
    const dim3 pairs = grid_pairs(G), cols = columns_of(G, pairs, kLayers);
    const int nlev = (int)ctx->M.size(), gr = graph ? 1 : 0;
    traced(tr, "g3_helm_rhs", G, s, [&] {
        k_helm_rhs<R><<<columns_of(G, grid_of(G), kLayersHeavy), kBlk, 0, s>>>(a, ctx->L[0], xin, c, r, A.wd, v.w);
    });
    traced(tr, mx ? "g3_mx_rb_start" : "g3_rb_start", G, s, [&] {
        if (single) k_rb_start<R, true><<<cols, kBlk, 0, s>>>(A, r, wf, v, a.sc, a.part);
        else k_rb_start<R, false><<<cols, kBlk, 0, s>>>(A, r, wf, v, a.sc, a.part);
    });
    fixed += 2 + vcycle<R>(ctx, a, v, s, tr);
    const int body = 4 + (nlev == 1 ? 0 : 4 * (nlev - 1)) + 1;
    const int rc = loop(L_CG, ctx->C.cg_maxit, [&](cudaStream_t bs, cudaGraphConditionalHandle h) {
        traced(tr, mx ? "g3_mx_pupd" : "g3_pupd", G, bs, [&] { k_pupd<R><<<pairs, kBlk, 0, bs>>>(G, v, a.sc); });
        traced(tr, mx ? "g3_mx_spmv_red" : "g3_spmv_red", G, bs,
               [&] { k_spmv_red<R><<<pairs, kBlk, 0, bs>>>(A, v, a.sc); });
        traced(tr, mx ? "g3_mx_spmv_black" : "g3_spmv_black", G, bs,
               [&] { k_spmv_black<R><<<cols, kBlk, 0, bs>>>(A, v, a.sc, a.part); });
        traced(tr, mx ? "g3_mx_update" : "g3_update", G, bs, [&] {
            if (single) k_update<R, true><<<cols, kBlk, 0, bs>>>(G, wf, v, tol2, a.sc, a.part);
            else k_update<R, false><<<cols, kBlk, 0, bs>>>(G, wf, v, tol2, a.sc, a.part);
        });
        vcycle<R>(ctx, a, v, bs, tr);
        k_ctl<<<1, 1, 0, bs>>>(a.sc, h, gr, L_CG, ctx->C.cg_maxit, body);
    });
    if (rc) return rc;
    traced(tr, mx ? "g3_mx_solution" : "g3_solution", G, s, [&] {
        k_solution<R><<<pairs, kBlk, 0, s>>>(A, r, v, xin, a.N.pp, a.sc);
    });
    ++fixed;
    return GEA_OK;
}

// The kernel sequence of one step reading slot `from` (Section 3: Step 1,
// Step 2, n_corr PISO correctors). graph: captured on s, the loops as WHILE
// nodes; otherwise launched eagerly with host-checked loops, each launch
// bracketed by tr (if given).
int record3(gea3d_ctx *ctx, int from, cudaStream_t s, bool graph, Trace3 *tr)
{
    const Args a = args_of(ctx, from);
    Lev *L = ctx->L.data();
    Lev32 *M = ctx->M.data();
    const int nlev = (int)ctx->M.size();
    const Geo &G = ctx->G;
    const dim3 grid = grid_of(G);
    const dim3 gridh = columns_of(G, grid, kLayersHeavy);   // column kernels
    const int jtrips = (ctx->C.jac_maxit + 1) / 2;
    const int gr = graph ? 1 : 0;
    int fixed = 0, rc;
    auto loop = [&](int which, int maxtrips, auto body) {
        return graph ? capture_while3(ctx, s, body) : eager_while3(ctx, s, which, maxtrips, body);
    };
    k_begin<<<1, 1, 0, s>>>(a.sc); ++fixed;
    if (ctx->mueff) { traced(tr, "g3_les", G, s, [&] { k_les<<<grid, kBlk, 0, s>>>(a); }); ++fixed; }
    traced(tr, "g3_pred", G, s, [&] { k_pred<<<gridh, kBlk, 0, s>>>(a); }); ++fixed;
    const Mx &m = ctx->mx;
    if (ctx->mixed) {
        // FP64 residuals, FP32 Jacobi on the increments (pairs end in du[0]), FP64 update
        traced(tr, "g3_mx_r0mom", G, s, [&] { k_mx_r0mom<<<gridh, kBlk, 0, s>>>(a, m); }); ++fixed;
        rc = loop(L_MOM, jtrips, [&](cudaStream_t bs, cudaGraphConditionalHandle h) {
            traced(tr, "g3_mx_mom", G, bs, [&] {
                k_mx_mom<<<grid, kBlk, 0, bs>>>(a, m, m.du[0], m.dv[0], m.dw[0], m.du[1], m.dv[1], m.dw[1], 0);
            });
            traced(tr, "g3_mx_mom", G, bs, [&] {
                k_mx_mom<<<grid, kBlk, 0, bs>>>(a, m, m.du[1], m.dv[1], m.dw[1], m.du[0], m.dv[0], m.dw[0], 1);
            });
            k_ctl<<<1, 1, 0, bs>>>(a.sc, h, gr, L_MOM, jtrips, 3);
        });
        if (rc) return rc;
        traced(tr, "g3_mx_u1", G, s, [&] { k_mx_u1<<<grid, kBlk, 0, s>>>(a, m.du[0], m.dv[0], m.dw[0]); }); ++fixed;
    } else {
        rc = loop(L_MOM, jtrips, [&](cudaStream_t bs, cudaGraphConditionalHandle h) {
            traced(tr, "g3_mom", G, bs, [&] { k_mom<<<gridh, kBlk, 0, bs>>>(a, a.ua, a.va, a.wa, a.ub, a.vb, a.wb, 0); });
            traced(tr, "g3_mom", G, bs, [&] { k_mom<<<gridh, kBlk, 0, bs>>>(a, a.ub, a.vb, a.wb, a.ua, a.va, a.wa, 1); });
            k_ctl<<<1, 1, 0, bs>>>(a.sc, h, gr, L_MOM, jtrips, 3);
        });
        if (rc) return rc;
    }
    traced(tr, "g3_kin", G, s, [&] { k_kin<<<grid, kBlk, 0, s>>>(a, a.ua, a.va, a.wa); }); ++fixed;
    traced(tr, "g3_enth_rhs", G, s, [&] { k_enth_rhs<<<gridh, kBlk, 0, s>>>(a, a.wa); }); ++fixed;
    if (ctx->mixed) {
        traced(tr, "g3_mx_r0h", G, s, [&] { k_mx_r0h<<<gridh, kBlk, 0, s>>>(a, m); }); ++fixed;
        rc = loop(L_ENTH, jtrips, [&](cudaStream_t bs, cudaGraphConditionalHandle h) {
            traced(tr, "g3_mx_enth", G, bs, [&] { k_mx_enth<<<grid, kBlk, 0, bs>>>(a, m, m.dh[0], m.dh[1], 0); });
            traced(tr, "g3_mx_enth", G, bs, [&] { k_mx_enth<<<grid, kBlk, 0, bs>>>(a, m, m.dh[1], m.dh[0], 1); });
            k_ctl<<<1, 1, 0, bs>>>(a.sc, h, gr, L_ENTH, jtrips, 3);
        });
        if (rc) return rc;
        traced(tr, "g3_mx_h1", G, s, [&] { k_mx_h1<<<grid, kBlk, 0, s>>>(a, m.dh[0]); }); ++fixed;
    } else {
        rc = loop(L_ENTH, jtrips, [&](cudaStream_t bs, cudaGraphConditionalHandle h) {
            traced(tr, "g3_enth", G, bs, [&] { k_enth<<<gridh, kBlk, 0, bs>>>(a, a.ha, a.hb, 0); });
            traced(tr, "g3_enth", G, bs, [&] { k_enth<<<gridh, kBlk, 0, bs>>>(a, a.hb, a.ha, 1); });
            k_ctl<<<1, 1, 0, bs>>>(a.sc, h, gr, L_ENTH, jtrips, 3);
        });
        if (rc) return rc;
    }
    traced(tr, "g3_eos", G, s, [&] { k_eos<<<grid, kBlk, 0, s>>>(a, L[0], M[0], a.ha); }); ++fixed;
    traced(tr, "g3_faces", G, s, [&] { k_faces<<<grid, kBlk, 0, s>>>(a, L[0], M[0]); }); ++fixed;
    traced(tr, "g3_diag", G, s, [&] {
        if (ctx->mixed) k_diag<false><<<grid, kBlk, 0, s>>>(L[0], M[0], a.sc);
        else k_diag<true><<<grid, kBlk, 0, s>>>(L[0], M[0], a.sc);
    });
    ++fixed;
    for (int l = 0; l + 1 < nlev; ++l, ++fixed)
        traced(tr, "g3_coarsen", M[l + 1].G, s, [&] {
            k_coarsen<<<grid_of(M[l + 1].G), kBlk, 0, s>>>(M[l], M[l + 1]);
        });
    const Op<double> A{G, L[0].d, L[0].ax, L[0].ay, L[0].az, L[0].wd};
    const Op<float> Af{G, M[0].d, M[0].ax, M[0].ay, M[0].az, M[0].w};
    for (int c = 0; c < ctx->C.n_corr; ++c) {
        const double *U = c == 0 ? a.ua : a.N.u, *V = c == 0 ? a.va : a.N.v, *W = c == 0 ? a.wa : a.N.w;
        traced(tr, "g3_H", G, s, [&] { k_H<<<grid, kBlk, 0, s>>>(a, U, V, W); }); ++fixed;
        const double *xin = c == 0 ? a.S.pp : a.N.pp;
        rc = ctx->mixed ? solve_pressure<float>(ctx, a, Af, m.r, ctx->rbf, m.tol2, xin, c, s, graph, tr, loop, fixed)
                        : solve_pressure<double>(ctx, a, A, L[0].r, ctx->rb, a.ctol2, xin, c, s, graph, tr, loop, fixed);
        if (rc) return rc;
        traced(tr, "g3_correct", G, s, [&] { k_correct<<<grid, kBlk, 0, s>>>(a); }); ++fixed;
    }
    ++fixed;
    k_end<<<1, 1, 0, s>>>(a.sc, fixed);
    return cudaGetLastError() == cudaSuccess ? GEA_OK : fail3(ctx, GEA_ERR_CUDA, "kernel launch failed");
}

int build3(gea3d_ctx *ctx, int from)
{
    cudaStream_t s = ctx->cap;
    CK3(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    const int rc = record3(ctx, from, s, true, nullptr);
    cudaGraph_t g = nullptr;
    const cudaError_t e = cudaStreamEndCapture(s, &g);
    if (rc) {
        if (g) cudaGraphDestroy(g);
        return rc;
    }
    if (e != cudaSuccess) return fail3(ctx, GEA_ERR_CUDA, "graph capture: %s", cudaGetErrorString(e));
    ctx->graph[from] = g;
    CK3(cudaGraphInstantiate(&ctx->exec[from], g, 0));
    return GEA_OK;
}

}  // namespace

extern "C" {

int gea3d_create(const gea3d_grid *grid, const gea_constants *c, gea3d_ctx **out)
{
    if (!grid || !c || !out) return GEA_ERR_INVAL;
    *out = nullptr;
    if (grid->nx < 4 || grid->ny < 4 || grid->nz < 4 || !(grid->lx > 0) || !(grid->ly > 0) || !(grid->lz > 0))
        return GEA_ERR_INVAL;
    if ((long long)grid->nx * grid->ny * grid->nz > (1LL << 31) / 4) return GEA_ERR_INVAL;
    // the kernels index a field (ghost layers and row padding included) with
    // 32-bit integers
    if ((long long)(grid->nz + 1) * (grid->ny + 1) * ((grid->nx + 1 + 31) / 32 * 32) > INT_MAX) return GEA_ERR_INVAL;
    if (!(c->R > 0) || !(c->cp > c->R) || !(c->g >= 0) || !(c->p0 > 0) || !(c->mu >= 0) || !(c->Pr > 0) ||
        !(c->dt > 0) || c->n_corr < 1 || c->n_corr > 4 || !(c->jac_rtol > 0) || c->jac_maxit < 1 ||
        !(c->cg_rtol > 0) || c->cg_maxit < 1 || c->mg_min_cells < 0 || (c->flags & ~GEA_FLAG_MIXED) != 0 ||
        c->reading_flags != 0 ||
        (!(c->flags & GEA_FLAG_MIXED) && c->mp_rtol != 0.0) ||
        ((c->flags & GEA_FLAG_MIXED) && c->mp_rtol != 0.0 && !(c->mp_rtol >= 1e-7 && c->mp_rtol < 1.0)) ||
        !(c->cs >= 0.0) || (c->cs > 0.0 && c->Pr != 1.0))
        return GEA_ERR_INVAL;
    gea3d_ctx *ctx = new gea3d_ctx();
    ctx->C = *c;
    ctx->G = make_geo(grid->nx, grid->ny, grid->nz, grid->lx, grid->ly, grid->lz);
    ctx->F.R = c->R; ctx->F.cp = c->cp; ctx->F.g = c->g; ctx->F.mu = c->mu; ctx->F.nuh = c->mu / c->Pr;
    ctx->F.dt = c->dt; ctx->F.idt = 1.0 / c->dt; ctx->F.icp = 1.0 / c->cp;
    {
        const double delta = cbrt(ctx->G.dx * ctx->G.dy * ctx->G.dz);
        ctx->F.les_d2 = c->cs * c->cs * delta * delta;
        Phy &F = ctx->F;
        const Geo &g = ctx->G;
        F.icv = 1.0 / (c->cp - c->R);
        F.mux = F.mu * g.idx2; F.muy = F.mu * g.idy2; F.muz = F.mu * g.idz2;
        F.mud = 2.0 * (F.mux + F.muy + F.muz);
        F.nud = 2.0 * F.nuh * (g.idx2 + g.idy2 + g.idz2);
        F.les = F.les_d2 > 0.0 ? 1 : 0;
        F.pr_ne1 = F.nuh != F.mu ? 1 : 0;
    }
    // multigrid levels: halve all three sizes while they are even and >= 8
    // and (unless mg_min_cells is given) the Laplacian-to-diagonal estimate
    // 2 dt^2 R T (1/dx^2 + 1/dy^2 + 1/dz^2) exceeds 1
    std::vector<Geo> lg{ctx->G};
    double ratio = 2.0 * c->dt * c->dt * c->R * kRefT *
                   (1.0 / (ctx->G.dx * ctx->G.dx) + 1.0 / (ctx->G.dy * ctx->G.dy) + 1.0 / (ctx->G.dz * ctx->G.dz));
    for (;;) {
        const Geo &f = lg.back();
        if (f.nx % 2 || f.ny % 2 || f.nz % 2 || f.nx < 8 || f.ny < 8 || f.nz < 8) break;
        if (c->mg_min_cells > 0 && (long long)f.nx * f.ny * f.nz <= c->mg_min_cells) break;
        if (c->mg_min_cells == 0 && ratio <= kCoarsestRatio) break;
        if ((int)lg.size() >= kMaxLev) break;
        lg.push_back(make_geo(f.nx / 2, f.ny / 2, f.nz / 2, f.nx * f.dx, f.ny * f.dy, f.nz * f.dz));
        ratio *= 0.25;
    }
    bool ok = true;
    auto take = [&](size_t n) -> double * {
        void *p = nullptr;
        if (!ok) return nullptr;
        if (cudaMalloc(&p, n * sizeof(double)) != cudaSuccess) {
            cudaGetLastError();
            ok = false;
            return nullptr;
        }
        cudaMemset(p, 0, n * sizeof(double));
        ctx->allocs.push_back(p);
        return static_cast<double *>(p);
    };
    const size_t E = elems(ctx->G);
    for (int s = 0; s < 2; ++s) {
        St &S = ctx->S[s];
        double **f[12] = {&S.rho, &S.u, &S.v, &S.w, &S.T, &S.h, &S.p, &S.pp, &S.pold, &S.phix, &S.phiy, &S.phiz};
        for (auto pp : f) *pp = take(E);
    }
    double **sc[] = {&ctx->rho1, &ctx->dinvu, &ctx->dinvh, &ctx->bu, &ctx->bv, &ctx->bw, &ctx->ua, &ctx->va,
                     &ctx->wa, &ctx->ub, &ctx->vb, &ctx->wb, &ctx->bh, &ctx->ha, &ctx->hb, &ctx->rho2,
                     &ctx->psi, &ctx->Dx, &ctx->Dy, &ctx->Dz, &ctx->Hx, &ctx->Hy, &ctx->Hz};
    for (auto pp : sc) *pp = take(E);
    for (int m = 0; m < NCF; ++m) ctx->cf.c[m] = take(E);
    ctx->dtr1 = take(E);
    ctx->kin = take(E);
    if (c->cs > 0.0) ctx->mueff = take(E);
    {
        // the heights g z of the cell centres and of the horizontal faces,
        // rounded as the expressions g ((k + 1/2) dz) and g (k dz)
        const int nz = ctx->G.nz;
        std::vector<double> h(5 * (size_t)nz + 2);
        for (int k = 0; k < nz; ++k) h[k] = c->g * ((k + 0.5) * ctx->G.dz);
        for (int k = 0; k <= nz; ++k) h[nz + k] = c->g * (k * ctx->G.dz);
        // and twice these over the spacings (Args::gx2, gy2, gz2)
        double *t = h.data() + 2 * nz + 1;
        for (int k = 0; k < nz; ++k) t[k] = h[k] * ctx->G.tidx;
        for (int k = 0; k < nz; ++k) t[nz + k] = h[k] * ctx->G.tidy;
        for (int k = 0; k <= nz; ++k) t[2 * nz + k] = h[nz + k] * ctx->G.tidz;
        ctx->gz = take(h.size());
        if (ctx->gz && cudaMemcpy(ctx->gz, h.data(), h.size() * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess)
            ok = false;
    }
    ctx->mixed = (c->flags & GEA_FLAG_MIXED) != 0;
    if (ctx->mixed) {
        Mx &m = ctx->mx;
        auto tf = [&]() { return reinterpret_cast<float *>(take((E + 1) / 2)); };
        for (int s = 0; s < NCF; ++s) m.c[s] = tf();
        m.dinvu = tf(); m.dinvh = tf(); m.r0u = tf(); m.r0v = tf(); m.r0w = tf(); m.r0h = tf();
        for (int b = 0; b < 2; ++b) { m.du[b] = tf(); m.dv[b] = tf(); m.dw[b] = tf(); m.dh[b] = tf(); }
        m.r = tf();
        const double rt = c->mp_rtol != 0.0 ? c->mp_rtol : 1e-5;
        m.tol2 = rt * rt;
    }
    ctx->stage = take(5 * (size_t)grid->nx * grid->ny * grid->nz);
    {
        Lev l;
        l.G = ctx->G;
        l.c = take(E); l.d = take(E); l.ax = take(E); l.ay = take(E); l.az = take(E);
        l.r = take(E); l.wd = take(E);
        ctx->L.push_back(l);
    }
    auto takef = [&](size_t n) -> float * {
        // FP32 arrays: half as many doubles, rounded up
        return reinterpret_cast<float *>(take((n + 1) / 2));
    };
    const double hmin = std::min({ctx->G.dx, ctx->G.dy, ctx->G.dz});
    for (size_t lv = 0; lv < lg.size(); ++lv) {
        Lev32 m;
        m.G = lg[lv];
        m.fx = 0.125 * gea::coarse_scale(ctx->G.dx, hmin);
        m.fy = 0.125 * gea::coarse_scale(ctx->G.dy, hmin);
        m.fz = 0.125 * gea::coarse_scale(ctx->G.dz, hmin);
        const size_t e = elems(lg[lv]);
        m.c = takef(e); m.d = takef(e); m.ax = takef(e); m.ay = takef(e); m.az = takef(e);
        m.w = takef(e);
        m.e = lv ? takef(e) : nullptr;
        m.r = lv ? takef(e) : nullptr;
        m.e2 = lv ? takef(e) : nullptr;
        ctx->M.push_back(m);
    }
    {
        // the pressure solve's vectors, a value per pair of cells (P is even)
        auto half = [&](auto &v) {
            using R = std::remove_reference_t<decltype(*v.p)>;
            const size_t n = E / 2, d = (n * sizeof(R) + sizeof(double) - 1) / sizeof(double);
            for (R **x : {&v.p, &v.w, &v.q, &v.rb, &v.xb}) *x = reinterpret_cast<R *>(take(d));
            v.ef = takef(n);
            v.z = ctx->M.size() > 1 ? takef(n) : v.ef;
        };
        if (ctx->mixed) half(ctx->rbf);
        else half(ctx->rb);
    }
    {
        const size_t nb = nblocks(ctx->G), ng = (nb + kGroup - 1) / kGroup;
        if (ng > 2 * (size_t)kCntSlots) {
            gea3d_destroy(ctx);
            return GEA_ERR_INVAL;
        }
        ctx->part = take(kCntSlots + 3 * nb + 3 * ng + 64);
    }
    ctx->sc = reinterpret_cast<Sc *>(take((sizeof(Sc) + 7) / 8));
    if (!ok) {
        gea3d_destroy(ctx);
        return GEA_ERR_NOMEM;
    }
    if (cudaStreamCreateWithFlags(&ctx->cap, cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamCreateWithFlags(&ctx->cap2, cudaStreamNonBlocking) != cudaSuccess ||
        cudaDeviceSynchronize() != cudaSuccess) {
        gea3d_destroy(ctx);
        return GEA_ERR_CUDA;
    }
    *out = ctx;
    return GEA_OK;
}

int gea3d_set_stream(gea3d_ctx *ctx, void *stream)
{
    if (!ctx) return GEA_ERR_INVAL;
    ctx->stream = (cudaStream_t)stream;
    return GEA_OK;
}

int gea3d_set_conservative(gea3d_ctx *ctx, const double *rho, const double *rhou, const double *rhov,
                           const double *rhow, const double *rhoe, int32_t mem)
{
    if (!ctx || !rho || !rhou || !rhov || !rhow || !rhoe || (mem != GEA_MEM_HOST && mem != GEA_MEM_DEVICE))
        return GEA_ERR_INVAL;
    const Geo &G = ctx->G;
    const size_t n = (size_t)G.nx * G.ny * G.nz;
    // the old state is being replaced: until this call succeeds the context
    // holds none
    ctx->have_state = false;
    CK3(cudaMemsetAsync(ctx->sc, 0, sizeof(Sc), ctx->stream));
    const double *src[5] = {rho, rhou, rhov, rhow, rhoe};
    for (int f = 0; f < 5; ++f)
        CK3(cudaMemcpyAsync(ctx->stage + f * n, src[f], n * sizeof(double), cudaMemcpyDefault, ctx->stream));
    k_derive<<<grid_of(G), kBlk, 0, ctx->stream>>>(G, ctx->F, ctx->stage, ctx->stage + n, ctx->stage + 2 * n,
                                                   ctx->stage + 3 * n, ctx->stage + 4 * n, ctx->gz, ctx->S[0], ctx->sc);
    CK3(cudaGetLastError());
    Sc h;
    CK3(cudaMemcpyAsync(&h, ctx->sc, sizeof(Sc), cudaMemcpyDeviceToHost, ctx->stream));
    CK3(cudaStreamSynchronize(ctx->stream));
    if (h.bad_cells) {
        ctx->have_state = false;
        return fail3(ctx, GEA_ERR_INVAL, "%d cells with rho <= 0 or T <= 0", h.bad_cells);
    }
    ctx->steps_at_sync = 0;
    ctx->have_state = true;
    return GEA_OK;
}

int gea3d_step_async(gea3d_ctx *ctx, int32_t n)
{
    if (!ctx || n < 0) return GEA_ERR_INVAL;
    if (!ctx->have_state) return fail3(ctx, GEA_ERR_STATE, "no state set");
    for (int f = 0; f < 2; ++f)
        if (!ctx->exec[f]) {
            const int rc = build3(ctx, f);
            if (rc) return rc;
        }
    for (int s = 0; s < n; ++s) {
        CK3(cudaGraphLaunch(ctx->exec[ctx->steps_at_sync & 1], ctx->stream));
        ctx->steps_at_sync += 1;
    }
    return GEA_OK;
}

int gea3d_sync(gea3d_ctx *ctx)
{
    if (!ctx) return GEA_ERR_INVAL;
    Sc h;
    CK3(cudaMemcpyAsync(&h, ctx->sc, sizeof(Sc), cudaMemcpyDeviceToHost, ctx->stream));
    CK3(cudaStreamSynchronize(ctx->stream));
    ctx->steps_at_sync = h.steps_done;
    if (h.last_status == GEA_ERR_NOCONV) return fail3(ctx, GEA_ERR_NOCONV, "a linear solve reached its iteration cap");
    if (h.last_status) return fail3(ctx, h.last_status, "device status %d", h.last_status);
    return GEA_OK;
}

int gea3d_step(gea3d_ctx *ctx, int32_t n)
{
    const int rc = gea3d_step_async(ctx, n);
    return rc ? rc : gea3d_sync(ctx);
}

int gea3d_get_state(gea3d_ctx *ctx, double *rho, double *u, double *v, double *w, double *T, double *p,
                    double *pp, int32_t mem)
{
    if (!ctx || (mem != GEA_MEM_HOST && mem != GEA_MEM_DEVICE)) return GEA_ERR_INVAL;
    if (!ctx->have_state) return fail3(ctx, GEA_ERR_STATE, "no state set");
    Sc h;
    CK3(cudaMemcpyAsync(&h, ctx->sc, sizeof(Sc), cudaMemcpyDeviceToHost, ctx->stream));
    CK3(cudaStreamSynchronize(ctx->stream));
    const St &S = ctx->S[h.steps_done & 1];
    const Geo &G = ctx->G;
    double *dst[7] = {rho, u, v, w, T, p, pp};
    const double *src[7] = {S.rho, S.u, S.v, S.w, S.T, S.p, S.pp};
    for (int f = 0; f < 7; ++f) {
        if (!dst[f]) continue;
        // (k (ny+1) + j) P + i -> (k ny + j) nx + i: one 3D copy per field (rows
        // of nx values, ny rows a layer out of the source's ny + 1, nz layers)
        cudaMemcpy3DParms c = {};
        c.srcPtr = make_cudaPitchedPtr(const_cast<double *>(src[f]), (size_t)G.P * sizeof(double),
                                       (size_t)G.nx * sizeof(double), (size_t)G.ny + 1);
        c.dstPtr = make_cudaPitchedPtr(dst[f], (size_t)G.nx * sizeof(double), (size_t)G.nx * sizeof(double),
                                       (size_t)G.ny);
        c.extent = make_cudaExtent((size_t)G.nx * sizeof(double), (size_t)G.ny, (size_t)G.nz);
        c.kind = cudaMemcpyDefault;
        CK3(cudaMemcpy3DAsync(&c, ctx->stream));
    }
    CK3(cudaStreamSynchronize(ctx->stream));
    return GEA_OK;
}

int gea3d_get_diag(gea3d_ctx *ctx, const double *theta_bar, double *theta_prime, double *mass, double *energy)
{
    if (!ctx) return GEA_ERR_INVAL;
    if (!ctx->have_state) return fail3(ctx, GEA_ERR_STATE, "no state set");
    if (theta_prime && !theta_bar) return fail3(ctx, GEA_ERR_INVAL, "theta_prime needs theta_bar");
    Sc h;
    CK3(cudaMemcpyAsync(&h, ctx->sc, sizeof(Sc), cudaMemcpyDeviceToHost, ctx->stream));
    CK3(cudaStreamSynchronize(ctx->stream));
    const St &S = ctx->S[h.steps_done & 1];
    const Geo &G = ctx->G;
    const size_t cells = (size_t)G.nx * G.ny * G.nz;
    // the staging area (5 dense fields) holds theta_bar, then theta'
    double *thb = ctx->stage, *tho = ctx->stage + cells;
    if (theta_bar) CK3(cudaMemcpyAsync(thb, theta_bar, G.nz * sizeof(double), cudaMemcpyDefault, ctx->stream));
    k_diag3<<<grid_of(G), kBlk, 0, ctx->stream>>>(G, ctx->F, ctx->C.p0, S, thb, ctx->gz,
                                                  theta_prime ? tho : nullptr, ctx->sc, ctx->part);
    CK3(cudaGetLastError());
    if (theta_prime)
        CK3(cudaMemcpyAsync(theta_prime, tho, cells * sizeof(double), cudaMemcpyDefault, ctx->stream));
    CK3(cudaMemcpyAsync(&h, ctx->sc, sizeof(Sc), cudaMemcpyDeviceToHost, ctx->stream));
    CK3(cudaStreamSynchronize(ctx->stream));
    if (mass) *mass = h.mass;
    if (energy) *energy = h.energy;
    return GEA_OK;
}

int gea3d_get_stats(gea3d_ctx *ctx, gea_stats *s)
{
    if (!ctx || !s) return GEA_ERR_INVAL;
    Sc h;
    CK3(cudaMemcpyAsync(&h, ctx->sc, sizeof(Sc), cudaMemcpyDeviceToHost, ctx->stream));
    CK3(cudaStreamSynchronize(ctx->stream));
    memset(s, 0, sizeof(*s));
    s->steps_done = h.steps_done;
    s->jac_u = h.last_sweeps[0];
    s->jac_h = h.last_sweeps[1];
    for (int c = 0; c < 4; ++c) { s->cg_iters[c] = h.last_cg_iters[c]; s->cg_relres[c] = h.last_cg_relres[c]; }
    s->status = h.last_status;
    s->mg_levels = (int)ctx->M.size();
    s->launches = h.launches;
    s->driver = ctx->mixed ? 2 : 0;
    return GEA_OK;
}

int gea3d_profile_step(gea3d_ctx *ctx, gea_kernel_time *out, int32_t max_entries, int32_t *n_entries)
{
    if (!ctx || max_entries < 0 || (!out && max_entries > 0) || !n_entries) return GEA_ERR_INVAL;
    if (!ctx->have_state) return fail3(ctx, GEA_ERR_STATE, "no state set");
    Sc h;
    CK3(cudaMemcpyAsync(&h, ctx->sc, sizeof(Sc), cudaMemcpyDeviceToHost, ctx->stream));
    CK3(cudaStreamSynchronize(ctx->stream));
    if (h.status) return fail3(ctx, h.status, "device status %d", h.status);
    {
        Trace3 tr;
        tr.dsc = ctx->sc;
        const int rc = record3(ctx, (int)(h.steps_done & 1), ctx->stream, false, &tr);
        if (rc) return rc;
        CK3(cudaStreamSynchronize(ctx->stream));
        std::vector<gea_kernel_time> agg;
        for (auto &r : tr.recs) {
            float ms = 0.f;
            CK3(cudaEventElapsedTime(&ms, r.e0, r.e1));
            size_t j = 0;
            while (j < agg.size() && strcmp(agg[j].name, r.name)) ++j;
            if (j == agg.size()) {
                gea_kernel_time k;
                memset(&k, 0, sizeof(k));
                snprintf(k.name, sizeof(k.name), "%s", r.name);
                agg.push_back(k);
            }
            agg[j].launches += 1;
            agg[j].cells += r.cells;
            agg[j].ms += ms;
        }
        *n_entries = (int32_t)agg.size();
        for (size_t j = 0; j < agg.size() && (int32_t)j < max_entries; ++j) out[j] = agg[j];
    }
    return gea3d_sync(ctx);
}

const char *gea3d_last_error(const gea3d_ctx *ctx) { return ctx ? ctx->err : "null context"; }

void gea3d_destroy(gea3d_ctx *ctx)
{
    if (!ctx) return;
    if (ctx->stream) cudaStreamSynchronize(ctx->stream);
    else cudaDeviceSynchronize();
    for (int f = 0; f < 2; ++f) {
        if (ctx->exec[f]) cudaGraphExecDestroy(ctx->exec[f]);
        if (ctx->graph[f]) cudaGraphDestroy(ctx->graph[f]);
    }
    if (ctx->cap) cudaStreamDestroy(ctx->cap);
    if (ctx->cap2) cudaStreamDestroy(ctx->cap2);
    for (void *p : ctx->allocs) cudaFree(p);
    delete ctx;
}

}  // extern "C"
