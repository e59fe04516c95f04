// gea_kernels.cu -- per-phase CUDA kernels (sm_103a, FP64) of one time step
// of the GEA pressure-based Euler solver (Girfoglio, Quaini & Rozza, arXiv
// 2303.10499, Section 3) and their host-side launchers: the graph path, one
// kernel per phase (the phase bodies are the tile functions of
// gea_tiles.cuh, one tile per block), with the solver loops as conditional
// WHILE nodes of a CUDA graph. The same kernels also serve the per-kernel
// profiled step. Reductions are deterministic: block partials, added in a
// fixed order by the last block to arrive. Kernels inside a device-side
// loop return early (uniformly across the grid) once the loop has converged
// or failed.
#include "gea_internal.cuh"
#include "gea_tiles.cuh"

#include <math.h>

namespace gea {

namespace {

using namespace tiles;

__device__ __forceinline__ bool loop_over(const Scal *sc, int which)
{
    return sc->status || sc->done[which];
}

// From rows of `pitch` values (the staging area's pitch, or nx: a caller's
// dense device arrays, read in place).
__global__ void k_derive(Geom G, Phys F, const double *__restrict__ rho,
                         const double *__restrict__ rhou, const double *__restrict__ rhow,
                         const double *__restrict__ rhoe, int pitch, const double *__restrict__ gzc, State S, Scal *sc)
{
    int i, k;
    if (!cell_of(G, blockIdx.x, blockIdx.y, i, k)) return;
    const int q = cidx(G, i, k);
    const size_t d = (size_t)k * pitch + i;
    const double gz = gzc[k];
    const double r = rho[d], ir = recip(r);
    const double ru = rhou[d], rw = rhow[d], re = rhoe[d];
    const double u = ru * ir, w = rw * ir;
    const double K = 0.5 * fma(u, u, w * w);
    // e = re / r rounded as a division would: T and with it p = rho R T carry the
    // hydrostatic balance
    const double e0 = re * ir, e = fma(fma(-r, e0, re), ir, e0);
    const double T = ((e - K) - gz) * F.icv;
    if (!(r > 0.0) || !(T > 0.0)) atomicAdd(&sc->bad_cells, 1);
    S.rho[q] = r;
    S.u[q] = u;
    S.w[q] = w;
    S.T[q] = T;
    S.h[q] = F.cp * T;
    const double p = r * F.R * T;
    S.p[q] = p;
    S.pp[q] = fma(r, gz, p);
    S.pold[q] = p;
    S.Kold[q] = K;   // K^{-1} := K^0
    S.phix[k * G.P + i] = i > 0 ? F.hdz * (rhou[d - 1] + ru) : 0.0;
    if (i == G.nx - 1) S.phix[k * G.P + G.nx] = 0.0;
    S.phiz[k * G.P + i] = k > 0 ? F.hdx * (rhow[d - pitch] + rw) : 0.0;
    if (k == G.nz - 1) S.phiz[G.nz * G.P + i] = 0.0;
}

// Conservative variables of a state (Section 2.1), the inverse of k_derive:
// rho, rho u, rho w and rho e with the total energy e = cv T + |u|^2/2 + g z.
// The state is slot (base + steps done) & 1. Into rows of `pitch` values;
// null arrays are left out.
__global__ void k_conserve(Geom G, Phys F, State S0, State S1, int base, const Scal *sc, double *__restrict__ rho,
                           double *__restrict__ rhou, double *__restrict__ rhow, double *__restrict__ rhoe, int pitch)
{
    int i, k;
    if (!cell_of(G, blockIdx.x, blockIdx.y, i, k)) return;
    const State &S = ((base + sc->steps_done) & 1) ? S1 : S0;
    const int q = cidx(G, i, k);
    const size_t d = (size_t)k * pitch + i;
    const double z = (k + 0.5) * G.dz;
    const double r = S.rho[q], u = S.u[q], w = S.w[q];
    const double K = 0.5 * (u * u + w * w);
    if (rho) rho[d] = r;
    if (rhou) rhou[d] = r * u;
    if (rhow) rhow[d] = r * w;
    if (rhoe) rhoe[d] = r * ((F.cp - F.R) * S.T[q] + K + F.g * z);
}

// A caller's dense device arrays to or from a state's pitched ones, all
// fields in one pass: one launch instead of a copy per field, which at 160 x 80
// cost as much as half a step. Cell fields are nz rows of nx values, x-face
// fluxes nz of nx + 1, z-face fluxes nz + 1 of nx. Null arrays are left out.
__device__ __forceinline__ void field_rows(const Geom &G, int f, int &cols, int &rows)
{
    cols = f == FIELD_PHIX ? G.nx + 1 : G.nx;
    rows = f == FIELD_PHIZ ? G.nz + 1 : G.nz;
}

__global__ void k_fields_in(Geom G, FieldPtrs dst, DenseFields src)
{
    const int i = blockIdx.x * BX + threadIdx.x, k = blockIdx.y * BZ + threadIdx.y;
#pragma unroll
    for (int f = 0; f < NFIELDS; ++f) {
        int cols, rows;
        field_rows(G, f, cols, rows);
        if (src.p[f] && i < cols && k < rows) dst.p[f][k * G.P + i] = src.p[f][(size_t)k * cols + i];
    }
}

// out of the state in slot (base + steps done) & 1
__global__ void k_fields_out(Geom G, FieldPtrs s0, FieldPtrs s1, int base, const Scal *sc, DenseFields dst)
{
    const int i = blockIdx.x * BX + threadIdx.x, k = blockIdx.y * BZ + threadIdx.y;
    const FieldPtrs &src = ((base + sc->steps_done) & 1) ? s1 : s0;
#pragma unroll
    for (int f = 0; f < NFIELDS; ++f) {
        int cols, rows;
        field_rows(G, f, cols, rows);
        if (dst.p[f] && i < cols && k < rows) dst.p[f][(size_t)k * cols + i] = src.p[f][k * G.P + i];
    }
}

// ---- Step 1 ----

__global__ void k_les(StepArgs a)
{
    if (a.sc->status) return;
    __shared__ double sm[2 * kT1];
    ph_les(a, sm, blockIdx.x, blockIdx.y);
}

__global__ void k_pred_setup(StepArgs a)
{
    if (a.sc->status) return;
    __shared__ double red[2 * NTHREADS];
    double acc[2] = {0.0, 0.0}, tot[2];
    ph_pred(a, blockIdx.x, blockIdx.y, acc);
    if (grid_sum<2>(acc, red, a.partials, &a.sc->counters[CNT_PRED], tot)) fin_pred(a.sc, tot);
}

// Sweeps run in pairs (X_a -> X_b -> X_a) so that the loop ends in X_a. The
// second sweep of a pair whose first sweep met the tolerance copies X_b back
// instead: the iteration stops after that sweep.
__global__ void k_mom_jacobi(StepArgs a, const double *uin, const double *win, double *uout,
                             double *wout, int second)
{
    if (a.sc->status) return;
    if (second && a.sc->done[LOOP_MOM]) {
        block_tiles(a.G, [&](int bx, int bz) {
            ph_copy(a.G, uin, uout, bx, bz);
            ph_copy(a.G, win, wout, bx, bz);
        });
        return;
    }
    __shared__ double sm[2 * kT2];
    __shared__ double red[2 * NTHREADS];
    double acc[2] = {0.0, 0.0}, tot[2];
    block_tiles(a.G, [&](int bx, int bz) { ph_mom(a, uin, win, uout, wout, sm, bx, bz, acc); });
    if (grid_sum<2>(acc, red, a.partials, &a.sc->counters[CNT_MOM], tot)) fin_mom(a.sc, tot, a.jac_rtol2);
}

// ---- Step 2 ----

__global__ void k_enth_rhs(StepArgs a)
{
    if (a.sc->status) return;
    __shared__ double sm[2 * kT2];
    __shared__ double red[NTHREADS];
    double acc[1] = {0.0}, tot[1];
    ph_enth_rhs(a, a.ua, a.wa, a.ha, sm, blockIdx.x, blockIdx.y, acc);
    if (grid_sum<1>(acc, red, a.partials, &a.sc->counters[CNT_ENTH_RHS], tot)) fin_enth_rhs(a.sc, tot);
}

__global__ void k_enth_jacobi(StepArgs a, const double *hin, double *hout, int second)
{
    if (a.sc->status) return;
    if (second && a.sc->done[LOOP_ENTH]) {
        block_tiles(a.G, [&](int bx, int bz) { ph_copy(a.G, hin, hout, bx, bz); });
        return;
    }
    __shared__ double sm[kT2];
    __shared__ double red[NTHREADS];
    double acc[1] = {0.0}, tot[1];
    block_tiles(a.G, [&](int bx, int bz) { ph_enth(a, hin, hout, sm, bx, bz, acc); });
    if (grid_sum<1>(acc, red, a.partials, &a.sc->counters[CNT_ENTH], tot)) fin_enth(a.sc, tot, a.jac_rtol2);
}

__global__ void k_eos_coef(StepArgs a, Level L)
{
    if (a.sc->status) return;
    __shared__ double sm[2 * kT1 + kFaces];
    ph_eos(a, L, a.ha, sm, blockIdx.x, blockIdx.y);
}

template <class R>
__global__ void k_mg_coarsen(LevelT<R> f, LevelT<R> c, double cfx, double cfz)
{
    ph_coarsen<R>(f, c, cfx, cfz, blockIdx.x, blockIdx.y);
}

// ---- Step 3 ----

__global__ void k_H(StepArgs a, const double *U, const double *W)
{
    if (a.sc->status) return;
    __shared__ double sm[2 * kT2];
    ph_H(a, U, W, sm, blockIdx.x, blockIdx.y);
}

__global__ void k_helm_rhs(StepArgs a, Level L, const double *xin, double *xout, int corr)
{
    if (a.sc->status) return;
    __shared__ double sm[4 * kT1];
    __shared__ double red[2 * NTHREADS];
    double acc[2] = {0.0, 0.0}, tot[2];
    ph_helm_rhs(a, L, xin, xout, sm, blockIdx.x, blockIdx.y, acc);
    if (grid_sum<2>(acc, red, a.partials, &a.sc->counters[CNT_HELM], tot))
        fin_helm(a.sc, tot, a.cg_rtol2, corr);
}

// ---- the pressure solve (R: double, or float for the mixed-precision step) ----

template <class R>
__global__ void k_rb_start(LevelT<R> L, Scal *sc, double *partials)
{
    if (loop_over(sc, LOOP_CG)) return;
    __shared__ R sm[kPH1];
    __shared__ double red[NTHREADS];
    R acc[1] = {(R)0};
    double tot[1];
    block_tiles(L.G, [&](int bx, int bz) {
        ph_rb_start<R>(L, black_res(L, 0), L.e2, reinterpret_cast<double *>(sm), bx, bz, acc);
    });
    if (grid_sum<1, R>(acc, red, partials, &sc->counters[CNT_RZ], tot)) fin_rz(sc, tot);
}

template <bool FINE, class R>
__global__ void k_mg_down(LevelT<R> f, LevelT<R> c, Phys F, Scal *sc)
{
    if (loop_over(sc, LOOP_CG)) return;
    __shared__ R sm[kPH2 + kPH1 + BZ * BX];
    ph_mg_down<FINE, R>(f, c, FINE ? black_res(f, 0) : nullptr, F, reinterpret_cast<double *>(sm), blockIdx.x,
                        blockIdx.y);
}

// FINEST: also r.z
template <bool FINEST, class R>
__global__ void k_mg_up(LevelT<R> f, const R *ec, int Pc, Phys F, Scal *sc, double *partials)
{
    if (loop_over(sc, LOOP_CG)) return;
    __shared__ R sm[kPH2 + kPH1];
    __shared__ double red[NTHREADS];
    R acc[1] = {(R)0};
    double tot[1];
    block_tiles(f.G, [&](int bx, int bz) {
        ph_mg_up<FINEST, R>(f, f.r, ec, Pc, f.e2, F, reinterpret_cast<double *>(sm), bx, bz, acc);
    });
    if (!FINEST) return;
    if (grid_sum<1, R>(acc, red, partials, &sc->counters[CNT_RZ], tot)) fin_rz(sc, tot);
}

template <class R>
__global__ void k_rb_up(LevelT<R> f, const R *ec, int Pc, Phys F, Scal *sc, double *partials)
{
    if (loop_over(sc, LOOP_CG)) return;
    __shared__ double red[NTHREADS];
    R acc[1] = {(R)0};
    double tot[1];
    const R *rb = black_res(f, sc->cg_it);
    block_tiles(f.G, [&](int bx, int bz) { ph_rb_up<R>(f, rb, ec, Pc, f.e2, F, bx, bz, acc); });
    if (grid_sum<1, R>(acc, red, partials, &sc->counters[CNT_RZ], tot)) fin_rz(sc, tot);
}

// The directions alternate between p0 and p1 by iteration parity: iteration
// it reads p[it & 1] and writes p[(it + 1) & 1].
template <class R>
__global__ void k_cg_pspmv(LevelT<R> L, CgVecT<R> v, Scal *sc, double *partials)
{
    if (loop_over(sc, LOOP_CG)) return;
    __shared__ R sm[kPH2 + kPH1];
    __shared__ double red[NTHREADS];
    const int it = sc->cg_it;
    const R *pold = (it & 1) ? v.p1 : v.p0;
    R *pnew = (it & 1) ? v.p0 : v.p1;
    const double beta = sc->beta;
    R acc[1] = {(R)0};
    double tot[1];
    block_tiles(L.G, [&](int bx, int bz) {
        ph_pspmv<R>(L, L.e2, pold, pnew, v.q, beta, it == 0, reinterpret_cast<double *>(sm), bx, bz, acc);
    });
    if (grid_sum<1, R>(acc, red, partials, &sc->counters[CNT_PQ], tot)) fin_pq(sc, tot);
}

template <class R>
__global__ void k_cg_update_single(LevelT<R> L, CgVecT<R> v, Scal *sc, double *partials, double tol2)
{
    if (loop_over(sc, LOOP_CG)) return;
    __shared__ double red[2 * NTHREADS];
    const int it = sc->cg_it;
    const R *p = (it & 1) ? v.p0 : v.p1;
    const double alpha = sc->alpha;
    R acc[2] = {(R)0, (R)0};
    double tot[2];
    block_tiles(L.G, [&](int bx, int bz) {
        ph_update_single<R>(L, v.q, black_res(L, 0), L.e2, v.x, p, alpha, it == 0, bx, bz, acc);
    });
    if (grid_sum<2, R>(acc, red, partials, &sc->counters[CNT_UPD], tot)) {
        const double t0[1] = {tot[0]}, t1[1] = {tot[1]};
        fin_update(sc, t0, tol2);
        fin_rz(sc, t1);
    }
}

template <class R>
__global__ void k_cg_update_down(LevelT<R> f, LevelT<R> c, CgVecT<R> v, Phys F, Scal *sc, double *partials, double tol2)
{
    if (loop_over(sc, LOOP_CG)) return;
    __shared__ R sm[kPH1 + BZ * BX];
    __shared__ double red[NTHREADS];
    const int it = sc->cg_it;
    const R *p = (it & 1) ? v.p0 : v.p1;
    const double alpha = sc->alpha;
    R acc[1] = {(R)0};
    double tot[1];
    block_tiles(f.G, [&](int bx, int bz) {
        ph_update_down<R>(f, c, v.q, black_res(f, it), black_res(f, it + 1), v.x, p, alpha, it == 0, F,
                          reinterpret_cast<double *>(sm), bx, bz, acc);
    });
    if (grid_sum<1, R>(acc, red, partials, &sc->counters[CNT_UPD], tot)) fin_update(sc, tot, tol2);
}

template <class R>
__global__ void k_correct(StepArgs a, LevelT<R> L, SolveT<R> v, double *ppout)
{
    if (a.sc->status) return;
    __shared__ double sm[kCorrectSmem];
    ph_correct<R>(a, L, v, v.xb && a.sc->cg_it > 0, ppout, sm, blockIdx.x, blockIdx.y);
}

// ---- loop control and step bookkeeping (one thread) ----

__global__ void k_loop_ctl(Scal *sc, cudaGraphConditionalHandle h, int graph, int which,
                           int maxtrips, int body_launches)
{
    const int trips = ++sc->trips[which];
    const int done = sc->done[which];
    sc->launches += body_launches;
    if (!done && !sc->status && trips >= maxtrips) sc->status = GEA_ERR_NOCONV;
    if (graph) cudaGraphSetConditional(h, (done || sc->status || trips >= maxtrips) ? 0u : 1u);
}

// Before a gated loop: run it only while it is not finished.
__global__ void k_loop_gate(Scal *sc, cudaGraphConditionalHandle h, int which)
{
    cudaGraphSetConditional(h, (sc->done[which] || sc->status) ? 0u : 1u);
}

__global__ void k_step_begin(Scal *sc)
{
    sc->u1_slot = sc->h1_slot = 0;
    for (int c = 0; c < 4; ++c) { sc->cg_iters[c] = 0; sc->cg_b2[c] = 0.0; }
    sc->sweeps[0] = sc->sweeps[1] = 0;
}

__global__ void k_step_end(Scal *sc, int fixed_launches)
{
    sc->launches += fixed_launches;
    if (sc->status) {
        sc->last_status = sc->status;
        return;
    }
    sc->steps_done += 1;
    sc->last_sweeps[0] = sc->sweeps[0];
    sc->last_sweeps[1] = sc->sweeps[1];
    for (int c = 0; c < 4; ++c) {
        sc->last_cg_iters[c] = sc->cg_iters[c];
        sc->last_cg_relres[c] = cg_relres(*sc, c);
    }
    sc->last_status = 0;
}

// ---- diagnostics (Remark 2) ----

__global__ void k_diag(Geom G, Phys F, State S, const double *__restrict__ thbar,
                       double *__restrict__ th, Scal *sc, double *partials)
{
    __shared__ double red[2 * NTHREADS];
    int i, k;
    const bool in = cell_of(G, blockIdx.x, blockIdx.y, i, k);
    double v[2] = {0.0, 0.0};
    if (in) {
        const int q = cidx(G, i, k);
        const double z = (k + 0.5) * G.dz;
        if (th) th[q] = S.T[q] / pow(S.p[q] / F.p0, F.R / F.cp) - thbar[k];
        const double V = G.dx * G.dz;
        const double K = 0.5 * (S.u[q] * S.u[q] + S.w[q] * S.w[q]);
        v[0] = S.rho[q] * V;
        v[1] = S.rho[q] * ((F.cp - F.R) * S.T[q] + K + F.g * z) * V;
    }
    double tot[2];
    if (grid_sum<2>(v, red, partials, &sc->counters[CNT_DIAG], tot)) {
        sc->mass = tot[0];
        sc->energy = tot[1];
    }
}

inline dim3 grid_of(const Geom &G) { return dim3((G.nx + BX - 1) / BX, (G.nz + BZ - 1) / BZ); }
inline dim3 grid_pairs(const Geom &G) { return grid_pair_tiles(G, 1); }
const dim3 kBlock(BX, BZ);

}  // namespace

int max_blocks(const Geom &G)
{
    dim3 g = grid_of(G);
    return (int)(g.x * g.y);
}

void launch_derive(const Geom &G, const Phys &F, const double *rho, const double *rhou,
                   const double *rhow, const double *rhoe, int pitch, const double *gzc, const State &S, Scal *sc,
                   cudaStream_t st)
{
    k_derive<<<grid_of(G), kBlock, 0, st>>>(G, F, rho, rhou, rhow, rhoe, pitch, gzc, S, sc);
}

void launch_conserve(const Geom &G, const Phys &F, const State S[2], int base, const Scal *sc, double *rho,
                     double *rhou, double *rhow, double *rhoe, int pitch, cudaStream_t st)
{
    k_conserve<<<grid_of(G), kBlock, 0, st>>>(G, F, S[0], S[1], base, sc, rho, rhou, rhow, rhoe, pitch);
}

// covers the extra column of the x-faces and the extra row of the z-faces
inline dim3 grid_faces(const Geom &G) { return dim3(G.nx / BX + 1, G.nz / BZ + 1); }

void launch_fields_in(const Geom &G, const State &S, const DenseFields &src, cudaStream_t st)
{
    k_fields_in<<<grid_faces(G), kBlock, 0, st>>>(G, state_fields(S), src);
}

void launch_fields_out(const Geom &G, const State S[2], int base, const Scal *sc, const DenseFields &dst,
                       cudaStream_t st)
{
    k_fields_out<<<grid_faces(G), kBlock, 0, st>>>(G, state_fields(S[0]), state_fields(S[1]), base, sc, dst);
}

// Launch with an optional trace bracket.
#define TRACED(tr, name, cells, launch)                         \
    do {                                                        \
        if (tr) (tr)->begin(name, (long long)(cells), st);      \
        launch;                                                 \
        if (tr) (tr)->end(st);                                  \
    } while (0)

inline long long ncell(const Geom &G) { return (long long)G.nx * G.nz; }

void launch_les(const StepArgs &a, cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "les", ncell(a.G), (k_les<<<grid_of(a.G), kBlock, 0, st>>>(a)));
}

void launch_pred_setup(const StepArgs &a, cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "pred_setup", ncell(a.G), (k_pred_setup<<<grid_of(a.G), kBlock, 0, st>>>(a)));
}

void launch_mom_jacobi(const StepArgs &a, const double *uin, const double *win, double *uout,
                       double *wout, int second, cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "mom_jacobi", ncell(a.G),
           (k_mom_jacobi<<<grid_tiles(a.G, a.tiles_per_block), kBlock, 0, st>>>(a, uin, win, uout, wout, second)));
}

void launch_enth_rhs(const StepArgs &a, cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "enth_rhs", ncell(a.G), (k_enth_rhs<<<grid_of(a.G), kBlock, 0, st>>>(a)));
}

void launch_enth_jacobi(const StepArgs &a, const double *hin, double *hout, int second,
                        cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "enth_jacobi", ncell(a.G),
           (k_enth_jacobi<<<grid_tiles(a.G, a.tiles_per_block), kBlock, 0, st>>>(a, hin, hout, second)));
}

void launch_eos_coef(const StepArgs &a, const Level &L0, cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "eos_coef", ncell(a.G), (k_eos_coef<<<grid_of(a.G), kBlock, 0, st>>>(a, L0)));
}

// launch names: the FP32 kernels of the mixed-precision step carry "mx_"
template <class R>
const char *name_of(const char *f64, const char *f32)
{
    return sizeof(R) == sizeof(double) ? f64 : f32;
}

template <class R>
void launch_mg_coarsen(const LevelT<R> &f, const LevelT<R> &c, double cfx, double cfz, cudaStream_t st,
                       Tracer *tr)
{
    TRACED(tr, name_of<R>("mg_coarsen", "mx_coarsen"), ncell(c.G),
           (k_mg_coarsen<R><<<grid_of(c.G), kBlock, 0, st>>>(f, c, cfx, cfz)));
}

void launch_H(const StepArgs &a, const double *U, const double *W, cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "H", ncell(a.G), (k_H<<<grid_of(a.G), kBlock, 0, st>>>(a, U, W)));
}

void launch_helm_rhs(const StepArgs &a, const Level &L0, const double *xin, double *xout,
                     int corr, cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "helm_rhs", ncell(a.G),
           (k_helm_rhs<<<grid_of(a.G), kBlock, 0, st>>>(a, L0, xin, xout, corr)));
}

namespace {

// V-cycle levels below the finest: down halves of levels 1 .. nlev-2, the
// coarsest sweep, up halves to level 1.
template <class R>
int vcycle_below(const StepArgs &a, const LevelT<R> *L, int nlev, cudaStream_t st, Tracer *tr)
{
    int n = 0;
    for (int l = 1; l + 1 < nlev; ++l, ++n)
        TRACED(tr, name_of<R>("mg_down", "mx_mg_down"), ncell(L[l].G),
               (k_mg_down<false, R><<<grid_pairs(L[l].G), kBlock, 0, st>>>(L[l], L[l + 1], a.F, a.sc)));
    for (int l = nlev - 1; l >= 1; --l, ++n) {
        const bool last = l == nlev - 1;
        const R *ec = last ? nullptr : L[l + 1].e2;
        TRACED(tr, last ? name_of<R>("mg_coarse", "mx_mg_coarse") : name_of<R>("mg_up", "mx_mg_up"), ncell(L[l].G),
               (k_mg_up<false, R><<<grid_pairs(L[l].G), kBlock, 0, st>>>(L[l], ec, last ? 0 : L[l + 1].G.P, a.F, a.sc,
                                                                         a.partials)));
    }
    return n;
}

// the finest level's up half of the red-black iteration
template <class R>
void rb_up(const StepArgs &a, const LevelT<R> *L, cudaStream_t st, Tracer *tr)
{
    TRACED(tr, name_of<R>("rb_up", "mx_rb_up"), ncell(L[0].G),
           (k_rb_up<R><<<grid_pair_tiles(L[0].G, a.tiles_per_block), kBlock, 0, st>>>(L[0], L[1].e2, L[1].G.P, a.F,
                                                                                      a.sc, a.partials)));
}

}  // namespace

template <class R>
int launch_vcycle(const StepArgs &a, const LevelT<R> *L, int nlev, cudaStream_t st, Tracer *tr)
{
    int n = 0;
    if (nlev > 1) {
        TRACED(tr, name_of<R>("mg_down", "mx_mg_down"), ncell(L[0].G),
               (k_mg_down<false, R><<<grid_pairs(L[0].G), kBlock, 0, st>>>(L[0], L[1], a.F, a.sc)));
        n = 1 + vcycle_below<R>(a, L, nlev, st, tr);
    }
    const R *ec = nlev > 1 ? L[1].e2 : nullptr;
    TRACED(tr, name_of<R>("mg_up", "mx_mg_up"), ncell(L[0].G),
           (k_mg_up<true, R><<<grid_pair_tiles(L[0].G, a.tiles_per_block), kBlock, 0, st>>>(
               L[0], ec, nlev > 1 ? L[1].G.P : 0, a.F, a.sc, a.partials)));
    return n + 1;
}

template <class R>
int launch_cg_start(const StepArgs &a, const LevelT<R> *L, int nlev, cudaStream_t st, Tracer *tr)
{
    if (nlev == 1) {
        TRACED(tr, name_of<R>("rb_start", "mx_rb_start"), ncell(a.G),
               (k_rb_start<R><<<grid_pair_tiles(a.G, a.tiles_per_block), kBlock, 0, st>>>(L[0], a.sc, a.partials)));
        return 1;
    }
    TRACED(tr, name_of<R>("mg_down", "mx_mg_down"), ncell(a.G),
           (k_mg_down<true, R><<<grid_pairs(a.G), kBlock, 0, st>>>(L[0], L[1], a.F, a.sc)));
    const int n = vcycle_below<R>(a, L, nlev, st, tr);
    rb_up<R>(a, L, st, tr);
    return n + 2;
}

template <class R>
int launch_cg_iter(const StepArgs &a, const LevelT<R> *L, int nlev, const CgVecT<R> &v, double tol2, cudaStream_t st,
                   Tracer *tr)
{
    const dim3 grid = grid_pair_tiles(a.G, a.tiles_per_block);
    TRACED(tr, name_of<R>("cg_pspmv", "mx_pspmv"), ncell(a.G),
           (k_cg_pspmv<R><<<grid, kBlock, 0, st>>>(L[0], v, a.sc, a.partials)));
    if (nlev == 1) {
        TRACED(tr, name_of<R>("cg_update_single", "mx_update_single"), ncell(a.G),
               (k_cg_update_single<R><<<grid, kBlock, 0, st>>>(L[0], v, a.sc, a.partials, tol2)));
        return 2;
    }
    TRACED(tr, name_of<R>("cg_update_down", "mx_update_down"), ncell(a.G),
           (k_cg_update_down<R><<<grid, kBlock, 0, st>>>(L[0], L[1], v, a.F, a.sc, a.partials, tol2)));
    const int n = vcycle_below<R>(a, L, nlev, st, tr);
    rb_up<R>(a, L, st, tr);
    return n + 3;
}

template <class R>
void launch_correct(const StepArgs &a, const LevelT<R> &L, const SolveT<R> &v, double *ppout, cudaStream_t st,
                    Tracer *tr)
{
    TRACED(tr, "correct", ncell(a.G), (k_correct<R><<<grid_of(a.G), kBlock, 0, st>>>(a, L, v, ppout)));
}

#define INSTANTIATE(R)                                                                                              \
    template void launch_mg_coarsen<R>(const LevelT<R> &, const LevelT<R> &, double, double, cudaStream_t,          \
                                       Tracer *);                                                                   \
    template int launch_vcycle<R>(const StepArgs &, const LevelT<R> *, int, cudaStream_t, Tracer *);                \
    template int launch_cg_start<R>(const StepArgs &, const LevelT<R> *, int, cudaStream_t, Tracer *);              \
    template int launch_cg_iter<R>(const StepArgs &, const LevelT<R> *, int, const CgVecT<R> &, double,             \
                                   cudaStream_t, Tracer *);                                                         \
    template void launch_correct<R>(const StepArgs &, const LevelT<R> &, const SolveT<R> &, double *, cudaStream_t, \
                                    Tracer *);
INSTANTIATE(double)
INSTANTIATE(float)
#undef INSTANTIATE

namespace {

// graph = 1: block (0,0) also sets the IF condition of the network pass
// (run it only while the solve is not finished)
template <class R>
__global__ void k_guess_in(Geom G, const R *r, float *dense, Scal *sc, cudaGraphConditionalHandle h, int graph,
                           int body_launches)
{
    const bool over = loop_over(sc, LOOP_CG);
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && threadIdx.y == 0) {
        if (graph) cudaGraphSetConditional(h, over ? 0u : 1u);
        if (!over) sc->launches += body_launches;
    }
    if (over) return;
    int i, k;
    if (!cell_of(G, blockIdx.x, blockIdx.y, i, k)) return;
    dense[(size_t)k * G.nx + i] = (float)r[cidx(G, i, k)];
}

template <class R>
__global__ void k_guess_dots(LevelT<R> L, const float *e, const R *r, R *q, Scal *sc, double *partials)
{
    if (loop_over(sc, LOOP_CG)) return;
    __shared__ double sm[kT1];
    __shared__ double red[2 * NTHREADS];
    R acc[2] = {(R)0, (R)0};
    double tot[2];
    ph_guess_dots<R>(L, e, r, q, sm, blockIdx.x, blockIdx.y, acc);
    if (grid_sum<2, R>(acc, red, partials, &sc->counters[CNT_GUESS], tot)) fin_guess_dots(sc, tot);
}

template <class R>
__global__ void k_guess_apply(LevelT<R> L, const float *e, const R *q, R *r, R *x, Scal *sc, double *partials,
                              double tol2)
{
    if (loop_over(sc, LOOP_CG)) return;
    __shared__ double red[NTHREADS];
    R acc[1] = {(R)0};
    double tot[1];
    ph_guess_apply<R>(L, e, q, r, x, sc->galpha, blockIdx.x, blockIdx.y, acc);
    if (grid_sum<1, R>(acc, red, partials, &sc->counters[CNT_GUESS], tot)) fin_guess_apply(sc, tot, tol2);
}

// ---- flexible CG with a two-stage preconditioner (attach mode 2) ----
//
// z = g e + M(r - g A e): the network's correction e = N(r) with the step g
// that minimises the A-norm error along it, then one multigrid V-cycle M on
// the residual it leaves. The network alone stagnates (it cannot represent
// the residual its own step leaves), the V-cycle keeps the linear part.
// The preconditioner is nonlinear, so the one-term recurrence is written in
// the form that stays a descent method for a changing preconditioner
// (flexible CG truncated to one previous direction): beta = -(z.q_old) /
// (p_old.q_old), p = z + beta p_old, alpha = r.p / p.A p.

// A e at cell (i, k) of a tile holding e (FP64, halo 1).
__device__ __forceinline__ double fcg_ae(const Level &L, int q, int i, int k, const Tile<1> &se, int y, int x)
{
    return helm_tile<1, double>(L, q, i, k, se, y, x);
}

// The network's correction e (FP32, dense) on the tile and its halo.
__device__ __forceinline__ void fcg_load_e(Tile<1> &se, const Geom &G, const float *e, int bx, int bz)
{
    load_tile_fn<1, double>(se, G, bx, bz, [&](int, int i, int k) { return (double)e[(size_t)k * G.nx + i]; });
}

// acc += (r.e, e.A e); g = r.e / e.A e (0 unless e.A e > 0).
__global__ void k_fcg_dots(Level L, const float *e, Scal *sc, double *partials)
{
    if (loop_over(sc, LOOP_CG)) return;
    __shared__ double sm[kT1];
    __shared__ double red[2 * NTHREADS];
    const Geom &G = L.G;
    const double *r = res_of(L, sc->cg_it);
    Tile<1> &se = tile_at<1>(sm, 0);
    fcg_load_e(se, G, e, blockIdx.x, blockIdx.y);
    __syncthreads();
    double acc[2] = {0.0, 0.0}, tot[2];
    int i, k;
    if (cell_of(G, blockIdx.x, blockIdx.y, i, k)) {
        const int q = cidx(G, i, k);
        const int y = threadIdx.y + 1, x = threadIdx.x + 1;
        const double ev = se[y][x];
        acc[0] = ld(&r[q]) * ev;
        acc[1] = ev * fcg_ae(L, q, i, k, se, y, x);
    }
    if (grid_sum<2>(acc, red, partials, &sc->counters[CNT_GUESS], tot))
        sc->galpha = (tot[1] > 0.0 && isfinite(tot[0]) && isfinite(tot[1])) ? tot[0] / tot[1] : 0.0;
}

// s = r - g A e, the V-cycle's input.
__global__ void k_fcg_rest(Level L, const float *e, double *s, Scal *sc)
{
    if (loop_over(sc, LOOP_CG)) return;
    __shared__ double sm[kT1];
    const Geom &G = L.G;
    const double *r = res_of(L, sc->cg_it);
    const double g = sc->galpha;
    Tile<1> &se = tile_at<1>(sm, 0);
    fcg_load_e(se, G, e, blockIdx.x, blockIdx.y);
    __syncthreads();
    int i, k;
    if (cell_of(G, blockIdx.x, blockIdx.y, i, k)) {
        const int q = cidx(G, i, k);
        const int y = threadIdx.y + 1, x = threadIdx.x + 1;
        s[q] = fma(-g, fcg_ae(L, q, i, k, se, y, x), ld(&r[q]));
    }
}

// z = g e + z_MG (the V-cycle's output in e2), written to e2; acc += z.q_old
// (none before the first direction); beta = -z.q_old / p_old.q_old.
__global__ void k_fcg_out(Level L, const float *e, const double *q_old, Scal *sc, double *partials)
{
    if (loop_over(sc, LOOP_CG)) return;
    __shared__ double red[NTHREADS];
    const Geom &G = L.G;
    const bool first = sc->cg_it == 0;
    const double g = sc->galpha;
    double acc[1] = {0.0}, tot[1];
    int i, k;
    if (cell_of(G, blockIdx.x, blockIdx.y, i, k)) {
        const int q = cidx(G, i, k);
        const double z = fma(g, (double)e[(size_t)k * G.nx + i], L.e2[q]);
        L.e2[q] = z;
        if (!first) acc[0] = z * ld(&q_old[q]);
    }
    if (grid_sum<1>(acc, red, partials, &sc->counters[CNT_RZ], tot)) {
        sc->beta = (first || sc->pq == 0.0) ? 0.0 : -tot[0] / sc->pq;
        if (!isfinite(tot[0])) sc->status = GEA_ERR_NONFINITE;
    }
}

// r for the network (FP32, dense), from the residual of the current iteration.
__global__ void k_fcg_stage_in(Level L, float *dense, Scal *sc)
{
    if (loop_over(sc, LOOP_CG)) return;
    const Geom &G = L.G;
    int i, k;
    if (!cell_of(G, blockIdx.x, blockIdx.y, i, k)) return;
    dense[(size_t)k * G.nx + i] = (float)ld(&res_of(L, sc->cg_it)[cidx(G, i, k)]);
}

// p = z + beta p_old (on the tile and its halo), q = A p; acc += (p.q, r.p);
// alpha = r.p / p.q.
__global__ void k_fcg_pspmv(StepArgs a, Level L)
{
    Scal *sc = a.sc;
    if (loop_over(sc, LOOP_CG)) return;
    __shared__ double sm[kT1];
    __shared__ double red[2 * NTHREADS];
    const Geom &G = L.G;
    const int it = sc->cg_it;
    const double *pold = (it & 1) ? a.p1 : a.p0;
    double *pnew = (it & 1) ? a.p0 : a.p1;
    const double *r = res_of(L, it);
    const double beta = sc->beta;
    const int bx = blockIdx.x, bz = blockIdx.y;
    Tile<1> &sp = tile_at<1>(sm, 0);
    if (it == 0)
        load_tile_fn<1, double>(sp, G, bx, bz, [&](int q, int, int) { return ld(&L.e2[q]); });
    else
        load_tile_fn<1, double>(sp, G, bx, bz, [&](int q, int, int) { return fma(beta, ld(&pold[q]), ld(&L.e2[q])); });
    __syncthreads();
    double acc[2] = {0.0, 0.0}, tot[2];
    int i, k;
    if (cell_of(G, bx, bz, i, k)) {
        const int q = cidx(G, i, k);
        const int y = threadIdx.y + 1, x = threadIdx.x + 1;
        const double pq = sp[y][x];
        const double Ap = helm_tile<1, double>(L, q, i, k, sp, y, x);
        pnew[q] = pq;
        a.q[q] = Ap;
        acc[0] = pq * Ap;
        acc[1] = ld(&r[q]) * pq;
    }
    if (grid_sum<2>(acc, red, a.partials, &sc->counters[CNT_PQ], tot)) {
        sc->pq = tot[0];
        sc->alpha = tot[0] != 0.0 ? tot[1] / tot[0] : 0.0;
        if (!isfinite(tot[0]) || !isfinite(tot[1])) sc->status = GEA_ERR_NONFINITE;
    }
}

// x += alpha p, r_new = r - alpha q (into the other residual buffer); acc += r_new^2.
__global__ void k_fcg_update(StepArgs a, Level L, double *x)
{
    Scal *sc = a.sc;
    if (loop_over(sc, LOOP_CG)) return;
    __shared__ double red[NTHREADS];
    const Geom &G = L.G;
    const int it = sc->cg_it;
    const double *p = (it & 1) ? a.p0 : a.p1;
    const double *rin = res_of(L, it);
    double *rout = res_of(L, it + 1);
    const double alpha = sc->alpha;
    double acc[1] = {0.0}, tot[1];
    int i, k;
    if (cell_of(G, blockIdx.x, blockIdx.y, i, k)) {
        const int q = cidx(G, i, k);
        x[q] = fma(alpha, ld(&p[q]), x[q]);
        const double rn = fma(-alpha, ld(&a.q[q]), ld(&rin[q]));
        rout[q] = rn;
        acc[0] = rn * rn;
    }
    if (grid_sum<1>(acc, red, a.partials, &sc->counters[CNT_UPD], tot)) fin_update(sc, tot, a.cg_rtol2);
}

}  // namespace

template <class R>
void launch_guess_in(const StepArgs &a, const LevelT<R> &L, const R *r, float *dense_r,
                     cudaGraphConditionalHandle h, bool graph, cudaStream_t st, Tracer *tr)
{
    const Geom &G = L.G;
    TRACED(tr, "guess_in", ncell(G),
           (k_guess_in<R><<<grid_of(G), kBlock, 0, st>>>(G, r, dense_r, a.sc, h, graph ? 1 : 0,
                                                          2 + gea_net_launches())));
}

template <class R>
int launch_net_guess(const StepArgs &a, const LevelT<R> &L, R *r, R *q, R *x, double tol2, gea_net *net,
                     float *dense_r, float *dense_e, cudaStream_t st, Tracer *tr)
{
    const Geom &G = L.G;
    if (tr) tr->begin("net_forward", ncell(G), st);
    const int nk = gea_net_run(net, st, 1, G.nz, G.nx, dense_r, dense_e);
    if (tr) tr->end(st);
    if (nk < 0) return -1;
    TRACED(tr, "guess_dots", ncell(G),
           (k_guess_dots<R><<<grid_of(G), kBlock, 0, st>>>(L, dense_e, r, q, a.sc, a.partials)));
    TRACED(tr, "guess_apply", ncell(G),
           (k_guess_apply<R><<<grid_of(G), kBlock, 0, st>>>(L, dense_e, q, r, x, a.sc, a.partials, tol2)));
    return 2 + nk;
}

int launch_fcg_iter(const StepArgs &a, Level *L, int nlev, double *x, gea_net *net, float *dense_r,
                    float *dense_e, double *s_buf, cudaStream_t st, Tracer *tr)
{
    const Geom &G = L[0].G;
    TRACED(tr, "fcg_stage_in", ncell(G), (k_fcg_stage_in<<<grid_of(G), kBlock, 0, st>>>(L[0], dense_r, a.sc)));
    if (tr) tr->begin("net_forward", ncell(G), st);
    const int nk = gea_net_run(net, st, 1, G.nz, G.nx, dense_r, dense_e);
    if (tr) tr->end(st);
    if (nk < 0) return -1;
    TRACED(tr, "fcg_dots", ncell(G), (k_fcg_dots<<<grid_of(G), kBlock, 0, st>>>(L[0], dense_e, a.sc, a.partials)));
    TRACED(tr, "fcg_rest", ncell(G),
           (k_fcg_rest<<<grid_of(G), kBlock, 0, st>>>(L[0], dense_e, s_buf, a.sc)));
    // the V-cycle on s: a copy of the levels whose finest residual buffers
    // both name s_buf
    Level M[kMaxLevels];
    for (int l = 0; l < nlev; ++l) M[l] = L[l];
    M[0].r = M[0].r_alt = s_buf;
    const int nv = launch_vcycle<double>(a, M, nlev, st, tr);
    TRACED(tr, "fcg_out", ncell(G),
           (k_fcg_out<<<grid_of(G), kBlock, 0, st>>>(L[0], dense_e, a.q, a.sc, a.partials)));
    TRACED(tr, "fcg_pspmv", ncell(G), (k_fcg_pspmv<<<grid_of(G), kBlock, 0, st>>>(a, L[0])));
    TRACED(tr, "fcg_update", ncell(G), (k_fcg_update<<<grid_of(G), kBlock, 0, st>>>(a, L[0], x)));
    return 6 + nk + nv;
}

template void launch_guess_in<double>(const StepArgs &, const LevelT<double> &, const double *, float *,
                                      cudaGraphConditionalHandle, bool, cudaStream_t, Tracer *);
template void launch_guess_in<float>(const StepArgs &, const LevelT<float> &, const float *, float *,
                                     cudaGraphConditionalHandle, bool, cudaStream_t, Tracer *);
template int launch_net_guess<double>(const StepArgs &, const LevelT<double> &, double *, double *, double *,
                                      double, gea_net *, float *, float *, cudaStream_t, Tracer *);
template int launch_net_guess<float>(const StepArgs &, const LevelT<float> &, float *, float *, float *, double,
                                     gea_net *, float *, float *, cudaStream_t, Tracer *);

void launch_loop_ctl(Scal *sc, cudaGraphConditionalHandle h, bool graph, int which,
                     int maxtrips, int body_launches, cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "loop_ctl", 1,
           (k_loop_ctl<<<1, 1, 0, st>>>(sc, h, graph ? 1 : 0, which, maxtrips, body_launches)));
}

void launch_loop_gate(Scal *sc, cudaGraphConditionalHandle h, int which, cudaStream_t st)
{
    k_loop_gate<<<1, 1, 0, st>>>(sc, h, which);
}

void launch_step_begin(Scal *sc, cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "step_begin", 1, (k_step_begin<<<1, 1, 0, st>>>(sc)));
}

void launch_step_end(Scal *sc, int fixed_launches, cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "step_end", 1, (k_step_end<<<1, 1, 0, st>>>(sc, fixed_launches)));
}

void launch_diag(const Geom &G, const Phys &F, const State &S, const double *theta_bar,
                 double *theta_out, Scal *sc, double *partials, cudaStream_t st)
{
    k_diag<<<grid_of(G), kBlock, 0, st>>>(G, F, S, theta_bar, theta_out, sc, partials);
}

}  // namespace gea
