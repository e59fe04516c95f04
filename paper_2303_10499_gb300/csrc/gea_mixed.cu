// gea_mixed.cu -- per-phase kernels of the mixed-precision time step (the
// GEA pressure-based Euler scheme of Girfoglio, Quaini & Rozza, arXiv
// 2303.10499, Section 3, unchanged) and their launchers.
//
// On GB300 FP32 issues 64 times faster than FP64. The mixed path keeps
// everything that carries the hydrostatic balance or the conservation
// properties in FP64 -- the state, p' = p + rho g z, rho^{2/3}, the face
// forces, the right-hand sides, H(u), the flux correction -- and moves the
// iterative solves to FP32 by defect correction: each implicit problem
// T x = b gets one FP64 residual r0 = b - T x_old, an FP32 solve T dx = r0 to a
// relative residual of mp_rtol, 1e-5 by default (Jacobi for the predictors, multigrid-
// preconditioned CG for the pressure equation) and the FP64 update
// x = x_old + dx. Increments have homogeneous wall conditions (the h ghost
// offset g dz cancels). FP32 reductions are summed per block in FP32 and
// across blocks in FP64.
#include "gea_internal.cuh"
#include "gea_tiles.cuh"

namespace gea {

namespace {

using namespace tiles;

__global__ void k_mx_pred(StepArgs a, MixedArgs m)
{
    if (a.sc->status) return;
    __shared__ double sm[2 * kT2];
    __shared__ double red[2 * NTHREADS];
    double acc[2] = {0.0, 0.0}, tot[2];
    ph_pred_t<true>(a, m, sm, blockIdx.x, blockIdx.y, acc);
    if (grid_sum<2>(acc, red, a.partials, &a.sc->counters[CNT_PRED], tot)) fin_pred(a.sc, tot);
}

// Sweep pairs as in the FP64 path: the second sweep of a pair copies once the
// first met the tolerance.
__global__ void k_mx_mom(StepArgs a, MixedArgs m, const float *ui, const float *wi, float *uo, float *wo,
                         int second)
{
    if (a.sc->status) return;
    if (second && a.sc->done[LOOP_MOM]) {
        block_tiles(a.G, [&](int bx, int bz) {
            ph_copy(a.G, ui, uo, bx, bz);
            ph_copy(a.G, wi, wo, bx, bz);
        });
        return;
    }
    __shared__ double sm[kT2];
    __shared__ double red[2 * NTHREADS];
    float acc[2] = {0.0f, 0.0f};
    double tot[2];
    block_tiles(a.G, [&](int bx, int bz) {
        ph_sweep2<float, BC_U, BC_W>(a.G, a.F, m.T, m.dinvu, m.r0u, m.r0w, ui, wi, uo, wo, sm, bx, bz, acc);
    });
    if (grid_sum<2, float>(acc, red, a.partials, &a.sc->counters[CNT_MOM], tot)) fin_mom(a.sc, tot, m.tol2);
}

__global__ void k_mx_enth_rhs(StepArgs a, MixedArgs m)
{
    if (a.sc->status) return;
    __shared__ double sm[3 * kT2];
    __shared__ double red[NTHREADS];
    double acc[1] = {0.0}, tot[1];
    ph_enth_rhs_t<true>(a, m, nullptr, nullptr, nullptr, sm, blockIdx.x, blockIdx.y, acc);
    if (grid_sum<1>(acc, red, a.partials, &a.sc->counters[CNT_ENTH_RHS], tot)) fin_enth_rhs(a.sc, tot);
}

__global__ void k_mx_enth(StepArgs a, MixedArgs m, const float *hi, float *ho, int second)
{
    if (a.sc->status) return;
    if (second && a.sc->done[LOOP_ENTH]) {
        block_tiles(a.G, [&](int bx, int bz) { ph_copy(a.G, hi, ho, bx, bz); });
        return;
    }
    __shared__ double sm[kT2];
    __shared__ double red[NTHREADS];
    float acc[1] = {0.0f};
    double tot[1];
    block_tiles(a.G, [&](int bx, int bz) {
        ph_sweep1<float, BC_EVEN>(a.G, a.F, m.T, m.dinvh, m.r0h, (float)(a.F.mu - a.F.nuh), hi, ho, sm, bx, bz,
                                  acc);
    });
    if (grid_sum<1, float>(acc, red, a.partials, &a.sc->counters[CNT_ENTH], tot)) fin_enth(a.sc, tot, m.tol2);
}

__global__ void k_mx_eos(StepArgs a, Level L, LevelF L32, const float *dh)
{
    if (a.sc->status) return;
    __shared__ double sm[2 * kT1 + kFaces];
    ph_eos_t<true>(a, L, L32, nullptr, dh, sm, blockIdx.x, blockIdx.y);
}

__global__ void k_mx_helm_rhs(StepArgs a, Level L, LevelF L32, MixedArgs m, const double *xin,
                              bool guess, int corr)
{
    if (a.sc->status) return;
    __shared__ double sm[4 * kT1];
    __shared__ double red[2 * NTHREADS];
    double acc[2] = {0.0, 0.0}, tot[2];
    ph_helm_rhs_t<true>(a, L, L32, m, xin, nullptr, guess, sm, blockIdx.x, blockIdx.y, acc);
    if (grid_sum<2>(acc, red, a.partials, &a.sc->counters[CNT_HELM], tot))
        fin_helm_mixed(a.sc, tot, a.cg_rtol2, corr);
}

inline dim3 grid_of(const Geom &G) { return dim3((G.nx + BX - 1) / BX, (G.nz + BZ - 1) / BZ); }
const dim3 kBlock(BX, BZ);
inline long long ncell(const Geom &G) { return (long long)G.nx * G.nz; }

#define TRACED(tr, name, cells, launch)                         \
    do {                                                        \
        if (tr) (tr)->begin(name, (long long)(cells), st);      \
        launch;                                                 \
        if (tr) (tr)->end(st);                                  \
    } while (0)

}  // namespace

void launch_mx_pred(const StepArgs &a, const MixedArgs &m, cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "mx_pred", ncell(a.G), (k_mx_pred<<<grid_of(a.G), kBlock, 0, st>>>(a, m)));
}

void launch_mx_mom(const StepArgs &a, const MixedArgs &m, const float *ui, const float *wi, float *uo,
                   float *wo, int second, cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "mx_mom", ncell(a.G),
           (k_mx_mom<<<grid_tiles(a.G, a.tiles_per_block), kBlock, 0, st>>>(a, m, ui, wi, uo, wo, second)));
}

void launch_mx_enth_rhs(const StepArgs &a, const MixedArgs &m, cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "mx_enth_rhs", ncell(a.G), (k_mx_enth_rhs<<<grid_of(a.G), kBlock, 0, st>>>(a, m)));
}

void launch_mx_enth(const StepArgs &a, const MixedArgs &m, const float *hi, float *ho, int second,
                    cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "mx_enth", ncell(a.G), (k_mx_enth<<<grid_tiles(a.G, a.tiles_per_block), kBlock, 0, st>>>(a, m, hi, ho, second)));
}

void launch_mx_eos(const StepArgs &a, const Level &L0, const LevelF &L32, const float *dh, cudaStream_t st,
                   Tracer *tr)
{
    TRACED(tr, "mx_eos", ncell(a.G), (k_mx_eos<<<grid_of(a.G), kBlock, 0, st>>>(a, L0, L32, dh)));
}

void launch_mx_helm_rhs(const StepArgs &a, const Level &L0, const LevelF &L32, const MixedArgs &m,
                        const double *xin, bool guess, int corr, cudaStream_t st, Tracer *tr)
{
    TRACED(tr, "mx_helm_rhs", ncell(a.G),
           (k_mx_helm_rhs<<<grid_of(a.G), kBlock, 0, st>>>(a, L0, L32, m, xin, guess, corr)));
}

}  // namespace gea
