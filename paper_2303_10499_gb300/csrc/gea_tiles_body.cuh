// gea_tiles_body.cuh -- the phases of one time step of the GEA
// pressure-based Euler solver (Girfoglio, Quaini & Rozza, arXiv 2303.10499,
// Section 3) as tile-level device functions. A tile is BX x BZ cells, one
// per thread of a BX x BZ block of NTHREADS = 256 threads; (bx, bz) are the
// tile's coordinates. Both the per-phase kernels (gea_kernels.cu) and the
// persistent step kernels (gea_persistent_body.cuh) run these functions; the
// persistent kernel walks the tiles of a phase in a block-stride loop and
// separates phases with grid barriers.
//
// This file has no include guard and no namespace of its own: it is
// included inside one namespace per tile shape, where BX and BZ name the
// shape (gea_tiles.cuh: namespace gea::tiles, the 32 x 8 tile of the
// per-phase kernels; gea_persistent_*.cu: one namespace per shape of the
// persistent kernels, whose shape the tile-shape autotuner picks).
//
// GB300 executes FP64 at 1/64 of its FP32 rate (two FP64 lanes per SM per
// clock, about 1.2 TFLOP/s) while HBM delivers about 6.8 TB/s, so every phase
// is FP64-issue-bound. The functions execute as few FP64 instructions as
// possible and spend loads, integer and shared-memory work instead:
//  - neighbour values come from a shared-memory tile with a halo, wall ghosts
//    filled while loading, so the arithmetic has no boundary branches;
//  - the implicit transport operator of Steps 1-2 is assembled once per step
//    as a 9-point stencil; a Jacobi sweep and H(u) are 9 FMAs per component;
//  - the Helmholtz operator is kept as d x - sum a x_N with 1/d stored; values
//    needed at neighbours are computed once per tile cell;
//  - divisions are done once per step into stored reciprocals.
// Global reads go through L2 (ld.global.cg): within one persistent launch a
// buffer is rewritten by other blocks between phases, and L1 is not coherent
// across SMs.
//
// Shared memory: each function takes `sm`, a block-wide scratch area of at
// least kTileSmem doubles, and ends with a __syncthreads() so the next tile
// can reuse it. Reduction contributions are added to the caller's per-thread
// accumulators.
static_assert(BX * BZ == NTHREADS && BX % 2 == 0 && BZ % 2 == 0,
              "a tile is NTHREADS cells with even sides (2 x 2 restriction within a tile)");

template <int H, class R = double>
using Tile = R[BZ + 2 * H][BX + 2 * H];

constexpr int kT1 = (BZ + 2) * (BX + 2);   // doubles of a halo-1 tile
constexpr int kT2 = (BZ + 4) * (BX + 4);   // doubles of a halo-2 tile
constexpr int cmax(int a, int b) { return a > b ? a : b; }
constexpr int kPW = BX + 2;                // columns of a pair tile (red-black phases)
constexpr int kPH2 = (BZ + 4) * kPW;       // doubles of a pair tile with two halo rows
constexpr int kPH1 = (BZ + 2) * kPW;       // with one
constexpr int kFaces = BZ * (BX + 1) + (BZ + 1) * BX;   // x- and z-face values of a tile
constexpr int kCorrectSmem = 2 * kT1 + cmax(kFaces, kT2);   // of the correction
// the largest phase footprint: four halo-1 tiles (pressure right-hand
// side), three halo-2 tiles (enthalpy right-hand side), two halo-1 tiles and
// the face values or a halo-2 tile (EOS, correction), or two pair tiles and
// a tile of residuals (V-cycle)
constexpr int kTileSmem =
    cmax(cmax(4 * kT1, 3 * kT2), cmax(kCorrectSmem, kPH2 + kPH1 + BZ * BX));

template <int H, class R = double>
__device__ __forceinline__ Tile<H, R> &tile_at(double *sm, int slot)
{
    return *reinterpret_cast<Tile<H, R> *>(reinterpret_cast<R *>(sm) + slot * (BZ + 2 * H) * (BX + 2 * H));
}

__device__ __forceinline__ double ld(const double *p) { return __ldcg(p); }
__device__ __forceinline__ float ld(const float *p) { return __ldcg(p); }

__device__ __forceinline__ bool cell_of(const Geom &G, int bx, int bz, int &i, int &k)
{
    i = bx * BX + threadIdx.x;
    k = bz * BZ + threadIdx.y;
    return i < G.nx && k < G.nz;
}

// Cell value at (i,k) just outside the box: the one-layer wall ghost of rule
// BC (wall-normal velocity odd, tangential velocity and scalars even, h with
// dh/dz = -g at the horizontal walls).
template <int BC, class R>
__device__ __forceinline__ R ghost(const Geom &G, const Phys &F, const R *X, int i, int k)
{
    if (i < 0) {
        const R v = ld(&X[k * G.P]);
        return BC == BC_U ? -v : v;
    }
    if (i >= G.nx) {
        const R v = ld(&X[k * G.P + G.nx - 1]);
        return BC == BC_U ? -v : v;
    }
    if (k < 0) {
        const R v = ld(&X[i]);
        if (BC == BC_W) return -v;
        if (BC == BC_H) return v + (R)(F.g * G.dz);
        return v;
    }
    const R v = ld(&X[(G.nz - 1) * G.P + i]);
    if (BC == BC_W) return -v;
    if (BC == BC_H) return v - (R)(F.g * G.dz);
    return v;
}

// Fill the (BZ+2H) x (BX+2H) tile of X around tile (bx, bz): cells inside the
// box, the one-layer wall ghosts of rule BC, zero elsewhere (deeper ghosts and
// corners only ever meet zero coefficients).
template <int BC, int H, class R>
__device__ __forceinline__ void load_tile(Tile<H, R> &s, const Geom &G, const Phys &F, const R *X,
                                          int bx, int bz)
{
    const int i0 = bx * BX - H, k0 = bz * BZ - H;
    // h differs from an even field only in its ghost rows below and above
    // the box; a tile that reaches neither (block-uniform test) loads it as
    // even, without the ghost offset's FP64 arithmetic in the loop
    if constexpr (BC == BC_H) {
        if (k0 >= 0 && k0 + BZ + 2 * H <= G.nz) {
            load_tile<BC_EVEN, H, R>(s, G, F, X, bx, bz);
            return;
        }
    }
    const int tid = threadIdx.x + threadIdx.y * BX;
    constexpr int W = BX + 2 * H, NE = (BZ + 2 * H) * (BX + 2 * H);
    for (int e = tid; e < NE; e += NTHREADS) {
        const int tk = e / W, ti = e - tk * W;
        const int i = i0 + ti, k = k0 + tk;
        const bool xin = i >= 0 && i < G.nx, zin = k >= 0 && k < G.nz;
        R v = 0;
        if (xin && zin) v = ld(&X[k * G.P + i]);
        else if (zin && (i == -1 || i == G.nx)) v = ghost<BC>(G, F, X, i, k);
        else if (xin && (k == -1 || k == G.nz)) v = ghost<BC>(G, F, X, i, k);
        s[tk][ti] = v;
    }
}

// Tile of X + Y (FP64 field plus FP32 increment with the same wall rule).
template <int BC, int H>
__device__ __forceinline__ void load_tile_sum(Tile<H> &s, const Geom &G, const Phys &F, const double *X,
                                              const float *Y, int bx, int bz)
{
    const int i0 = bx * BX - H, k0 = bz * BZ - H;
    const int tid = threadIdx.x + threadIdx.y * BX;
    constexpr int W = BX + 2 * H, NE = (BZ + 2 * H) * (BX + 2 * H);
    for (int e = tid; e < NE; e += NTHREADS) {
        const int tk = e / W, ti = e - tk * W;
        const int i = i0 + ti, k = k0 + tk;
        const bool xin = i >= 0 && i < G.nx, zin = k >= 0 && k < G.nz;
        double v = 0.0;
        if (xin && zin) v = ld(&X[k * G.P + i]) + (double)ld(&Y[k * G.P + i]);
        else if ((zin && (i == -1 || i == G.nx)) || (xin && (k == -1 || k == G.nz)))
            v = ghost<BC>(G, F, X, i, k) + (double)ghost<BC == BC_H ? BC_EVEN : BC>(G, F, Y, i, k);
        s[tk][ti] = v;
    }
}

// Same for a field given by f(q, i, k) at cell (i, k), index q (zero outside
// the box).
template <int H, class R, class Fn>
__device__ __forceinline__ void load_tile_fn(Tile<H, R> &s, const Geom &G, int bx, int bz, Fn f)
{
    const int i0 = bx * BX - H, k0 = bz * BZ - H;
    const int tid = threadIdx.x + threadIdx.y * BX;
    constexpr int W = BX + 2 * H, NE = (BZ + 2 * H) * (BX + 2 * H);
    for (int e = tid; e < NE; e += NTHREADS) {
        const int tk = e / W, ti = e - tk * W;
        const int i = i0 + ti, k = k0 + tk;
        s[tk][ti] = (i >= 0 && i < G.nx && k >= 0 && k < G.nz) ? (R)f(k * G.P + i, i, k) : (R)0;
    }
}

// Y = X on the tile's cells.
template <class R>
__device__ __forceinline__ void ph_copy(const Geom &G, const R *X, R *Y, int bx, int bz)
{
    int i, k;
    if (cell_of(G, bx, bz, i, k)) Y[cidx(G, i, k)] = ld(&X[cidx(G, i, k)]);
}

// 5-point Laplacian (X_E + X_W - 2 X_C)/dx^2 + (X_N + X_S - 2 X_C)/dz^2.
template <int H, class R>
__device__ __forceinline__ R lap5(const Phys &F, const Tile<H, R> &s, int y, int x)
{
    const R c2 = (R)2 * s[y][x];
    return (s[y][x + 1] + s[y][x - 1] - c2) * (R)F.ix2 + (s[y + 1][x] + s[y - 1][x] - c2) * (R)F.iz2;
}

// A x = d x - sum a x_N at tile position (y, x) of cell (i, k) (zero tile
// entries and zero wall coefficients beyond the box).
template <int H, class R>
__device__ __forceinline__ R helm_tile(const LevelT<R> &L, int q, int i, int k, const Tile<H, R> &s,
                                       int y, int x)
{
    const Geom &G = L.G;
    R t = ld(&L.d[q]) * s[y][x];
    t = fma(-ld(&L.ax[k * G.P + i]), s[y][x - 1], t);
    t = fma(-ld(&L.ax[k * G.P + i + 1]), s[y][x + 1], t);
    t = fma(-ld(&L.az[k * G.P + i]), s[y - 1][x], t);
    t = fma(-ld(&L.az[(k + 1) * G.P + i]), s[y + 1][x], t);
    return t;
}

// The coefficients of the Helmholtz operator at a cell. With kPrefetch (set
// by the includer: the persistent kernels, whose occupancy the register
// file already fixes at three blocks per SM) the phases load a cell's own
// coefficients and inputs ahead of the tile barrier (they do not depend on
// the tile), so that their L2 latency overlaps the halo loads; without it
// (the per-phase kernels, where the extra live registers would cost
// occupancy) after the barrier. Two phases load early in every instance:
// the single-field Jacobi sweep and the CG direction update with A p, which
// measured faster that way in the per-phase kernels too (the 4096 x 2048
// enthalpy sweep went from 0.47 to 0.80 of the FP64 peak), while the
// two-field sweep, the multigrid phases and the right-hand sides lost
// occupancy and speed.
constexpr bool kPrefetchSweep1 = true;
constexpr bool kPrefetchSpmv = true;
template <class R>
struct HelmCoef {
    R d, aw, ae, as, an;
};

template <class R>
__device__ __forceinline__ HelmCoef<R> helm_coef(const LevelT<R> &L, int q, int i, int k)
{
    const Geom &G = L.G;
    return HelmCoef<R>{ld(&L.d[q]), ld(&L.ax[k * G.P + i]), ld(&L.ax[k * G.P + i + 1]), ld(&L.az[k * G.P + i]),
                       ld(&L.az[(k + 1) * G.P + i])};
}

// A x = d x - sum a x_N from preloaded coefficients (helm_tile's order).
template <int H, class R>
__device__ __forceinline__ R helm_apply(const HelmCoef<R> &c, const Tile<H, R> &s, int y, int x)
{
    R t = c.d * s[y][x];
    t = fma(-c.aw, s[y][x - 1], t);
    t = fma(-c.ae, s[y][x + 1], t);
    t = fma(-c.as, s[y - 1][x], t);
    t = fma(-c.an, s[y + 1][x], t);
    return t;
}

// The nine stencil weights of the transport operator at a cell, likewise
// loaded ahead of the tile barrier.
template <class R>
struct Coef9 {
    R cC, cE1, cW1, cN1, cS1, cE2, cW2, cN2, cS2;
};

template <class R>
__device__ __forceinline__ Coef9<R> coef9(const Stencil9T<R> &T, int q)
{
    return Coef9<R>{ld(&T.cC[q]),  ld(&T.cE1[q]), ld(&T.cW1[q]), ld(&T.cN1[q]), ld(&T.cS1[q]),
                    ld(&T.cE2[q]), ld(&T.cW2[q]), ld(&T.cN2[q]), ld(&T.cS2[q])};
}

// b - sum_o c_o X_o as one chain of nine FMAs.
template <int H, class R>
__device__ __forceinline__ R sub9c(R b, const Coef9<R> &c, const Tile<H, R> &s, int y, int x)
{
    R acc = fma(-c.cC, s[y][x], b);
    acc = fma(-c.cE1, s[y][x + 1], acc);
    acc = fma(-c.cW1, s[y][x - 1], acc);
    acc = fma(-c.cN1, s[y + 1][x], acc);
    acc = fma(-c.cS1, s[y - 1][x], acc);
    acc = fma(-c.cE2, s[y][x + 2], acc);
    acc = fma(-c.cW2, s[y][x - 2], acc);
    acc = fma(-c.cN2, s[y + 2][x], acc);
    return fma(-c.cS2, s[y - 2][x], acc);
}

// ---------------------------------------------------------------------------
// Smagorinsky eddy viscosity (LES): mu_eff = mu + rho (cs Delta)^2 |S| from
// rho^n and u^n, |S|^2 = 2 (du/dx)^2 + 2 (dw/dz)^2 + (du/dz + dw/dx)^2 with
// central differences (ghosts by the wall rules)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void ph_les(const StepArgs &a, double *sm, int bx, int bz)
{
    const Geom &G = a.G;
    const Phys &F = a.F;
    Tile<1> &su = tile_at<1>(sm, 0), &sw = tile_at<1>(sm, 1);
    load_tile<BC_U, 1>(su, G, F, a.S.u, bx, bz);
    load_tile<BC_W, 1>(sw, G, F, a.S.w, bx, bz);
    __syncthreads();
    int i, k;
    if (cell_of(G, bx, bz, i, k)) {
        const int q = cidx(G, i, k);
        const int y = threadIdx.y + 1, x = threadIdx.x + 1;
        const double hx = 0.5 * G.idx, hz = 0.5 * G.idz;
        const double dudx = (su[y][x + 1] - su[y][x - 1]) * hx, dudz = (su[y + 1][x] - su[y - 1][x]) * hz;
        const double dwdx = (sw[y][x + 1] - sw[y][x - 1]) * hx, dwdz = (sw[y + 1][x] - sw[y - 1][x]) * hz;
        const double sh = dudz + dwdx;
        const double S = sqrt(2.0 * dudx * dudx + 2.0 * dwdz * dwdz + sh * sh);
        a.mueff[q] = fma(ld(&a.S.rho[q]) * F.les_d2, S, F.mu);
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// Step 1 (eq. e1_d and eq. step2_sd, first line)
// ---------------------------------------------------------------------------

// rho^{n+1/3} = rho^n - dt sum_j phi_j / V; the transport operator
//   T(X) = (rho1/dt) X + C(X) - mu L(X)
// as a 9-point stencil: the east face contributes f_e (-X_W1 + 7 X_C + 7 X_E1
// - X_E2) with f_e = phi_e / (12 V), the west face -f_w (-X_W2 + 7 X_W1 + 7 X_C
// - X_E1), likewise in z, and -mu L adds 2 mu (1/dx^2 + 1/dz^2) at the centre
// and -mu/dx^2, -mu/dz^2 at the nearest neighbours; the Jacobi reciprocals of
// the momentum (mu) and enthalpy (mu/Pr) diagonals; b = rho^n u^n / dt - G_cell^n
// with G_cell the average of the two face forces grad p'^n - g z grad rho^n
// per direction (zero on wall faces); the initial guess u^n.
// acc += (b_u^2, b_w^2).
//
// MX (mixed-precision path): instead of b, the reciprocals and the initial
// guess, the FP64 residuals r0 = b - T(u^n) of both components, FP32 copies
// of the operator, the reciprocals and r0, and the first FP32 Jacobi sweep
// from zero, du = r0 / T_CC; acc += (r0_u^2, r0_w^2).
//
// SW1 (FP64): also the first Jacobi sweep of the momentum predictor from the
// guess u^n, r0 = b - T(u^n), u = u^n + r0 / T_CC into ua, wa (the stencil of
// the cell is at hand and u^n needs no barrier); acc += (b_u^2, b_w^2,
// r0_u^2, r0_w^2).
template <bool MX, bool SW1 = false>
__device__ __forceinline__ void ph_pred_t(const StepArgs &a, const MixedArgs &m, double *sm, int bx,
                                          int bz, double (&acc)[SW1 ? 4 : 2])
{
    const Geom &G = a.G;
    const Phys &F = a.F;
    const State &S = a.S;
    if (MX || SW1) {
        load_tile<BC_U, 2>(tile_at<2>(sm, 0), G, F, S.u, bx, bz);
        load_tile<BC_W, 2>(tile_at<2>(sm, 1), G, F, S.w, bx, bz);
        __syncthreads();
    }
    int i, k;
    if (cell_of(G, bx, bz, i, k)) {
        const int q = cidx(G, i, k);
        const double pw = ld(&S.phix[q]), pe = ld(&S.phix[q + 1]), ps = ld(&S.phiz[q]), pn = ld(&S.phiz[q + G.P]);
        const double div = (pe - pw + pn - ps) * G.iV;
        const double rq = ld(&S.rho[q]);
        const double rho1 = fma(-F.dt, div, rq);
        const double fe = pe * F.s12, fw = pw * F.s12, fn = pn * F.s12, fs = ps * F.s12;
        // diffusion: mu/dx^2 per face, or with LES the face mean of mu_eff
        // (a wall face takes the cell's own)
        double me, mw, mn, ms, md;
        if (F.les) {
            const double mc = ld(&a.mueff[q]);
            me = (mc + (i + 1 < G.nx ? ld(&a.mueff[q + 1]) : mc)) * F.hix2;
            mw = (mc + (i > 0 ? ld(&a.mueff[q - 1]) : mc)) * F.hix2;
            mn = (mc + (k + 1 < G.nz ? ld(&a.mueff[q + G.P]) : mc)) * F.hiz2;
            ms = (mc + (k > 0 ? ld(&a.mueff[q - G.P]) : mc)) * F.hiz2;
            md = (me + mw) + (mn + ms);
        } else {
            me = mw = F.mux;
            mn = ms = F.muz;
            md = F.mud;
        }
        const double cC = fma(rho1, F.idt, fma(7.0 / 12.0, div, md));
        const double cE1 = fma(7.0, fe, fw) - me, cW1 = -fma(7.0, fw, fe) - mw;
        const double cN1 = fma(7.0, fn, fs) - mn, cS1 = -fma(7.0, fs, fn) - ms;
        const double cE2 = -fe, cW2 = fw, cN2 = -fn, cS2 = fs;
        a.T.cC[q] = cC;
        a.T.cE1[q] = cE1;
        a.T.cW1[q] = cW1;
        a.T.cE2[q] = cE2;
        a.T.cW2[q] = cW2;
        a.T.cN1[q] = cN1;
        a.T.cS1[q] = cS1;
        a.T.cN2[q] = cN2;
        a.T.cS2[q] = cS2;
        const double diu = recip(cC);
        double dih = diu;
        rarely(F.pr_ne1, [&] { dih = recip(fma(2.0 * (F.nuh - F.mu), F.ix2 + F.iz2, cC)); });
        if (!MX) {
            a.dinvu[q] = diu;
            a.dinvh[q] = dih;
        }
        // the sum of the two face forces p'_b - p'_a - g z_f (rho_b - rho_a) of each
        // direction (over the spacing): in x both faces have the cell's height;
        // a wall face carries none, which the cell's own values in the place of
        // the missing neighbour's give
        const int qe = i + 1 < G.nx ? q + 1 : q, qw = i > 0 ? q - 1 : q;
        const int qn = k + 1 < G.nz ? q + G.P : q, qs = k > 0 ? q - G.P : q;
        const double sx = fma(-ld(&a.gzc[k]), ld(&S.rho[qe]) - ld(&S.rho[qw]), ld(&S.pp[qe]) - ld(&S.pp[qw]));
        const double sz = fma(-ld(&a.gzf[k + 1]), ld(&S.rho[qn]) - rq,
                              fma(-ld(&a.gzf[k]), rq - ld(&S.rho[qs]), ld(&S.pp[qn]) - ld(&S.pp[qs])));
        const double u = ld(&S.u[q]), w = ld(&S.w[q]);
        const double rdt = rq * F.idt;
        const double bu = fma(-F.hix, sx, rdt * u);
        const double bw = fma(-F.hiz, sz, rdt * w);
        a.rho1[q] = rho1;
        a.dtr1[q] = F.dt * recip(rho1);
        const int y = threadIdx.y + 2, x = threadIdx.x + 2;
        // b - T(X) at the cell from a halo-2 tile
        const Coef9<double> c9{cC, cE1, cW1, cN1, cS1, cE2, cW2, cN2, cS2};
        if (!MX) {
            a.bu[q] = bu;
            a.bw[q] = bw;
            acc[0] = fma(bu, bu, acc[0]);
            acc[1] = fma(bw, bw, acc[1]);
            if (SW1) {
                const double r0u = sub9c<2>(bu, c9, tile_at<2>(sm, 0), y, x), r0w = sub9c<2>(bw, c9, tile_at<2>(sm, 1), y, x);
                a.ua[q] = fma(r0u, diu, u);
                a.wa[q] = fma(r0w, diu, w);
                acc[SW1 ? 2 : 0] = fma(r0u, r0u, acc[SW1 ? 2 : 0]);
                acc[SW1 ? 3 : 1] = fma(r0w, r0w, acc[SW1 ? 3 : 1]);
            } else {
                a.ua[q] = u;
                a.wa[q] = w;
            }
        } else {
            const double r0u = sub9c<2>(bu, c9, tile_at<2>(sm, 0), y, x), r0w = sub9c<2>(bw, c9, tile_at<2>(sm, 1), y, x);
            m.T.cC[q] = (float)cC;
            m.T.cE1[q] = (float)cE1;
            m.T.cW1[q] = (float)cW1;
            m.T.cE2[q] = (float)cE2;
            m.T.cW2[q] = (float)cW2;
            m.T.cN1[q] = (float)cN1;
            m.T.cS1[q] = (float)cS1;
            m.T.cN2[q] = (float)cN2;
            m.T.cS2[q] = (float)cS2;
            const float fdiu = (float)diu;
            m.dinvu[q] = fdiu;
            m.dinvh[q] = (float)dih;
            const float fru = (float)r0u, frw = (float)r0w;
            m.r0u[q] = fru;
            m.r0w[q] = frw;
            m.du[0][q] = fru * fdiu;
            m.dw[0][q] = frw * fdiu;
            acc[0] = fma(r0u, r0u, acc[0]);
            acc[1] = fma(r0w, r0w, acc[1]);
        }
    }
    if (MX || SW1) __syncthreads();
}

__device__ __forceinline__ void ph_pred(const StepArgs &a, int bx, int bz, double (&acc)[2])
{
    ph_pred_t<false>(a, MixedArgs{}, nullptr, bx, bz, acc);
}

__device__ __forceinline__ void ph_pred_sweep(const StepArgs &a, double *sm, int bx, int bz, double (&acc)[4])
{
    ph_pred_t<false, true>(a, MixedArgs{}, sm, bx, bz, acc);
}

// One Jacobi sweep of T(X) = b for two fields with wall rules BCA, BCB:
// r = b - T(X), X <- X + r / T_CC. acc += (r_a^2, r_b^2).
template <class R, int BCA, int BCB>
__device__ __forceinline__ void ph_sweep2(const Geom &G, const Phys &F, const Stencil9T<R> &T,
                                          const R *dinv, const R *ba, const R *bb, const R *xa,
                                          const R *xb, R *ya, R *yb, double *sm, int bx, int bz,
                                          R (&acc)[2])
{
    Tile<2, R> &sa = tile_at<2, R>(sm, 0), &sb = tile_at<2, R>(sm, 1);
    int i, k;
    const bool in = cell_of(G, bx, bz, i, k);
    const int q = in ? cidx(G, i, k) : 0;
    Coef9<R> c{};
    R di = 0, bva = 0, bvb = 0;
    auto fetch = [&] {
        c = coef9(T, q);
        di = ld(&dinv[q]);
        bva = ld(&ba[q]);
        bvb = ld(&bb[q]);
    };
    if (kPrefetch && in) fetch();
    load_tile<BCA, 2, R>(sa, G, F, xa, bx, bz);
    load_tile<BCB, 2, R>(sb, G, F, xb, bx, bz);
    __syncthreads();
    if (in) {
        if (!kPrefetch) fetch();
        const int y = threadIdx.y + 2, x = threadIdx.x + 2;
        const R ra = sub9c<2, R>(bva, c, sa, y, x);
        const R rb = sub9c<2, R>(bvb, c, sb, y, x);
        ya[q] = fma(ra, di, sa[y][x]);
        yb[q] = fma(rb, di, sb[y][x]);
        acc[0] = fma(ra, ra, acc[0]);
        acc[1] = fma(rb, rb, acc[1]);
    }
    __syncthreads();
}

// One Jacobi sweep of T(X) + lc L(X) = b for one field with wall rule BC
// (lc = mu - mu/Pr turns the momentum stencil into the enthalpy one).
// acc += r^2.
template <class R, int BC>
__device__ __forceinline__ void ph_sweep1(const Geom &G, const Phys &F, const Stencil9T<R> &T,
                                          const R *dinv, const R *bv, R lc, const R *xin, R *xout,
                                          double *sm, int bx, int bz, R (&acc)[1])
// (lc is used when F.pr_ne1, i.e. mu/Pr != mu)
{
    Tile<2, R> &sh = tile_at<2, R>(sm, 0);
    int i, k;
    const bool in = cell_of(G, bx, bz, i, k);
    const int q = in ? cidx(G, i, k) : 0;
    Coef9<R> c{};
    R di = 0, bq = 0;
    auto fetch = [&] {
        c = coef9(T, q);
        di = ld(&dinv[q]);
        bq = ld(&bv[q]);
    };
    if (kPrefetchSweep1 && in) fetch();
    load_tile<BC, 2, R>(sh, G, F, xin, bx, bz);
    __syncthreads();
    if (in) {
        if (!kPrefetchSweep1) fetch();
        const int y = threadIdx.y + 2, x = threadIdx.x + 2;
        R r = sub9c<2, R>(bq, c, sh, y, x);
        rarely(F.pr_ne1, [&] { r = fma(-lc, lap5<2, R>(F, sh, y, x), r); });
        xout[q] = fma(r, di, sh[y][x]);
        acc[0] = fma(r, r, acc[0]);
    }
    __syncthreads();
}

// Momentum predictor sweep: u odd in x, w odd in z.
__device__ __forceinline__ void ph_mom(const StepArgs &a, const double *uin, const double *win,
                                       double *uout, double *wout, double *sm, int bx, int bz,
                                       double (&acc)[2])
{
    ph_sweep2<double, BC_U, BC_W>(a.G, a.F, a.T, a.dinvu, a.bu, a.bw, uin, win, uout, wout, sm, bx,
                                  bz, acc);
}

// ---------------------------------------------------------------------------
// Step 2 (eq. step3_sd, step3_2sd, step3_3sd)
// ---------------------------------------------------------------------------

// Right-hand side of the enthalpy equation:
//   (rho^n h^n + rho^n K^n - p^{n-1})/dt - rho1 K1/dt - C(K1) + p^n/dt - rho1 g w1
// with K1 = |u^{n+1/3}|^2/2 (eq. step1_3sd); initial guess h^n (into h0).
// acc += b_h^2.
// MX: u^{n+1/3} = u^n + du (written to ua, wa), and instead of b_h and h0 the
// FP64 residual r0 = b_h - T_h(h^n) (h^n with its wall rule), its FP32 copy
// and the first FP32 sweep dh = r0 / T_h,CC; acc += r0^2 instead.
// SW1 (FP64): h0 receives the first Jacobi sweep from h^n instead of h^n,
// r0 = b_h - T_h(h^n), h = h^n + r0 / T_h,CC; acc += (b_h^2, r0^2).
template <bool MX, bool SW1 = false>
__device__ __forceinline__ void ph_enth_rhs_t(const StepArgs &a, const MixedArgs &m, const double *u1,
                                              const double *w1, double *h0, double *sm, int bx,
                                              int bz, double (&acc)[SW1 ? 2 : 1])
{
    const Geom &G = a.G;
    const Phys &F = a.F;
    const State &S = a.S;
    Tile<2> &su = tile_at<2>(sm, 0), &sw = tile_at<2>(sm, 1);
    if (MX) {
        load_tile_sum<BC_U, 2>(su, G, F, S.u, m.du[0], bx, bz);
        load_tile_sum<BC_W, 2>(sw, G, F, S.w, m.dw[0], bx, bz);
        load_tile<BC_H, 2>(tile_at<2>(sm, 2), G, F, S.h, bx, bz);
    } else {
        load_tile<BC_U, 2>(su, G, F, u1, bx, bz);
        load_tile<BC_W, 2>(sw, G, F, w1, bx, bz);
        if (SW1) load_tile<BC_H, 2>(tile_at<2>(sm, 2), G, F, S.h, bx, bz);
    }
    __syncthreads();
    // 2 K1 in place of u (ghost velocities give the mirrored cell's K); u1 and
    // w1 at the cell centre are kept aside first
    const double u1c = su[threadIdx.y + 2][threadIdx.x + 2], w1c = sw[threadIdx.y + 2][threadIdx.x + 2];
    __syncthreads();
    {
        const int tid = threadIdx.x + threadIdx.y * BX;
        for (int e = tid; e < kT2; e += NTHREADS) {
            const int tk = e / (BX + 4), ti = e - tk * (BX + 4);
            su[tk][ti] = fma(su[tk][ti], su[tk][ti], sw[tk][ti] * sw[tk][ti]);
        }
    }
    __syncthreads();
    int i, k;
    if (cell_of(G, bx, bz, i, k)) {
        const int q = cidx(G, i, k);
        const int y = threadIdx.y + 2, x = threadIdx.x + 2;
        const Tile<2> &K = su;
        // convective sum of K1 with the four-point face values (wall faces
        // carry phi = 0)
        double c = ld(&S.phix[q + 1]) * (7.0 * (K[y][x] + K[y][x + 1]) - (K[y][x - 1] + K[y][x + 2]));
        c -= ld(&S.phix[q]) * (7.0 * (K[y][x - 1] + K[y][x]) - (K[y][x - 2] + K[y][x + 1]));
        c += ld(&S.phiz[q + G.P]) * (7.0 * (K[y][x] + K[y + 1][x]) - (K[y - 1][x] + K[y + 2][x]));
        c -= ld(&S.phiz[q]) * (7.0 * (K[y - 1][x] + K[y][x]) - (K[y - 2][x] + K[y + 1][x]));
        const double rq = ld(&S.rho[q]), u = ld(&S.u[q]), w = ld(&S.w[q]), h = ld(&S.h[q]);
        // b~_e carries rho^n K^n, or rho^n K^{n-1} in the literal reading
        double Kn = 0.5 * fma(u, u, w * w);
        rarely(F.k_lagged, [&] { Kn = ld(&S.Kold[q]); });
        const double rho1 = ld(&a.rho1[q]);
        const double te = fma(rq, h + Kn, -ld(&S.pold[q])) + ld(&S.p[q]);
        const double bh =
            fma(-rho1 * F.g, w1c, fma(F.idt, fma(-0.5 * rho1, K[y][x], te), -(F.s24 * c)));
        if (!MX) {
            a.bh[q] = bh;
            acc[0] = fma(bh, bh, acc[0]);
            if (SW1) {
                const Tile<2> &sh = tile_at<2>(sm, 2);
                double r0 = sub9c<2>(bh, coef9(a.T, q), sh, y, x);
                rarely(F.pr_ne1, [&] { r0 = fma(F.nuh - F.mu, lap5<2>(F, sh, y, x), r0); });
                h0[q] = fma(r0, ld(&a.dinvh[q]), sh[y][x]);
                acc[SW1 ? 1 : 0] = fma(r0, r0, acc[SW1 ? 1 : 0]);
            } else {
                h0[q] = h;
            }
        } else {
            a.ua[q] = u1c;
            a.wa[q] = w1c;
            const Tile<2> &sh = tile_at<2>(sm, 2);
            double r0 = sub9c<2>(bh, coef9(a.T, q), sh, y, x);
            rarely(F.pr_ne1, [&] { r0 = fma(F.nuh - F.mu, lap5<2>(F, sh, y, x), r0); });
            const float fr = (float)r0;
            m.r0h[q] = fr;
            m.dh[0][q] = fr * ld(&m.dinvh[q]);
            acc[0] = fma(r0, r0, acc[0]);
        }
    }
    __syncthreads();
}

__device__ __forceinline__ void ph_enth_rhs(const StepArgs &a, const double *u1, const double *w1,
                                            double *h0, double *sm, int bx, int bz, double (&acc)[1])
{
    ph_enth_rhs_t<false>(a, MixedArgs{}, u1, w1, h0, sm, bx, bz, acc);
}

__device__ __forceinline__ void ph_enth_rhs_sweep(const StepArgs &a, const double *u1, const double *w1,
                                                  double *h0, double *sm, int bx, int bz, double (&acc)[2])
{
    ph_enth_rhs_t<false, true>(a, MixedArgs{}, u1, w1, h0, sm, bx, bz, acc);
}

// One Jacobi sweep of (rho1/dt) h + C(h) - (mu/Pr) L(h) = b_h (dh/dz = -g on
// the horizontal walls): the momentum stencil plus (mu - mu/Pr) L(h).
// acc += r^2.
__device__ __forceinline__ void ph_enth(const StepArgs &a, const double *hin, double *hout,
                                        double *sm, int bx, int bz, double (&acc)[1])
{
    ph_sweep1<double, BC_H>(a.G, a.F, a.T, a.dinvh, a.bh, a.F.mu - a.F.nuh, hin, hout, sm, bx, bz, acc);
}

// T^{n+1} = T^n + (h^{n+1} - h^n)/cp; psi = 1/(R T^{n+1}); rho^{n+2/3} = p^n/(R T^{n+1})
// (eq. step3_3sd); face coefficients D_f = dt rho2_f / rho1_f (linear face
// averages); the fine Helmholtz operator c = psi/dt, a_f = D_f |A_f|/(V Delta_f),
// d = c + sum a_f and 1/d. h1 holds h^{n+1}.
// MX: h^{n+1} = h^n + dh, and FP32 copies of the fine operator into L32.
template <bool MX>
__device__ __forceinline__ void ph_eos_t(const StepArgs &a, const Level &L, const LevelF &L32,
                                         const double *h1, const float *dh, double *sm, int bx, int bz)
{
    const Geom &G = a.G;
    const Phys &F = a.F;
    Tile<1> &s2 = tile_at<1>(sm, 0), &s1 = tile_at<1>(sm, 1);   // dt rho^{n+2/3}, rho^{n+1/3}
    double(*fx)[BX + 1] = reinterpret_cast<double(*)[BX + 1]>(sm + 2 * kT1);
    double(*fz)[BX] = reinterpret_cast<double(*)[BX]>(sm + 2 * kT1 + BZ * (BX + 1));
    const State &S = a.S;
    auto h1_of = [&](int q) { return MX ? ld(&S.h[q]) + (double)ld(&dh[q]) : ld(&h1[q]); };
    int i, k;
    const bool in = cell_of(G, bx, bz, i, k);
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int y = ty + 1, x = tx + 1;
    const int q = in ? cidx(G, i, k) : 0;
    // the cell's own update in registers, and its share of the tile; the ring
    // of halo cells (corners are not used) repeats the density alone
    double h1q = 0.0, T1 = 0.0, psi = 0.0, rho2 = 0.0;
    auto eos = [&](int c, double &hv, double &Tv, double &ps) {
        hv = h1_of(c);
        Tv = fma(hv - ld(&S.h[c]), F.icp, ld(&S.T[c]));
        ps = recip(F.R * Tv);
        return ld(&S.p[c]) * ps;
    };
    if (in) rho2 = eos(q, h1q, T1, psi);
    s2[y][x] = F.dt * rho2;
    s1[y][x] = in ? ld(&a.rho1[q]) : 0.0;
    for (int e = tx + ty * BX; e < 2 * (BX + BZ); e += NTHREADS) {
        const bool row = e < 2 * BX;
        const int tk = row ? (e < BX ? 0 : BZ + 1) : 1 + ((e - 2 * BX) >> 1);
        const int ti = row ? 1 + (e < BX ? e : e - BX) : ((e & 1) ? BX + 1 : 0);
        const int ii = bx * BX - 1 + ti, kk = bz * BZ - 1 + tk;
        double v2 = 0.0, v1 = 0.0;
        if (ii >= 0 && ii < G.nx && kk >= 0 && kk < G.nz) {
            const int c = cidx(G, ii, kk);
            double hv, Tv, ps;
            v2 = F.dt * eos(c, hv, Tv, ps);
            v1 = ld(&a.rho1[c]);
        }
        s2[tk][ti] = v2;
        s1[tk][ti] = v1;
    }
    __syncthreads();
    // dt rho2_f / rho1_f with linear face averages (the two halves cancel
    // exactly in binary)
    auto dface = [&](int ya, int xa, int yb, int xb) {
        return (s2[ya][xa] + s2[yb][xb]) * recip(s1[ya][xa] + s1[yb][xb]);
    };
    if (in) {
        fx[ty][tx] = i > 0 ? dface(y, x - 1, y, x) : 0.0;
        fz[ty][tx] = k > 0 ? dface(y - 1, x, y, x) : 0.0;
        if (tx == BX - 1 || i == G.nx - 1) fx[ty][tx + 1] = i + 1 < G.nx ? dface(y, x, y, x + 1) : 0.0;
        if (ty == BZ - 1 || k == G.nz - 1) fz[ty + 1][tx] = k + 1 < G.nz ? dface(y, x, y + 1, x) : 0.0;
    }
    __syncthreads();
    if (in) {
        a.N.T[q] = T1;
        a.N.h[q] = h1q;
        a.rho2[q] = rho2;
        a.psi[q] = psi;
        const double Dw = fx[ty][tx], De = fx[ty][tx + 1], Ds = fz[ty][tx], Dn = fz[ty + 1][tx];
        a.Dx[k * G.P + i] = Dw;
        a.Dz[k * G.P + i] = Ds;
        const double aw = Dw * F.ix2, as = Ds * F.iz2;
        L.ax[k * G.P + i] = aw;
        L.az[k * G.P + i] = as;
        if (i == G.nx - 1) { a.Dx[k * G.P + G.nx] = 0.0; L.ax[k * G.P + G.nx] = 0.0; }
        if (k == G.nz - 1) { a.Dz[G.nz * G.P + i] = 0.0; L.az[G.nz * G.P + i] = 0.0; }
        const double c = psi * F.idt;
        const double d = fma(Ds + Dn, F.iz2, fma(Dw + De, F.ix2, c));
        L.c[q] = c;
        L.d[q] = d;
        const double id = recip(d);
        L.wd[q] = id;
        if (MX) {
            L32.c[q] = (float)c;
            L32.d[q] = (float)d;
            L32.wd[q] = (float)id;
            L32.ax[k * G.P + i] = (float)aw;
            L32.az[k * G.P + i] = (float)as;
            if (i == G.nx - 1) L32.ax[k * G.P + G.nx] = 0.0f;
            if (k == G.nz - 1) L32.az[G.nz * G.P + i] = 0.0f;
        }
    }
    __syncthreads();
}

__device__ __forceinline__ void ph_eos(const StepArgs &a, const Level &L, const double *h1,
                                       double *sm, int bx, int bz)
{
    ph_eos_t<false>(a, L, LevelF{}, h1, nullptr, sm, bx, bz);
}

// Coarse operator for piecewise-constant transfer: the coarse reaction term
// averages the four fine ones; a coarse face coefficient is cfx or cfz times
// the sum of its two fine faces: a quarter, the Galerkin value, times
// coarse_scale of its direction (an eighth where the spacings are equal). The
// factors are the same on every level; kept in each level's struct they made
// the other kernels' arguments longer (4096x2048: 13.59 -> 13.66 ms a step).
// (bx, bz) is a tile of the coarse level.
template <class R>
__device__ __forceinline__ void ph_coarsen(const LevelT<R> &f, const LevelT<R> &c, double cfx, double cfz,
                                           int bx, int bz)
{
    const Geom &G = c.G;
    int I, K;
    if (!cell_of(G, bx, bz, I, K)) return;
    const int Pf = f.G.P;
    const int q00 = (2 * K) * Pf + 2 * I;
    const int Q = cidx(G, I, K);
    const R q4 = (R)0.25, fx = (R)cfx, fz = (R)cfz;
    const R cc = q4 * (ld(&f.c[q00]) + ld(&f.c[q00 + 1]) + ld(&f.c[q00 + Pf]) + ld(&f.c[q00 + Pf + 1]));
    const R aw = fx * (ld(&f.ax[q00]) + ld(&f.ax[q00 + Pf]));
    const R ae = fx * (ld(&f.ax[q00 + 2]) + ld(&f.ax[q00 + Pf + 2]));
    const R as = fz * (ld(&f.az[q00]) + ld(&f.az[q00 + 1]));
    const R an = fz * (ld(&f.az[q00 + 2 * Pf]) + ld(&f.az[q00 + 2 * Pf + 1]));
    c.c[Q] = cc;
    c.ax[K * G.P + I] = aw;
    c.az[K * G.P + I] = as;
    if (I == G.nx - 1) c.ax[K * G.P + G.nx] = ae;
    if (K == G.nz - 1) c.az[G.nz * G.P + I] = an;
    const R d = cc + aw + ae + as + an;
    c.d[Q] = d;
    c.wd[Q] = (R)1 / d;
}

// ---------------------------------------------------------------------------
// Step 3: PISO corrector (eq. step2_sd second line, eq. p_prime_sd, step4_4sd)
// ---------------------------------------------------------------------------

// H(u) = rho^n u^n/dt - C(u) + mu L(u) = rho^n u^n/dt + (rho1/dt) u - T(u) at the
// newest velocity.
__device__ __forceinline__ void ph_H(const StepArgs &a, const double *U, const double *W, double *sm,
                                     int bx, int bz)
{
    const Geom &G = a.G;
    const Phys &F = a.F;
    Tile<2> &su = tile_at<2>(sm, 0), &sw = tile_at<2>(sm, 1);
    int i, k;
    const bool in = cell_of(G, bx, bz, i, k);
    const int q = in ? cidx(G, i, k) : 0;
    // the cell's stencil weights (shared by both components) and state,
    // loaded ahead of the tile barrier
    Coef9<double> c{};
    double ru = 0.0, rw = 0.0;
    auto fetch = [&] {
        c = coef9(a.T, q);
        const double rdt = ld(&a.S.rho[q]) * F.idt;
        ru = rdt * ld(&a.S.u[q]);
        rw = rdt * ld(&a.S.w[q]);
        c.cC = fma(-ld(&a.rho1[q]), F.idt, c.cC);   // the stencil without its time term
    };
    if (kPrefetch && in) fetch();
    load_tile<BC_U, 2>(su, G, F, U, bx, bz);
    load_tile<BC_W, 2>(sw, G, F, W, bx, bz);
    __syncthreads();
    if (in) {
        if (!kPrefetch) fetch();
        const int y = threadIdx.y + 2, x = threadIdx.x + 2;
        a.Hx[q] = sub9c<2>(ru, c, su, y, x);
        a.Hz[q] = sub9c<2>(rw, c, sw, y, x);
    }
    __syncthreads();
}

// Right-hand side of the pressure equation,
//   b_i = (rho^n_i + psi_i rho2_i g z_i)/dt
//         - (1/V) sum_f D_f |A_f| [H_f . n + g z_f (rho2_N - rho2_i)/Delta_f],
// and the initial residual r = b - A x (x = xin, copied to xout unless null).
// acc += (b^2, r^2).
// MX: r0 rounded to FP32 into L32.r (instead of L.r), and with a learned guess
// its increment m.x set to zero.
template <bool MX>
__device__ __forceinline__ void ph_helm_rhs_t(const StepArgs &a, const Level &L, const LevelF &L32,
                                              const MixedArgs &m, const double *xin, double *xout, bool guess,
                                              double *sm, int bx, int bz, double (&acc)[2])
{
    const Geom &G = a.G;
    const Phys &F = a.F;
    Tile<1> &sx = tile_at<1>(sm, 0), &s2 = tile_at<1>(sm, 1), &shx = tile_at<1>(sm, 2),
            &shz = tile_at<1>(sm, 3);
    int i, k;
    const bool in = cell_of(G, bx, bz, i, k);
    const int q0 = in ? cidx(G, i, k) : 0;
    // the cell's face coefficients and operator, loaded ahead of the tile
    // barrier
    double Dw = 0.0, De = 0.0, Ds = 0.0, Dn = 0.0;
    HelmCoef<double> hc{};
    auto fetch = [&] {
        Dw = ld(&a.Dx[k * G.P + i]);
        De = ld(&a.Dx[k * G.P + i + 1]);
        Ds = ld(&a.Dz[k * G.P + i]);
        Dn = ld(&a.Dz[(k + 1) * G.P + i]);
        hc = helm_coef(L, q0, i, k);
    };
    if (kPrefetch && in) fetch();
    load_tile_fn<1>(sx, G, bx, bz, [&](int q, int, int) { return ld(&xin[q]); });
    load_tile_fn<1>(s2, G, bx, bz, [&](int q, int, int) { return ld(&a.rho2[q]); });
    load_tile_fn<1>(shx, G, bx, bz, [&](int q, int, int) { return ld(&a.Hx[q]); });
    load_tile_fn<1>(shz, G, bx, bz, [&](int q, int, int) { return ld(&a.Hz[q]); });
    __syncthreads();
    if (in) {
        if (!kPrefetch) fetch();
        const int q = q0;
        const int y = threadIdx.y + 1, x = threadIdx.x + 1;
        const double gx2 = ld(&a.gx2[k]);
        const double r2q = s2[y][x], hxq = shx[y][x], hzq = shz[y][x];
        // twice the face flux over D and the spacing, H_a + H_b + 2 g z_f
        // (rho2_b - rho2_a) / Delta; wall faces have D = 0 and zero tile entries
        // beyond the box
        double fx = De * fma(gx2, s2[y][x + 1] - r2q, hxq + shx[y][x + 1]);
        fx = fma(-Dw, fma(gx2, r2q - s2[y][x - 1], hxq + shx[y][x - 1]), fx);
        double fz = Dn * fma(ld(&a.gz2[k + 1]), s2[y + 1][x] - r2q, hzq + shz[y + 1][x]);
        fz = fma(-Ds, fma(ld(&a.gz2[k]), r2q - s2[y - 1][x], hzq + shz[y - 1][x]), fz);
        const double flux = fma(F.hiz, fz, F.hix * fx);
        const double b = fma(fma(ld(&a.psi[q]) * r2q, ld(&a.gzc[k]), ld(&a.S.rho[q])), F.idt, -flux);
        double r = fma(-hc.d, sx[y][x], b);
        r = fma(hc.aw, sx[y][x - 1], r);
        r = fma(hc.ae, sx[y][x + 1], r);
        r = fma(hc.as, sx[y - 1][x], r);
        r = fma(hc.an, sx[y + 1][x], r);
        a.b[q] = b;
        if (!MX) {
            L.r[q] = r;
            if (xout) xout[q] = sx[y][x];
        } else {
            L32.r[q] = (float)r;
            if (guess) m.x[q] = 0.0f;
        }
        acc[0] = fma(b, b, acc[0]);
        acc[1] = fma(r, r, acc[1]);
    }
    __syncthreads();
}

__device__ __forceinline__ void ph_helm_rhs(const StepArgs &a, const Level &L, const double *xin,
                                            double *xout, double *sm, int bx, int bz,
                                            double (&acc)[2])
{
    ph_helm_rhs_t<false>(a, L, LevelF{}, MixedArgs{}, xin, xout, false, sm, bx, bz, acc);
}

// ---- pressure solve: red-black multigrid CG ----
//
// A cell (i, k) is black if i + k is even, red otherwise; the four neighbours
// of a cell have the other colour, so either colour is relaxed exactly in
// one pass. The solve is the conjugate gradient method preconditioned by a
// V(1,1)-cycle whose smoother is red-black Gauss-Seidel: before the coarse
// correction red then black, after it black then red (symmetric). On the
// finest level the red cells are relaxed before the first iteration. Every
// direction the cycle yields then leaves them relaxed, (A p)_red = 0, so the
// iteration runs on the black half of the vectors alone, with the Schur
// complement S = A_bb - A_br A_rr^-1 A_rb as its operator: the red part of a
// direction is A_rr^-1 A_rb p_b on the fly, the red residual stays zero, and
// the red part of the solution follows at the end from the black one.
//
// Why: FP64 issue bounds these phases. Against full vectors and a damped
// Jacobi smoother (pspmv 7.3, update with pre-smoothing 12, post-smoothing 9
// FP64 instructions per cell and iteration) the black half takes 7.1, 4.8
// and 3, and red-black smoothing contracts better: with the halved coarse
// faces (ph_coarsen) CG takes 9-11 iterations per ten decades where it took
// 14 (4096 x 2048) to 38 (400 x 400 at 2.5 m).
//
// Layout: a black-half array keeps black cell (2 j + (k & 1), k) at k P + j, a
// pair (j, k) being the cells 2 j and 2 j + 1 of row k. With s = k & 1 the
// black cell j of row k has the red neighbours j - 1 + s (west), j + s (east)
// and j (south, north), the red cell j the black ones j - s, j + 1 - s, j and
// j: four-point stencils on the pair grid, without strided access. A tile is
// BX pairs x BZ rows, one pair per thread. A cell beyond an odd nx is zero.

// Pairs of a row.
__host__ __device__ __forceinline__ int pairs_of(const Geom &G) { return (G.nx + 1) >> 1; }

template <int H, class R>
using PairTile = R[BZ + 2 * H][kPW];

template <int H, class R>
__device__ __forceinline__ PairTile<H, R> &pair_tile(double *sm, int at)
{
    return *reinterpret_cast<PairTile<H, R> *>(reinterpret_cast<R *>(sm) + at);
}

// The thread's pair (j, k); false outside the rows and pairs of the level.
// Tiles of fewer rows than BZ (an even number) keep all threads on the halo's
// elements and the first rows of threads on the own ones.
__device__ __forceinline__ bool pair_of(const Geom &G, int bx, int bz, int &j, int &k, int rows = BZ)
{
    j = bx * BX + threadIdx.x;
    k = bz * rows + threadIdx.y;
    return j < pairs_of(G) && k < G.nz && (int)threadIdx.y < rows;
}

// sum of the face coefficients of cell q times its four neighbours' values
template <class R>
__device__ __forceinline__ R faces4(const LevelT<R> &L, int q, R w, R e, R s, R n)
{
    R t = ld(&L.ax[q]) * w;
    t = fma(ld(&L.ax[q + 1]), e, t);
    t = fma(ld(&L.az[q]), s, t);
    return fma(ld(&L.az[q + L.G.P]), n, t);
}

// Fills rows -H .. rows + H - 1 and pairs -1 .. BX of a pair tile with
// f(q, c) at the cells of one colour (RED: the red ones) inside the box
// (q: cell index, c: pair index), zero elsewhere.
template <int H, bool RED, class R, class Fn>
__device__ __forceinline__ void fill_pairs(PairTile<H, R> &t, const Geom &G, int bx, int bz, Fn f, int rows = BZ)
{
    const int tid = threadIdx.x + threadIdx.y * BX;
    for (int e = tid; e < (rows + 2 * H) * kPW; e += NTHREADS) {
        const int tk = e / kPW, tj = e - tk * kPW;
        const int j = bx * BX - 1 + tj, k = bz * rows - H + tk;
        const int i = 2 * j + (RED ? 1 - (k & 1) : (k & 1));
        t[tk][tj] = (j >= 0 && i < G.nx && k >= 0 && k < G.nz) ? (R)f(k * G.P + i, k * G.P + j, j, k) : (R)0;
    }
}

// Same for values f(q, c, tk, tj) that combine the other colour's tile: only
// the BX + 1 pairs of each row that the own cells' stencils reach. The red
// pairs next to the black pairs 0 .. BX - 1 of a row are -1 + s .. BX - 1 + s,
// the black ones next to the red pairs -s .. BX - s (tile columns one more).
template <bool RED, class R, class Fn>
__device__ __forceinline__ void fill_next(PairTile<1, R> &t, const Geom &G, int bx, int bz, Fn f, int rows = BZ)
{
    const int tid = threadIdx.x + threadIdx.y * BX;
    for (int e = tid; e < (rows + 2) * (BX + 1); e += NTHREADS) {
        const int tk = e / (BX + 1);
        const int k = bz * rows - 1 + tk, s = k & 1;
        const int tj = e - tk * (BX + 1) + (RED ? s : 1 - s);
        const int j = bx * BX - 1 + tj;
        const int i = 2 * j + (RED ? 1 - s : s);
        t[tk][tj] = (j >= 0 && i < G.nx && k >= 0 && k < G.nz) ? (R)f(k * G.P + i, k * G.P + j, tk, tj, s) : (R)0;
    }
}

// Coarse residual of the tile's rows from the threads' contributions v (the
// residual of the pair's two cells after pre-smoothing): a quarter of the sum
// over the two pairs of a coarse cell, which has the pair's index.
template <class R>
__device__ __forceinline__ void restrict_pairs(const LevelT<R> &c, R v, R *sres, int bx, int bz, int rows = BZ)
{
    const int tx = threadIdx.x, ty = threadIdx.y;
    sres[ty * BX + tx] = v;
    __syncthreads();
    if (ty < rows / 2) {
        const int I = bx * BX + tx, K = bz * (rows / 2) + ty;
        if (I < c.G.nx && K < c.G.nz)
            c.r[cidx(c.G, I, K)] = (R)0.25 * (sres[2 * ty * BX + tx] + sres[(2 * ty + 1) * BX + tx]);
    }
}

// Start of a solve on the finest level of a one-level hierarchy: the red
// cells relaxed, the black residual that leaves, rb = r_b + sum a (r / d)_red,
// and z = rb / d; acc += rb z.
template <class R>
__device__ __forceinline__ void ph_rb_start(const LevelT<R> &L, R *rb, R *z, double *sm, int bx, int bz, R (&acc)[1])
{
    const Geom &G = L.G;
    PairTile<1, R> &st = pair_tile<1, R>(sm, 0);
    fill_pairs<1, true, R>(st, G, bx, bz, [&](int q, int, int, int) { return ld(&L.wd[q]) * ld(&L.r[q]); });
    __syncthreads();
    int j, k;
    if (pair_of(G, bx, bz, j, k)) {
        const int s = k & 1, i = 2 * j + s;
        if (i < G.nx) {
            const int q = cidx(G, i, k), c = cidx(G, j, k);
            const int y = threadIdx.y + 1, x = threadIdx.x + 1;
            const R g = ld(&L.r[q]) + faces4<R>(L, q, st[y][x - 1 + s], st[y][x + s], st[y - 1][x], st[y + 1][x]);
            const R zv = ld(&L.wd[q]) * g;
            rb[c] = g;
            z[c] = zv;
            acc[0] = fma(g, zv, acc[0]);
        }
    }
    __syncthreads();
}

// Down half of a level's V-cycle: e_r = r / d on red, e_b = w (r + sum a e_r) / d
// on black (w = omega), and the residual that leaves, sum a e_b on red and
// (1 - w) (r + sum a e_r) on black, restricted to level c. FINE (the start of
// a solve on the finest level): the black residual r + sum a e_r goes to rb.
// With w != 1, e_b is kept in f.e for the up half (on the finest level of the
// iteration it follows from rb).
template <bool FINE, class R>
__device__ __forceinline__ void ph_mg_down(const LevelT<R> &f, const LevelT<R> &c, R *rb, const Phys &F, double *sm,
                                           int bx, int bz, int rows = BZ)
{
    const Geom &G = f.G;
    PairTile<2, R> &st = pair_tile<2, R>(sm, 0);
    PairTile<1, R> &se = pair_tile<1, R>(sm, kPH2);
    R *sres = reinterpret_cast<R *>(sm) + kPH2 + kPH1;
    fill_pairs<2, true, R>(st, G, bx, bz, [&](int q, int, int, int) { return ld(&f.wd[q]) * ld(&f.r[q]); }, rows);
    __syncthreads();
    fill_next<false, R>(se, G, bx, bz, [&](int q, int cc, int tk, int tj, int s) {
        const R g = ld(&f.r[q]) + faces4<R>(f, q, st[tk + 1][tj - 1 + s], st[tk + 1][tj + s], st[tk][tj], st[tk + 2][tj]);
        R e = ld(&f.wd[q]) * g;
        const bool own = tk >= 1 && tk <= rows && tj >= 1 && tj <= BX;
        if (FINE && own) rb[cc] = g;
        rarely(F.om_ne1, [&] {
            e *= (R)F.omega;
            if (own && !FINE) f.e[q] = e;
        });
        return e;
    }, rows);
    __syncthreads();
    int j, k;
    R v = 0;
    if (pair_of(G, bx, bz, j, k, rows)) {
        const int s = k & 1, q = cidx(G, 2 * j + 1 - s, k);
        const int y = threadIdx.y + 1, x = threadIdx.x + 1;
        v = faces4<R>(f, q, se[y][x - s], se[y][x + 1 - s], se[y - 1][x], se[y + 1][x]);
        rarely(F.om_ne1, [&] {
            const R gb = ld(&f.d[cidx(G, 2 * j + s, k)]) * se[y][x];   // omega times the black residual
            v = fma((R)((1.0 - F.omega) / F.omega), gb, v);
        });
    }
    restrict_pairs<R>(c, v, sres, bx, bz, rows);
    __syncthreads();
}

// Up half of a level's V-cycle with the coarse correction ec (row pitch Pc;
// null on the coarsest level, whose solve is one symmetric red-black sweep):
// red e = r / d + P ec, black z = (1 - w) (e_b + P ec) + w (r + sum a e) / d with
// e_b of the down half, then red z = (r + sum a z) / d. Writes the whole
// correction. DOT (on the finest level): acc += r z.
template <bool DOT, class R>
__device__ __forceinline__ void ph_mg_up(const LevelT<R> &f, const R *res, const R *ec, int Pc, R *out, const Phys &F,
                                         double *sm, int bx, int bz, R (&acc)[1], int rows = BZ)
{
    const Geom &G = f.G;
    PairTile<2, R> &st = pair_tile<2, R>(sm, 0);
    PairTile<1, R> &sz = pair_tile<1, R>(sm, kPH2);
    fill_pairs<2, true, R>(st, G, bx, bz, [&](int q, int, int jj, int kk) {
        const R r = ld(&res[q]), w = ld(&f.wd[q]);
        return ec ? fma(w, r, ld(&ec[(kk >> 1) * Pc + jj])) : w * r;
    }, rows);
    __syncthreads();
    fill_next<false, R>(sz, G, bx, bz, [&](int q, int, int tk, int tj, int s) {
        const R r = ld(&res[q]);
        R z = ld(&f.wd[q]) *
              (r + faces4<R>(f, q, st[tk + 1][tj - 1 + s], st[tk + 1][tj + s], st[tk][tj], st[tk + 2][tj]));
        // the coarsest level keeps no down half: its one sweep is undamped
        rarely(F.om_ne1 && ec, [&] {
            z = fma((R)F.omega, z,
                    (R)(1.0 - F.omega) * (ld(&f.e[q]) + ld(&ec[((bz * rows - 1 + tk) >> 1) * Pc + bx * BX - 1 + tj])));
        });
        if (tk >= 1 && tk <= rows && tj >= 1 && tj <= BX) {
            out[q] = z;
            if (DOT) acc[0] = fma(r, z, acc[0]);
        }
        return z;
    }, rows);
    __syncthreads();
    int j, k;
    if (pair_of(G, bx, bz, j, k, rows)) {
        const int s = k & 1, i = 2 * j + 1 - s;
        if (i < G.nx) {
            const int q = cidx(G, i, k);
            const int y = threadIdx.y + 1, x = threadIdx.x + 1;
            const R r = ld(&res[q]);
            const R z = ld(&f.wd[q]) * (r + faces4<R>(f, q, sz[y][x - s], sz[y][x + 1 - s], sz[y - 1][x], sz[y + 1][x]));
            out[q] = z;
            if (DOT) acc[0] = fma(r, z, acc[0]);
        }
    }
    __syncthreads();
}

// Up half on the finest level of the black-half iteration (red residual
// zero): z = (1 - w) (w rb / d + P ec) + w (rb + sum a P ec) / d, pair by pair;
// acc += rb z.
template <class R>
__device__ __forceinline__ void ph_rb_up(const LevelT<R> &f, const R *rb, const R *ec, int Pc, R *z, const Phys &F,
                                         int bx, int bz, R (&acc)[1])
{
    const Geom &G = f.G;
    int j, k;
    if (!pair_of(G, bx, bz, j, k)) return;
    const int s = k & 1, q = cidx(G, 2 * j + s, k), c = cidx(G, j, k);
    // coarse values of the red neighbours; a neighbour beyond a wall meets a
    // zero coefficient, its index only stays inside the level
    const int jw = max(j - 1 + s, 0), je = min(j + s, pairs_of(G) - 1);
    const R *row = ec + (k >> 1) * Pc;
    const R *rs = ec + (max(k - 1, 0) >> 1) * Pc, *rn = ec + (min(k + 1, G.nz - 1) >> 1) * Pc;
    const R r = ld(&rb[c]), w = ld(&f.wd[q]);
    R zv = w * (r + faces4<R>(f, q, ld(&row[jw]), ld(&row[je]), ld(&rs[j]), ld(&rn[j])));
    rarely(F.om_ne1, [&] { zv = fma((R)F.omega, zv, (R)(1.0 - F.omega) * fma((R)F.omega * w, r, ld(&row[j]))); });
    z[c] = zv;
    acc[0] = fma(r, zv, acc[0]);
}

// ---- CG vector steps (black halves) ----

// p_new = z + beta p_old (first: z) and q = S p_new, with the red part of the
// direction formed on the tile; acc += p.q.
template <class R>
__device__ __forceinline__ void ph_pspmv(const LevelT<R> &L, const R *z, const R *pold, R *pnew, R *qv, double beta,
                                         bool first, double *sm, int bx, int bz, R (&acc)[1])
{
    const Geom &G = L.G;
    const R b = (R)beta;
    PairTile<2, R> &sp = pair_tile<2, R>(sm, 0);
    PairTile<1, R> &sw = pair_tile<1, R>(sm, kPH2);
    int j, k;
    const bool own = pair_of(G, bx, bz, j, k);
    const int s = k & 1, i = 2 * j + s;
    const bool in = own && i < G.nx;
    const int q = in ? cidx(G, i, k) : 0;
    HelmCoef<R> h{};
    if (kPrefetchSpmv && in) h = helm_coef(L, q, i, k);
    if (first)
        fill_pairs<2, false, R>(sp, G, bx, bz, [&](int, int c, int, int) { return ld(&z[c]); });
    else
        fill_pairs<2, false, R>(sp, G, bx, bz, [&](int, int c, int, int) { return fma(b, ld(&pold[c]), ld(&z[c])); });
    __syncthreads();
    fill_next<true, R>(sw, G, bx, bz, [&](int qr, int, int tk, int tj, int sr) {
        return ld(&L.wd[qr]) *
               faces4<R>(L, qr, sp[tk + 1][tj - sr], sp[tk + 1][tj + 1 - sr], sp[tk][tj], sp[tk + 2][tj]);
    });
    __syncthreads();
    if (in) {
        if (!kPrefetchSpmv) h = helm_coef(L, q, i, k);
        const int y = threadIdx.y + 1, x = threadIdx.x + 1, c = cidx(G, j, k);
        const R p = sp[y + 1][x];
        R t = h.d * p;
        t = fma(-h.aw, sw[y][x - 1 + s], t);
        t = fma(-h.ae, sw[y][x + s], t);
        t = fma(-h.as, sw[y - 1][x], t);
        t = fma(-h.an, sw[y + 1][x], t);
        pnew[c] = p;
        qv[c] = t;
        acc[0] = fma(p, t, acc[0]);
    }
    __syncthreads();
}

// One-level hierarchy: x += alpha p, rb -= alpha q and z = rb / d, cell by
// cell; acc += (rb^2, rb z).
template <class R>
__device__ __forceinline__ void ph_update_single(const LevelT<R> &L, const R *qv, R *rb, R *z, R *x, const R *p,
                                                 double alpha_d, bool first, int bx, int bz, R (&acc)[2])
{
    const Geom &G = L.G;
    const R alpha = (R)alpha_d;
    int j, k;
    if (!pair_of(G, bx, bz, j, k)) return;
    const int i = 2 * j + (k & 1);
    if (i >= G.nx) return;
    const int c = cidx(G, j, k);
    const R pq = ld(&p[c]);
    x[c] = fma(alpha, pq, first ? (R)0 : ld(&x[c]));
    const R rn = fma(-alpha, ld(&qv[c]), ld(&rb[c]));
    rb[c] = rn;
    const R zv = ld(&L.wd[cidx(G, i, k)]) * rn;
    z[c] = zv;
    acc[0] = fma(rn, rn, acc[0]);
    acc[1] = fma(rn, zv, acc[1]);
}

// Multigrid: x += alpha p and rb -= alpha q, fused with the down half of the
// finest level (a CG iteration then needs one grid-wide synchronisation
// less): e = w rb / d on the black cells and the residual that leaves, sum a e on
// red (and (1 - w) rb on black), restricted to level c. The residual is read
// from rin (halo included) and written to rout: other blocks still read the
// old one. acc += rb^2.
template <class R>
__device__ __forceinline__ void ph_update_down(const LevelT<R> &f, const LevelT<R> &c, const R *qv, const R *rin,
                                               R *rout, R *x, const R *p, double alpha_d, bool first, const Phys &F,
                                               double *sm, int bx, int bz, R (&acc)[1])
{
    const Geom &G = f.G;
    const R alpha = (R)alpha_d;
    PairTile<1, R> &se = pair_tile<1, R>(sm, 0);
    R *sres = reinterpret_cast<R *>(sm) + kPH1;
    fill_next<false, R>(se, G, bx, bz, [&](int q, int cc, int tk, int tj, int) {
        const R rn = fma(-alpha, ld(&qv[cc]), ld(&rin[cc]));
        if (tk >= 1 && tk <= BZ && tj >= 1 && tj <= BX) {
            rout[cc] = rn;
            const R pq = ld(&p[cc]);
            x[cc] = fma(alpha, pq, first ? (R)0 : ld(&x[cc]));
            acc[0] = fma(rn, rn, acc[0]);
        }
        return ld(&f.wd[q]) * rn;
    });
    __syncthreads();
    int j, k;
    R v = 0;
    if (pair_of(G, bx, bz, j, k)) {
        const int s = k & 1, q = cidx(G, 2 * j + 1 - s, k);
        const int y = threadIdx.y + 1, xx = threadIdx.x + 1;
        v = faces4<R>(f, q, se[y][xx - s], se[y][xx + 1 - s], se[y - 1][xx], se[y + 1][xx]);
        rarely(F.om_ne1,
               [&] { v = fma((R)F.omega, v, (R)(1.0 - F.omega) * ld(&f.d[cidx(G, 2 * j + s, k)]) * se[y][xx]); });
    }
    restrict_pairs<R>(c, v, sres, bx, bz);
    __syncthreads();
}

// ---- learned initial guess of a pressure solve ----

// The network's proposal e (dense FP32, row k at k nx): q = A e and
// acc += (r . e, e . A e).
template <class R>
__device__ __forceinline__ void ph_guess_dots(const LevelT<R> &L, const float *e, const R *r, R *q, double *sm,
                                              int bx, int bz, R (&acc)[2])
{
    const Geom &G = L.G;
    Tile<1, R> &se = tile_at<1, R>(sm, 0);
    load_tile_fn<1, R>(se, G, bx, bz, [&](int, int i, int k) { return (R)ld(&e[(size_t)k * G.nx + i]); });
    __syncthreads();
    int i, k;
    if (cell_of(G, bx, bz, i, k)) {
        const int qi = cidx(G, i, k);
        const int y = threadIdx.y + 1, x = threadIdx.x + 1;
        const R Ae = helm_tile<1, R>(L, qi, i, k, se, y, x);
        q[qi] = Ae;
        acc[0] = fma(ld(&r[qi]), se[y][x], acc[0]);
        acc[1] = fma(se[y][x], Ae, acc[1]);
    }
    __syncthreads();
}

// x += alpha e, r -= alpha q; acc += r^2.
template <class R>
__device__ __forceinline__ void ph_guess_apply(const LevelT<R> &L, const float *e, const R *q, R *r, R *x,
                                               double alpha_d, int bx, int bz, R (&acc)[1])
{
    int i, k;
    if (!cell_of(L.G, bx, bz, i, k)) return;
    const int qi = cidx(L.G, i, k);
    const R alpha = (R)alpha_d;
    x[qi] = fma(alpha, (R)ld(&e[(size_t)k * L.G.nx + i]), ld(&x[qi]));
    const R rn = fma(-alpha, ld(&q[qi]), ld(&r[qi]));
    r[qi] = rn;
    acc[0] = fma(rn, rn, acc[0]);
}

// p' on the tile and its one-cell halo. sd: scratch of a halo-2 tile.
template <class R>
__device__ __forceinline__ void load_solution(Tile<1> &sx, Tile<2, R> &sd, const LevelT<R> &L, const SolveT<R> &v,
                                              bool dx, int bx, int bz)
{
    const Geom &G = L.G;
    const int i0 = bx * BX, k0 = bz * BZ;
    auto start = [&](int q) {
        double x = ld(&v.x[q]);
        if (v.inc) x += (double)ld(&v.inc[q]);
        return x;
    };
    if (!dx) {
        load_tile_fn<1>(sx, G, bx, bz, [&](int q, int, int) { return start(q); });
        return;
    }
    const int tid = threadIdx.x + threadIdx.y * BX;
    constexpr int NJ = BX / 2 + 2;   // pairs that cover the halo: tile columns -2 .. BX + 1
    for (int e = tid; e < (BZ + 4) * NJ; e += NTHREADS) {
        const int tk = e / NJ, tj = e - tk * NJ;
        const int j = i0 / 2 - 1 + tj, k = k0 - 2 + tk, s = k & 1, i = 2 * j + s;
        sd[tk][2 * tj + s] = (j >= 0 && i < G.nx && k >= 0 && k < G.nz) ? ld(&v.xb[k * G.P + j]) : (R)0;
    }
    __syncthreads();
    for (int e = tid; e < (BZ + 2) * NJ; e += NTHREADS) {
        const int tk = e / NJ, tj = e - tk * NJ;
        const int j = i0 / 2 - 1 + tj, k = k0 - 1 + tk, s = k & 1;
        const bool zin = k >= 0 && k < G.nz && j >= 0;
        const int cb = 2 * tj + s, cr = 2 * tj + 1 - s;   // halo-2 tile columns of the pair's cells
        if (cb >= 1 && cb <= BX + 2)
            sx[tk][cb - 1] = zin && 2 * j + s < G.nx ? start(k * G.P + 2 * j + s) + (double)sd[tk + 1][cb] : 0.0;
        if (cr >= 1 && cr <= BX + 2) {
            double xv = 0.0;
            if (zin && 2 * j + 1 - s < G.nx) {
                const int q = k * G.P + 2 * j + 1 - s;
                const R t = ld(&L.r[q]) + faces4<R>(L, q, sd[tk + 1][cr - 1], sd[tk + 1][cr + 1], sd[tk][cr], sd[tk + 2][cr]);
                xv = start(q) + (double)(ld(&L.wd[q]) * t);
            }
            sx[tk][cr - 1] = xv;
        }
    }
}

// The solution of the pressure solve, and the flux and velocity correction:
// F_f = D_f (H_f - G_f) with
// G_f = (p'_b - p'_a)/Delta - g z_f (rho2_b - rho2_a)/Delta; u = (dt/rho1)(H - G_cell);
// p = p' - rho2 g z; rho = p / (R T^{n+1}) = p psi; phi = F |A|; p^{n-1} <- p^n
// (and K^{n-1} <- K^n in the literal reading of eq. step3_sd). p' goes to ppout
// (not the solve's start, which other blocks still read).
template <class R>
__device__ __forceinline__ void ph_correct(const StepArgs &a, const LevelT<R> &L, const SolveT<R> &v, bool dx,
                                           double *ppout, double *sm, int bx, int bz)
{
    const Geom &G = a.G;
    const Phys &F = a.F;
    Tile<1> &sx = tile_at<1>(sm, 0), &s2 = tile_at<1>(sm, 1);
    double(*gx)[BX + 1] = reinterpret_cast<double(*)[BX + 1]>(sm + 2 * kT1);
    double(*gz)[BX] = reinterpret_cast<double(*)[BX]>(sm + 2 * kT1 + BZ * (BX + 1));
    const State &N = a.N;
    int i, k;
    const bool in = cell_of(G, bx, bz, i, k);
    const int q0 = in ? cidx(G, i, k) : 0;
    // the cell's own inputs, loaded ahead of the tile barrier: H(u) at the
    // cell and at its west and south neighbours (the face averages), D on
    // the west and south faces, dt/rho1, psi, p^n
    double hxq = 0.0, hzq = 0.0, hxw = 0.0, hzs = 0.0, Dw = 0.0, Ds = 0.0, dtr1 = 0.0, psq = 0.0, pnq = 0.0;
    auto fetch = [&] {
        hxq = ld(&a.Hx[q0]);
        hzq = ld(&a.Hz[q0]);
        if (i > 0) {
            hxw = ld(&a.Hx[q0 - 1]);
            Dw = ld(&a.Dx[k * G.P + i]);
        }
        if (k > 0) {
            hzs = ld(&a.Hz[q0 - G.P]);
            Ds = ld(&a.Dz[k * G.P + i]);
        }
        dtr1 = ld(&a.dtr1[q0]);
        psq = ld(&a.psi[q0]);
        pnq = ld(&a.S.p[q0]);
    };
    if (kPrefetch && in) fetch();
    load_tile_fn<1>(s2, G, bx, bz, [&](int q, int, int) { return ld(&a.rho2[q]); });
    // the scratch lies where the face forces go after the barrier
    load_solution<R>(sx, tile_at<2, R>(sm + 2 * kT1, 0), L, v, dx, bx, bz);
    __syncthreads();
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int y = ty + 1, x = tx + 1;
    const double gzk = in ? ld(&a.gzc[k]) : 0.0;
    // Delta G_f
    auto gxf = [&](int xa) {   // x-face between tile columns xa and xa+1 of row y
        return fma(-gzk, s2[y][xa + 1] - s2[y][xa], sx[y][xa + 1] - sx[y][xa]);
    };
    auto gzf = [&](int ya, int kf) {   // z-face between tile rows ya and ya+1, face index kf
        return fma(-ld(&a.gzf[kf]), s2[ya + 1][x] - s2[ya][x], sx[ya + 1][x] - sx[ya][x]);
    };
    if (in) {
        gx[ty][tx] = i > 0 ? gxf(x - 1) : 0.0;
        gz[ty][tx] = k > 0 ? gzf(y - 1, k) : 0.0;
        if (tx == BX - 1 || i == G.nx - 1) gx[ty][tx + 1] = i + 1 < G.nx ? gxf(x) : 0.0;
        if (ty == BZ - 1 || k == G.nz - 1) gz[ty + 1][tx] = k + 1 < G.nz ? gzf(y, k + 1) : 0.0;
    }
    __syncthreads();
    if (in) {
        if (!kPrefetch) fetch();
        const int q = q0;
        const double gxw = gx[ty][tx], gxe = gx[ty][tx + 1], gzs = gz[ty][tx], gzn = gz[ty + 1][tx];
        // F |A| = D (|A| / 2) (H_a + H_b - 2 G); wall faces have D = 0 here
        N.phix[k * G.P + i] = (Dw * F.hdz) * fma(-F.tix, gxw, hxw + hxq);
        N.phiz[k * G.P + i] = (Ds * F.hdx) * fma(-F.tiz, gzs, hzs + hzq);
        if (i == G.nx - 1) N.phix[k * G.P + G.nx] = 0.0;
        if (k == G.nz - 1) N.phiz[G.nz * G.P + i] = 0.0;
        N.u[q] = dtr1 * fma(-F.hix, gxw + gxe, hxq);
        N.w[q] = dtr1 * fma(-F.hiz, gzs + gzn, hzq);
        ppout[q] = sx[y][x];
        const double pn = fma(-s2[y][x], gzk, sx[y][x]);
        N.p[q] = pn;
        N.rho[q] = pn * psq;
        N.pold[q] = pnq;
        rarely(F.k_lagged, [&] {
            const double un = ld(&a.S.u[q]), wn = ld(&a.S.w[q]);
            N.Kold[q] = 0.5 * fma(un, un, wn * wn);   // K^{n-1} of the next step
        });
    }
    __syncthreads();
}

// ---- what the block that completes a reduction does with the totals ----

__device__ __forceinline__ void fin_pred(Scal *sc, const double (&t)[2])
{
    sc->bn2[0] = t[0];
    sc->bn2[1] = t[1];
    sc->done[LOOP_MOM] = 0;
    sc->trips[LOOP_MOM] = 0;
    sc->sweeps[0] = 0;
}

__device__ __forceinline__ void fin_mom(Scal *sc, const double (&t)[2], double tol2)
{
    sc->sweeps[0] += 1;
    if (!isfinite(t[0]) || !isfinite(t[1])) sc->status = 5;
    else if (t[0] <= tol2 * sc->bn2[0] && t[1] <= tol2 * sc->bn2[1]) sc->done[LOOP_MOM] = 1;
}

__device__ __forceinline__ void fin_enth_rhs(Scal *sc, const double (&t)[1])
{
    sc->bn2[2] = t[0];
    sc->done[LOOP_ENTH] = 0;
    sc->trips[LOOP_ENTH] = 0;
    sc->sweeps[1] = 0;
}

__device__ __forceinline__ void fin_enth(Scal *sc, const double (&t)[1], double tol2)
{
    sc->sweeps[1] += 1;
    if (!isfinite(t[0])) sc->status = 5;
    else if (t[0] <= tol2 * sc->bn2[2]) sc->done[LOOP_ENTH] = 1;
}

__device__ __forceinline__ void fin_helm(Scal *sc, const double (&t)[2], double tol2, int corr)
{
    sc->b2 = t[0];
    sc->r2 = t[1];
    sc->cg_it = 0;
    sc->corr = corr;
    sc->trips[LOOP_CG] = 0;
    sc->rz = 0.0;
    sc->beta = 0.0;
    sc->done[LOOP_CG] = t[1] <= tol2 * t[0];
    sc->cg_iters[corr] = 0;
    sc->cg_r2[corr] = t[1];
    sc->cg_b2[corr] = t[0];
    if (!isfinite(t[0]) || !isfinite(t[1])) sc->status = 5;
}

// Mixed precision: the inner FP32 solve's tolerance is relative to the
// initial residual r0 = b - A p'_prev (kept in b2); nothing to solve if r0 is
// already at the FP64 tolerance relative to b.
__device__ __forceinline__ void fin_helm_mixed(Scal *sc, const double (&t)[2], double tol2_fp64, int corr)
{
    sc->b2 = t[1];
    sc->r2 = t[1];
    sc->cg_it = 0;
    sc->corr = corr;
    sc->trips[LOOP_CG] = 0;
    sc->rz = 0.0;
    sc->beta = 0.0;
    sc->done[LOOP_CG] = t[1] <= tol2_fp64 * t[0];
    sc->cg_iters[corr] = 0;
    sc->cg_r2[corr] = sc->cg_b2[corr] = t[1] > 0.0 ? t[1] : 1.0;
    if (!isfinite(t[0]) || !isfinite(t[1])) sc->status = GEA_ERR_NONFINITE;
}

__device__ __forceinline__ void fin_rz(Scal *sc, const double (&t)[1])
{
    sc->beta = (sc->cg_it == 0 || sc->rz == 0.0) ? 0.0 : t[0] / sc->rz;
    sc->rz = t[0];
}

__device__ __forceinline__ void fin_pq(Scal *sc, const double (&t)[1])
{
    sc->pq = t[0];
    sc->alpha = t[0] != 0.0 ? sc->rz / t[0] : 0.0;
    if (!isfinite(t[0])) sc->status = 5;
}

__device__ __forceinline__ void fin_update(Scal *sc, const double (&t)[1], double tol2)
{
    const int it = sc->cg_it + 1;
    sc->cg_it = it;
    sc->r2 = t[0];
    const int c = sc->corr;
    sc->cg_iters[c] = it;
    sc->cg_r2[c] = t[0];
    sc->cg_b2[c] = sc->b2;
    if (!isfinite(t[0])) sc->status = 5;
    else if (t[0] <= tol2 * sc->b2) sc->done[LOOP_CG] = 1;
}

// the step length minimising the A-norm error along e: alpha = r.e / e.Ae
// (0 if e.Ae is not positive)
__device__ __forceinline__ void fin_guess_dots(Scal *sc, const double (&t)[2])
{
    sc->galpha = (t[1] > 0.0 && isfinite(t[0]) && isfinite(t[1])) ? t[0] / t[1] : 0.0;
}

__device__ __forceinline__ void fin_guess_apply(Scal *sc, const double (&t)[1], double tol2)
{
    sc->r2 = t[0];
    sc->cg_r2[sc->corr] = t[0];
    sc->cg_b2[sc->corr] = sc->b2;
    if (!isfinite(t[0])) sc->status = GEA_ERR_NONFINITE;
    else if (t[0] <= tol2 * sc->b2) sc->done[LOOP_CG] = 1;
}
