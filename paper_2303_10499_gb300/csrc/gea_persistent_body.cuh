// gea_persistent_body.cuh -- n time steps of the GEA pressure-based Euler
// solver (Girfoglio, Quaini & Rozza, arXiv 2303.10499, Section 3) as one
// cooperative kernel.
//
// A step is a chain of 30 to several hundred phases. On small grids launching
// each as its own kernel leaves the GPU waiting on launch latency, and up to
// nearly two million cells (16 tiles a block; FP32 phases half of that) the
// launches and the gaps between them still cost more than the blocks in flight
// that this kernel gives up. Here the blocks stay resident for the whole step: each
// phase is a block-stride loop over tiles running the tile functions of
// gea_tiles_body.cuh, phases are separated by a grid barrier, and every
// residual norm or CG dot product rides on the barrier: each block writes its
// partial before arriving and, once released, adds all the partials itself
// in a fixed order. The Jacobi and CG loops run inside the kernel; every
// block takes the same decisions because it computes the same totals, bit
// for bit, and updates its own copy of the loop scalars with them.
//
// The barrier waits spin on an acquire load with an iteration cap; a block
// that gives up sets GEA_ERR_TIMEOUT in the context status, and every block
// leaves the step at its next phase boundary when the status is set, so the
// kernel always ends.
//
// Like the tile functions, this file is included once per tile shape, inside
// that shape's namespace and after its tile functions (gea_persistent.cu:
// 32 x 8; gea_persistent_16x16.cu, gea_persistent_64x4.cu): the kernels run
// one thread per cell of a BX x BZ tile, and the shape's host entry points
// are collected in `ops` (PersistOps, gea_internal.cuh).

namespace {

// values per thread a grid reduction may carry: the block-sum scratch after
// the tile area holds kRedVals x NTHREADS doubles
constexpr int kRedVals = 4;
// Blocks up to which one warp per value adds a grid reduction's partials. FP64 us
// a step, one warp / all threads: 32 blocks 587 / 608, 50 blocks 562 / 576, 64 blocks
// 593 / 606, 80 blocks 588 / 586, 100 blocks 615 / 590, 120 blocks 614 / 584 (128, where
// no lane has a partial more than another, 581 / 592): with two partials a
// lane and fewer the pass through shared memory costs more than the loads.
constexpr int kDirectPartials = 64;

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Arrival with acquire-release semantics: publishes this block's writes of
// the phase (ordered before it by the block barrier) and observes those of
// the blocks that arrived earlier.
__device__ __forceinline__ unsigned atom_add_acq_rel(unsigned *p, unsigned v)
{
    unsigned old;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}


__device__ __forceinline__ int rdi(const int *p) { return __ldcg(p); }

__device__ __forceinline__ unsigned long long globaltimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ int tid_of() { return threadIdx.x + threadIdx.y * BX; }

// The blocks that run one context's steps: this block's rank among them and
// their number (the whole grid for one context; a contiguous share of the
// grid per member in an ensemble launch), and the block's count of the
// barriers it has passed in this launch (shared memory; every block passes
// the same barriers).
struct Grp {
    int rank, nb;
    unsigned *gen;   // barriers this block has passed in this launch
    Scal *gs;        // the context's scalars in global memory (barrier words, status, results)
    unsigned long long spin_limit;   // polls of a barrier before the block gives up
    unsigned long long *trace;       // phase trace (null: off), see trace_entry
    int trace_bars;                  // barriers the trace holds
};

// Phase trace layout: 2 x nb values per row; row 0 holds each block's
// kernel entry time and SM, row k >= 1 each block's arrival at and release
// from the k-th grid barrier of the launch (%globaltimer, ns).
__device__ __forceinline__ void trace_entry(const Grp &g)
{
    if (g.trace && tid_of() == 0) {
        unsigned smid;
        asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
        g.trace[2 * (size_t)g.rank] = globaltimer();
        g.trace[2 * (size_t)g.rank + 1] = smid;
    }
}

// The block's own copy of the context's scalars. Every block finishes every
// grid reduction itself (the same partials added in the same order give
// every block the same totals, bit for bit) and applies the same update to
// its copy, so the loop decisions (convergence flags, iteration counts, CG
// step lengths) are taken from shared memory, identically in every block.
// Block rank 0 publishes what the host reads.
__shared__ Scal s_ctl;

// Block-uniform stop flag, set by thread 0 at kernel entry and at the end of
// every grid barrier (the context's status, or an error of the block's own
// reductions), so that all threads of a block leave a step at the same
// phase boundary.
__shared__ int s_stop;

// Copy the context's scalars into the block's copy (all threads; kernel entry).
__device__ __forceinline__ void load_ctl(const Scal *gs)
{
    static_assert(sizeof(Scal) % 4 == 0, "Scal is copied as 32-bit words");
    const int *src = reinterpret_cast<const int *>(gs);
    int *dst = reinterpret_cast<int *>(&s_ctl);
    for (int w = tid_of(); w < (int)(sizeof(Scal) / 4); w += NTHREADS) dst[w] = __ldcg(&src[w]);
}

// Grid barrier on a monotone arrival counter: barrier k of a launch is
// passed once the counter reaches 2 k x (blocks), so the last block to arrive
// releases the others by its arrival alone. A block arrives with one
// acquire-release add (thread 0, after the block barrier: it publishes the
// block's writes of the phase) and polls the counter with acquire loads
// (the adds form one release sequence, so reading the final count acquires
// every block's writes). Every data read across blocks goes through L2
// (ld.global.cg), ordered after the acquire by the block barrier. The count
// wraps modulo 2^32; the comparison is of the signed difference.
// A block that gives up sets the context's status and the counter's lowest
// bit; the others see the bit in the word they poll anyway, at this barrier or
// the next (a read of the status word after every barrier cost 0.2 us).
__device__ __forceinline__ void gbar(const Grp &g)
{
    Scal *gs = g.gs;
    __syncthreads();
    if (tid_of() == 0) {
        const unsigned k = *g.gen + 1u;
        const unsigned target = 2u * k * (unsigned)g.nb;
        unsigned long long *tr =
            (g.trace && k <= (unsigned)g.trace_bars) ? g.trace + 2 * ((size_t)k * g.nb + g.rank) : nullptr;
        if (tr) tr[0] = globaltimer();
        unsigned c = atom_add_acq_rel(&gs->bar_count, 2u) + 2u;
        unsigned long long spins = 0;
        while ((int)((c & ~1u) - target) < 0 && !(c & 1u)) {
            if (spins++ >= g.spin_limit) {
                atomicCAS(&gs->status, 0, GEA_ERR_TIMEOUT);
                __threadfence();   // whoever sees the bit sees the status
                atomicOr(&gs->bar_count, 1u);
                c |= 1u;
                break;
            }
            c = ld_acquire(&gs->bar_count);
        }
        if (tr) tr[1] = globaltimer();
        *g.gen = k;
        s_stop = (c & 1u) != 0 || s_ctl.status != 0;
    }
    __syncthreads();
}

// Every block leaves through here (all threads): the last of the launch's
// blocks to leave sets the arrival counter back to zero for the next launch
// (no block of this launch arrives again).
__device__ __forceinline__ void leave(const Grp &g)
{
    __syncthreads();
    if (tid_of() == 0 && atom_add_acq_rel(&g.gs->bar_exit, 1u) == (unsigned)g.nb - 1u) {
        g.gs->bar_count = 0u;
        g.gs->bar_exit = 0u;
    }
}

// Barrier with a deterministic grid-wide sum of NV per-thread values, which
// every block completes: it adds the block partials in a fixed order and
// thread 0 runs fin(tot) on the block's copy of the scalars. T is the type
// of the per-thread values and of the block sums (FP32 for the inner solves
// of the mixed-precision step); block partials and the total are FP64. The
// partials alternate between two buffers by barrier parity: a block
// writes a buffer again only two barriers later, after every block has read
// it.
template <int NV, class T, class Fin>
__device__ __forceinline__ void rbar(const Grp &g, const T (&v)[NV], double *red, double *partials, Fin fin)
{
    static_assert(NV <= kRedVals, "the block-sum scratch holds kRedVals values per thread");
    const int tid = tid_of();
    const int nb = g.nb;
    double *pb = partials + kGcntDoubles + (size_t)(*g.gen & 1u) * kRedVals * nb;
    T bt[NV];
    block_sum<NV, T>(v, reinterpret_cast<T *>(red), bt);
    if (tid == 0) {
#pragma unroll
        for (int j = 0; j < NV; ++j) pb[(size_t)j * nb + g.rank] = (double)bt[j];
    }
    gbar(g);
    double tot[NV];
    if (nb <= kDirectPartials) {
        // few blocks: warp j adds the partials of value j at once, without the
        // pass through shared memory (two per lane and the shuffle tree)
        const int lane = tid & 31;
        for (int j = tid / 32; j < NV; j += NTHREADS / 32) {
            double s = 0.0;
            for (int b = lane; b < nb; b += 32) {
                const double v = __ldcg(&pb[(size_t)j * nb + b]);
                s = b == lane ? v : s + v;
            }
            s = warp_sum(s);
            if (lane == 0) red[j] = s;
        }
        if (NV > 1) __syncthreads();
        if (tid == 0) {
#pragma unroll
            for (int j = 0; j < NV; ++j) tot[j] = red[j];
        }
    } else {
        double s[NV];
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            s[j] = 0.0;
            for (int b = tid; b < nb; b += NTHREADS) {
                const double v = __ldcg(&pb[(size_t)j * nb + b]);
                s[j] = b == tid ? v : s[j] + v;
            }
        }
        block_sum<NV>(s, red, tot);
    }
    if (tid == 0) {
        fin(tot);
        if (s_ctl.status) {
            s_stop = 1;
            if (g.rank == 0) atomicCAS(&g.gs->status, 0, s_ctl.status);
        }
    }
    __syncthreads();
}

template <class F>
__device__ __forceinline__ void for_tiles(const Grp &g, const Geom &G, F f)
{
    const int tx = (G.nx + BX - 1) / BX, tz = (G.nz + BZ - 1) / BZ;
    const int nt = tx * tz;
    for (int t = g.rank; t < nt; t += g.nb) f(t % tx, t / tx);
}

// the tiles of the red-black phases: BX pairs of cells wide
template <class F>
__device__ __forceinline__ void for_pair_tiles(const Grp &g, const Geom &G, F f, int rows = BZ)
{
    const int tx = (pairs_of(G) + BX - 1) / BX, tz = (G.nz + rows - 1) / rows;
    const int nt = tx * tz;
    for (int t = g.rank; t < nt; t += g.nb) f(t % tx, t / tx);
}

// A thread's sums over the tiles its block walks: a phase function adds one
// tile's values. In FP32 (the inner solves of the mixed-precision step) each
// tile's sums are added with the error of the addition kept beside the total,
// so that the sums are as good with many tiles a block (8 by the driver rule,
// hundreds for a large member of an ensemble on one block) as with one. FP32
// additions are next to free here: 640 x 320 349 -> 350 us a step, 36-member
// ensemble 4321 -> 4321, 1001 x 503 0.6 %.
template <class R, int NV>
struct TileSums {
    R v[NV] = {};
    template <class F>
    __device__ __forceinline__ void add(F f) { f(v); }
    __device__ __forceinline__ const R (&total())[NV] { return v; }
};
template <int NV>
struct TileSums<float, NV> {
    float v[NV] = {}, lost[NV] = {};
    template <class F>
    __device__ __forceinline__ void add(F f)
    {
        float t[NV] = {};
        f(t);
#pragma unroll
        for (int j = 0; j < NV; ++j) {   // Knuth's two-sum
            const float s = v[j] + t[j], b = s - v[j];
            lost[j] += (v[j] - (s - b)) + (t[j] - b);
            v[j] = s;
        }
    }
    __device__ __forceinline__ const float (&total())[NV]
    {
#pragma unroll
        for (int j = 0; j < NV; ++j) v[j] += lost[j];
        return v;
    }
};

// Rows of a coarse level's tiles: two where the blocks have at most one such
// tile each, else BZ. A phase of a coarse level lasts as long as its slowest
// block: with two rows the halo and the next colour's elements fit the threads
// in one round each instead of two, and a quarter of the warps share the SM's
// FP64 units. Five-level 400 x 400: 1831 us a step with 8 rows, 1700 with 4, 1657
// with 2; four-level 200 x 200: 1066, 973, 936. With more tiles than blocks the
// halos cost more than that. The rows are a run-time number: as a template
// argument the second copy of the cycle took registers from the single-level
// solve (640 x 320 0.8 % slower).
__device__ __forceinline__ int coarse_rows(const Grp &g, const Geom &G)
{
    return (pairs_of(G) + BX - 1) / BX * ((G.nz + 1) / 2) <= g.nb ? 2 : BZ;
}

__device__ __forceinline__ bool stop(const Scal *) { return s_stop != 0; }

// End of a step: its counters into the block's copy and, from block rank 0,
// into the context (what the host reads).
__device__ __forceinline__ void end_step(const Grp &g)
{
    gbar(g);
    if (tid_of() == 0 && !s_stop) {
        Scal &c = s_ctl;
        c.steps_done += 1;
        c.last_sweeps[0] = c.sweeps[0];
        c.last_sweeps[1] = c.sweeps[1];
        for (int k = 0; k < 4; ++k) {
            c.last_cg_iters[k] = c.cg_iters[k];
            if (g.rank == 0) c.last_cg_relres[k] = cg_relres(c, k);
        }
        c.last_status = 0;
        if (g.rank == 0) {
            Scal *gs = g.gs;
            gs->steps_done = c.steps_done;
            gs->last_sweeps[0] = c.last_sweeps[0];
            gs->last_sweeps[1] = c.last_sweeps[1];
            for (int k = 0; k < 4; ++k) {
                gs->last_cg_iters[k] = c.last_cg_iters[k];
                gs->last_cg_relres[k] = c.last_cg_relres[k];
            }
            gs->last_status = 0;
            gs->press_ns = c.press_ns;
        }
    }
}

// The pressure solve from the residual L[0].r (gea_tiles_body.cuh: red-black
// multigrid CG) to the relative residual tol2 (squared), after fin_helm; the
// increment is left in v.x.
template <class R>
__device__ __forceinline__ void pressure_solve(const Grp &g, const LevelT<R> *L, int nlev, const CgVecT<R> &v,
                                               const Phys &F, double tol2, int cg_maxit, double *partials, double *sm,
                                               double *red)
{
    Scal *sc = &s_ctl;
    const Geom &G = L[0].G;
    auto go = [&] { return s_stop == 0 && !sc->done[LOOP_CG]; };
    auto to_rz = [&](const double (&t)[1]) { fin_rz(sc, t); };
    // the V-cycle below the finest level's down half, then its up half
    auto vcycle = [&] {
        R none[1] = {(R)0};
        for (int l = 1; l + 1 < nlev; ++l) {
            const int rows = coarse_rows(g, L[l].G);
            for_pair_tiles(g, L[l].G, [&](int bx, int bz) {
                ph_mg_down<false, R>(L[l], L[l + 1], nullptr, F, sm, bx, bz, rows);
            }, rows);
            gbar(g);
        }
        for (int l = nlev - 1; l >= 1; --l) {
            const R *ec = l == nlev - 1 ? nullptr : L[l + 1].e2;
            const int Pc = l == nlev - 1 ? 0 : L[l + 1].G.P;
            const int rows = coarse_rows(g, L[l].G);
            for_pair_tiles(g, L[l].G, [&](int bx, int bz) {
                ph_mg_up<false, R>(L[l], L[l].r, ec, Pc, L[l].e2, F, sm, bx, bz, none, rows);
            }, rows);
            gbar(g);
        }
        TileSums<R, 1> acc;
        const R *rb = black_res(L[0], sc->cg_it);
        for_pair_tiles(g, G, [&](int bx, int bz) {
            acc.add([&](R (&t)[1]) { ph_rb_up<R>(L[0], rb, L[1].e2, L[1].G.P, L[0].e2, F, bx, bz, t); });
        });
        rbar<1>(g, acc.total(), red, partials, to_rz);
    };
    if (!go()) return;
    if (nlev == 1) {
        TileSums<R, 1> acc;
        for_pair_tiles(g, G, [&](int bx, int bz) {
            acc.add([&](R (&t)[1]) { ph_rb_start<R>(L[0], black_res(L[0], 0), L[0].e2, sm, bx, bz, t); });
        });
        rbar<1>(g, acc.total(), red, partials, to_rz);
    } else {
        for_pair_tiles(g, G, [&](int bx, int bz) {
            ph_mg_down<true, R>(L[0], L[1], black_res(L[0], 0), F, sm, bx, bz);
        });
        gbar(g);
        vcycle();
    }
    while (go()) {
        const int it = sc->cg_it;
        const R *pold = (it & 1) ? v.p1 : v.p0;
        R *pnew = (it & 1) ? v.p0 : v.p1;
        {
            const double beta = sc->beta;
            TileSums<R, 1> acc;
            for_pair_tiles(g, G, [&](int bx, int bz) {
                acc.add([&](R (&t)[1]) { ph_pspmv<R>(L[0], L[0].e2, pold, pnew, v.q, beta, it == 0, sm, bx, bz, t); });
            });
            rbar<1>(g, acc.total(), red, partials, [&](const double (&t)[1]) { fin_pq(sc, t); });
        }
        const double alpha = sc->alpha;
        auto cap = [&] {
            if (!sc->done[LOOP_CG] && !sc->status && sc->cg_it >= cg_maxit) sc->status = GEA_ERR_NOCONV;
        };
        if (nlev == 1) {
            TileSums<R, 2> acc;
            for_pair_tiles(g, G, [&](int bx, int bz) {
                acc.add([&](R (&t)[2]) {
                    ph_update_single<R>(L[0], v.q, black_res(L[0], 0), L[0].e2, v.x, pnew, alpha, it == 0, bx, bz, t);
                });
            });
            rbar<2>(g, acc.total(), red, partials, [&](const double (&t)[2]) {
                const double t0[1] = {t[0]}, t1[1] = {t[1]};
                fin_update(sc, t0, tol2);
                fin_rz(sc, t1);
                cap();
            });
        } else {
            TileSums<R, 1> acc;
            for_pair_tiles(g, G, [&](int bx, int bz) {
                acc.add([&](R (&t)[1]) {
                    ph_update_down<R>(L[0], L[1], v.q, black_res(L[0], it), black_res(L[0], it + 1), v.x, pnew, alpha,
                                      it == 0, F, sm, bx, bz, t);
                });
            });
            rbar<1>(g, acc.total(), red, partials, [&](const double (&t)[1]) {
                fin_update(sc, t, tol2);
                cap();
            });
            if (go()) vcycle();
        }
    }
}

// One time step reading a.S and writing a.N. Returns false if the step did
// not complete (a device error is set).
__device__ bool run_step(const PersistArgs &P, const StepArgs &a, const Grp &g, double *sm, double *red)
{
    Scal *sc = &s_ctl;   // the block's copy (decisions); g.gs holds the published values
    const Geom &G = a.G;
    const Level *L = P.L;
    const int nlev = P.nlev;

    // ---- Smagorinsky eddy viscosity of the step (LES) ----
    if (a.F.les) {
        for_tiles(g, G, [&](int bx, int bz) { ph_les(a, sm, bx, bz); });
        gbar(g);
        if (stop(sc)) return false;
    }
    // ---- Step 1: continuity predictor, transport operator, momentum RHS,
    // and the first Jacobi sweep of the momentum predictor (from u^n, which
    // needs no barrier) into ua, wa ----
    {
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        for_tiles(g, G, [&](int bx, int bz) { ph_pred_sweep(a, sm, bx, bz, acc); });
        rbar<4>(g, acc, red, a.partials, [&](const double (&t)[4]) {
            const double tb[2] = {t[0], t[1]}, tr[2] = {t[2], t[3]};
            fin_pred(sc, tb);
            for (int c = 0; c < 4; ++c) { sc->cg_iters[c] = 0; sc->cg_b2[c] = 0.0; }
            sc->sweeps[1] = 0;
            sc->press_ns = 0ull;
            fin_mom(sc, tr, a.jac_rtol2);
            if (!sc->done[LOOP_MOM] && !sc->status && sc->sweeps[0] >= P.jac_maxit) sc->status = GEA_ERR_NOCONV;
        });
    }
    if (stop(sc)) return false;
    // implicit momentum predictor: Jacobi until the sweep whose residual met
    // the tolerance
    const double *uin = a.ua, *win = a.wa;
    double *uout = a.ub, *wout = a.wb;
    while (!sc->done[LOOP_MOM]) {
        double acc[2] = {0.0, 0.0};
        for_tiles(g, G, [&](int bx, int bz) { ph_mom(a, uin, win, uout, wout, sm, bx, bz, acc); });
        rbar<2>(g, acc, red, a.partials, [&](const double (&t)[2]) {
            fin_mom(sc, t, a.jac_rtol2);
            if (!sc->done[LOOP_MOM] && !sc->status && sc->sweeps[0] >= P.jac_maxit) sc->status = GEA_ERR_NOCONV;
        });
        const double *tu = uin, *tw = win;
        uin = uout; win = wout;
        uout = const_cast<double *>(tu); wout = const_cast<double *>(tw);
        if (stop(sc)) break;
    }
    if (stop(sc)) return false;
    const double *u1 = uin, *w1 = win;

    // ---- Step 2: enthalpy right-hand side with the first enthalpy sweep
    // (from h^n) into ha, then temperature, rho^{n+2/3} ----
    {
        double acc[2] = {0.0, 0.0};
        for_tiles(g, G, [&](int bx, int bz) { ph_enth_rhs_sweep(a, u1, w1, a.ha, sm, bx, bz, acc); });
        rbar<2>(g, acc, red, a.partials, [&](const double (&t)[2]) {
            const double tb[1] = {t[0]}, tr[1] = {t[1]};
            fin_enth_rhs(sc, tb);
            fin_enth(sc, tr, a.jac_rtol2);
            if (!sc->done[LOOP_ENTH] && !sc->status && sc->sweeps[1] >= P.jac_maxit) sc->status = GEA_ERR_NOCONV;
        });
    }
    if (stop(sc)) return false;
    const double *hin = a.ha;
    double *hout = a.hb;
    while (!sc->done[LOOP_ENTH]) {
        double acc[1] = {0.0};
        for_tiles(g, G, [&](int bx, int bz) { ph_enth(a, hin, hout, sm, bx, bz, acc); });
        rbar<1>(g, acc, red, a.partials, [&](const double (&t)[1]) {
            fin_enth(sc, t, a.jac_rtol2);
            if (!sc->done[LOOP_ENTH] && !sc->status && sc->sweeps[1] >= P.jac_maxit) sc->status = GEA_ERR_NOCONV;
        });
        const double *t = hin;
        hin = hout;
        hout = const_cast<double *>(t);
        if (stop(sc)) break;
    }
    if (stop(sc)) return false;
    const double *h1 = hin;
    // the EOS update, and H(u^{n+1/3}) of the first corrector, which reads
    // nothing the EOS phase writes
    for_tiles(g, G, [&](int bx, int bz) { ph_eos(a, L[0], h1, sm, bx, bz); });
    for_tiles(g, G, [&](int bx, int bz) { ph_H(a, u1, w1, sm, bx, bz); });
    gbar(g);
    for (int l = 0; l + 1 < nlev; ++l) {
        for_tiles(g, L[l + 1].G, [&](int bx, int bz) { ph_coarsen(L[l], L[l + 1], a.F.cfx, a.F.cfz, bx, bz); });
        gbar(g);
    }
    if (stop(sc)) return false;
    if (g.rank == 0 && tid_of() == 0) {
        g.gs->u1_slot = (u1 == a.ub);
        g.gs->h1_slot = (h1 == a.hb);
    }

    // ---- Step 3: PISO correctors ----
    for (int c = 0; c < P.n_corr; ++c) {
        if (c > 0) {
            for_tiles(g, G, [&](int bx, int bz) { ph_H(a, a.N.u, a.N.w, sm, bx, bz); });
            gbar(g);
        }
        const double *x0 = pp_in(a, c, P.n_corr);
        unsigned long long t0 = 0;
        if (g.rank == 0 && tid_of() == 0) t0 = globaltimer();
        {
            double acc[2] = {0.0, 0.0};
            for_tiles(g, G, [&](int bx, int bz) { ph_helm_rhs(a, L[0], x0, nullptr, sm, bx, bz, acc); });
            rbar<2>(g, acc, red, a.partials, [&](const double (&t)[2]) { fin_helm(sc, t, a.cg_rtol2, c); });
        }
        pressure_solve<double>(g, L, nlev, cg_vecs(a), a.F, a.cg_rtol2, P.cg_maxit, a.partials, sm, red);
        if (stop(sc)) return false;
        if (g.rank == 0 && tid_of() == 0) sc->press_ns += globaltimer() - t0;
        {
            const SolveT<double> v{x0, nullptr, cg_vecs(a).x};
            const bool dx = sc->cg_it > 0;
            for_tiles(g, G, [&](int bx, int bz) { ph_correct<double>(a, L[0], v, dx, pp_out(a, c, P.n_corr), sm, bx, bz); });
        }
        if (c + 1 < P.n_corr) gbar(g);
    }
    end_step(g);
    return !stop(sc);
}

// One mixed-precision time step (the phases of the graph's mixed step, in
// its order): FP64 residuals, FP32 Jacobi and MG-CG solves of the
// increments, FP64 updates. Returns false if the step did not complete.
__device__ bool run_step_mixed(const PersistArgs &P, const MixedPersist &X, const StepArgs &a, const Grp &g,
                               double *sm, double *red)
{
    Scal *sc = &s_ctl;   // the block's copy (decisions); g.gs holds the published values
    const Geom &G = a.G;
    const MixedArgs &m = X.m;
    const LevelF *L = X.Lf;
    const int nlev = X.nlev;
    const Level &L0 = P.L[0];
    if (g.rank == 0 && tid_of() == 0) g.gs->u1_slot = g.gs->h1_slot = 0;

    if (a.F.les) {
        for_tiles(g, G, [&](int bx, int bz) { ph_les(a, sm, bx, bz); });
        gbar(g);
        if (stop(sc)) return false;
    }
    // ---- Step 1: FP64 residuals r0 = b - T(u^n), FP32 operator, first FP32
    // sweep from zero ----
    {
        double acc[2] = {0.0, 0.0};
        for_tiles(g, G, [&](int bx, int bz) { ph_pred_t<true>(a, m, sm, bx, bz, acc); });
        rbar<2>(g, acc, red, a.partials, [&](const double (&t)[2]) {
            fin_pred(sc, t);
            for (int c = 0; c < 4; ++c) { sc->cg_iters[c] = 0; sc->cg_b2[c] = 0.0; }
            sc->sweeps[1] = 0;
            sc->press_ns = 0ull;
        });
    }
    if (stop(sc)) return false;
    const float *ui = m.du[0], *wi = m.dw[0];
    float *uo = m.du[1], *wo = m.dw[1];
    for (;;) {
        TileSums<float, 2> acc;
        for_tiles(g, G, [&](int bx, int bz) {
            acc.add([&](float (&t)[2]) {
                ph_sweep2<float, BC_U, BC_W>(G, a.F, m.T, m.dinvu, m.r0u, m.r0w, ui, wi, uo, wo, sm, bx, bz, t);
            });
        });
        rbar<2>(g, acc.total(), red, a.partials, [&](const double (&t)[2]) {
            fin_mom(sc, t, m.tol2);
            if (!sc->done[LOOP_MOM] && !sc->status && sc->sweeps[0] >= P.jac_maxit) sc->status = GEA_ERR_NOCONV;
        });
        const float *tu = ui, *tw = wi;
        ui = uo; wi = wo;
        uo = const_cast<float *>(tu); wo = const_cast<float *>(tw);
        if (stop(sc) || sc->done[LOOP_MOM]) break;
    }
    if (stop(sc)) return false;

    // ---- Step 2: u^{n+1/3} = u^n + du, the enthalpy residual at h^n and the
    // first FP32 sweep; FP32 Jacobi on dh ----
    {
        MixedArgs mm = m;   // the momentum increments end in the buffers ui, wi
        mm.du[0] = const_cast<float *>(ui);
        mm.dw[0] = const_cast<float *>(wi);
        double acc[1] = {0.0};
        for_tiles(g, G, [&](int bx, int bz) {
            ph_enth_rhs_t<true>(a, mm, nullptr, nullptr, nullptr, sm, bx, bz, acc);
        });
        rbar<1>(g, acc, red, a.partials, [&](const double (&t)[1]) { fin_enth_rhs(sc, t); });
    }
    if (stop(sc)) return false;
    const float *hi = m.dh[0];
    float *ho = m.dh[1];
    const float lc = (float)(a.F.mu - a.F.nuh);
    for (;;) {
        TileSums<float, 1> acc;
        for_tiles(g, G, [&](int bx, int bz) {
            acc.add([&](float (&t)[1]) {
                ph_sweep1<float, BC_EVEN>(G, a.F, m.T, m.dinvh, m.r0h, lc, hi, ho, sm, bx, bz, t);
            });
        });
        rbar<1>(g, acc.total(), red, a.partials, [&](const double (&t)[1]) {
            fin_enth(sc, t, m.tol2);
            if (!sc->done[LOOP_ENTH] && !sc->status && sc->sweeps[1] >= P.jac_maxit) sc->status = GEA_ERR_NOCONV;
        });
        const float *t = hi;
        hi = ho;
        ho = const_cast<float *>(t);
        if (stop(sc) || sc->done[LOOP_ENTH]) break;
    }
    if (stop(sc)) return false;
    // h^{n+1} = h^n + dh, the EOS update, the FP64 finest Helmholtz level and
    // its FP32 copy; H(u^{n+1/3}) of the first corrector reads nothing of it
    for_tiles(g, G, [&](int bx, int bz) { ph_eos_t<true>(a, L0, L[0], nullptr, hi, sm, bx, bz); });
    for_tiles(g, G, [&](int bx, int bz) { ph_H(a, a.ua, a.wa, sm, bx, bz); });
    gbar(g);
    for (int l = 0; l + 1 < nlev; ++l) {
        for_tiles(g, L[l + 1].G, [&](int bx, int bz) { ph_coarsen<float>(L[l], L[l + 1], a.F.cfx, a.F.cfz, bx, bz); });
        gbar(g);
    }
    if (stop(sc)) return false;

    // ---- Step 3: PISO correctors, each pressure solve one defect correction ----
    for (int c = 0; c < P.n_corr; ++c) {
        if (c > 0) {
            for_tiles(g, G, [&](int bx, int bz) { ph_H(a, a.N.u, a.N.w, sm, bx, bz); });
            gbar(g);
        }
        const double *x0 = pp_in(a, c, P.n_corr);
        unsigned long long t0 = 0;
        if (g.rank == 0 && tid_of() == 0) t0 = globaltimer();
        {
            double acc[2] = {0.0, 0.0};
            for_tiles(g, G, [&](int bx, int bz) {
                ph_helm_rhs_t<true>(a, L0, L[0], m, x0, nullptr, false, sm, bx, bz, acc);
            });
            rbar<2>(g, acc, red, a.partials, [&](const double (&t)[2]) {
                fin_helm_mixed(sc, t, a.cg_rtol2, c);
            });
        }
        pressure_solve<float>(g, L, nlev, cg_vecs(m), a.F, m.tol2, P.cg_maxit, a.partials, sm, red);
        if (stop(sc)) return false;
        if (g.rank == 0 && tid_of() == 0) sc->press_ns += globaltimer() - t0;
        {
            // p' += dp, and the FP64 correction
            const SolveT<float> v{x0, nullptr, cg_vecs(m).x};
            const bool dx = sc->cg_it > 0;
            for_tiles(g, G, [&](int bx, int bz) { ph_correct<float>(a, L[0], v, dx, pp_out(a, c, P.n_corr), sm, bx, bz); });
        }
        if (c + 1 < P.n_corr) gbar(g);
    }
    end_step(g);
    return !stop(sc);
}

// Block rank in a launch of one context: blocks counted from the last. Block
// ids fill the SMs in order, and with three blocks an SM the first twelve
// land on four SMs (measured by %smid: 456 blocks, the first 100 on 92 SMs),
// the last 148 on as many. A phase of a coarse level has work for a few ranks
// only; counted from the front its tiles shared four SMs' FP64 units. 400 x 400
// with five levels: 2070 -> 1844 us a step, 200 x 200 (175 blocks) 1100 -> 1076.
__device__ __forceinline__ int single_rank() { return (int)(gridDim.x - 1 - blockIdx.x); }

// The argument block `src` copied to shared memory (whole words).
template <class T>
__device__ __forceinline__ const T &args_to_shared(void *dst, const T &src)
{
    static_assert(sizeof(T) % 4 == 0, "copied by words");
    const uint32_t *s = reinterpret_cast<const uint32_t *>(&src);
    uint32_t *d = reinterpret_cast<uint32_t *>(dst);
    for (int w = tid_of(); w < (int)(sizeof(T) / 4); w += NTHREADS) d[w] = s[w];
    return *reinterpret_cast<const T *>(dst);
}

// The step kernels read their arguments (pointers and sizes of the state, the
// work arrays and every level, several kB) from a copy in shared memory, as an
// ensemble's blocks do. Kernel parameters indexed by slot or level at run time
// come through the small constant cache, which the phases in turn overflow. Per
// pass: 640 x 320 2005 -> 1938 us, 160 x 80 267 -> 259, the multi-level grids 1 %.
constexpr size_t kArgsFp64 = sizeof(PersistArgs);
constexpr size_t kArgsMixed = sizeof(PersistArgs) + sizeof(MixedPersist);
constexpr size_t kPersistSmem =
    (size_t)(kTileSmem + kRedVals * NTHREADS) * sizeof(double) + (kArgsFp64 + 15) / 16 * 16;
constexpr size_t kPersistSmemMixed =
    (size_t)(kTileSmem + kRedVals * NTHREADS) * sizeof(double) + (kArgsMixed + 15) / 16 * 16;

__global__ void __launch_bounds__(NTHREADS, 3) k_persistent(const __grid_constant__ PersistArgs Pk)
{
    extern __shared__ double dsm[];
    double *sm = dsm;
    double *red = dsm + kTileSmem;
    const PersistArgs &P = args_to_shared(red + kRedVals * NTHREADS, Pk);
    // an error status is sticky until the next set_state, which clears it
    __shared__ unsigned gen;
    Scal *gs = Pk.a[0].sc;
    if (tid_of() == 0) {
        s_stop = rdi(&gs->status) != 0;
        gen = 0u;
    }
    load_ctl(gs);
    __syncthreads();
    const Grp g{single_rank(), (int)gridDim.x, &gen, gs, P.spin_limit, P.a[0].trace, P.a[0].trace_bars};
    trace_entry(g);
    if (!s_stop) {
        if (g.rank == 0 && tid_of() == 0) gs->launches += 1;
        for (int s = 0; s < P.nsteps; ++s) {
            const int slot = (P.first_slot + s) & 1;
            if (!run_step(P, P.a[slot], g, sm, red)) break;
        }
        if (g.rank == 0 && tid_of() == 0 && rdi(&gs->status)) gs->last_status = rdi(&gs->status);
    }
    leave(g);
}

// The mixed-precision step as one cooperative launch (small grids).
__global__ void __launch_bounds__(NTHREADS, 3)
    k_persistent_mixed(const __grid_constant__ PersistArgs Pk, const __grid_constant__ MixedPersist Xk)
{
    extern __shared__ double dsm[];
    double *sm = dsm;
    double *red = dsm + kTileSmem;
    char *args = reinterpret_cast<char *>(red + kRedVals * NTHREADS);
    const PersistArgs &P = args_to_shared(args, Pk);
    const MixedPersist &X = args_to_shared(args + sizeof(PersistArgs), Xk);
    __shared__ unsigned gen;
    Scal *gs = Pk.a[0].sc;
    if (tid_of() == 0) {
        s_stop = rdi(&gs->status) != 0;
        gen = 0u;
    }
    load_ctl(gs);
    __syncthreads();
    const Grp g{single_rank(), (int)gridDim.x, &gen, gs, P.spin_limit, P.a[0].trace, P.a[0].trace_bars};
    trace_entry(g);
    if (!s_stop) {
        if (g.rank == 0 && tid_of() == 0) gs->launches += 1;
        for (int s = 0; s < P.nsteps; ++s) {
            const int slot = (P.first_slot + s) & 1;
            if (!run_step_mixed(P, X, P.a[slot], g, sm, red)) break;
        }
        if (g.rank == 0 && tid_of() == 0 && rdi(&gs->status)) gs->last_status = rdi(&gs->status);
    }
    leave(g);
}

// An ensemble of independent contexts in one cooperative launch. The blocks
// form groups (table `groups`: ngroups + 1 first blocks, ngroups + 1 first
// entries of the member list, then the member list): a group of several
// blocks runs one member, with its own barrier and reductions over those
// blocks only, so members whose solves take different iteration counts never
// wait for one another; a group of one block may run several small members,
// one after another, each as a one-block grid. Each block keeps the argument
// block of the member it runs in shared memory: a PersistArgs block of
// `stride` bytes per member, for the mixed-precision step (MX) followed by
// the member's MixedPersist.
template <bool MX>
__global__ void __launch_bounds__(NTHREADS, 3) k_ensemble(const char *Pm, int stride, const int *groups, int ngroups)
{
    extern __shared__ double dsm[];
    double *sm = dsm;
    double *red = dsm + kTileSmem;
    PersistArgs *Ps = reinterpret_cast<PersistArgs *>(dsm + kTileSmem + kRedVals * NTHREADS);
    const int tid = tid_of();
    const int *gb = groups, *gm = groups + ngroups + 1, *order = gm + ngroups + 1;
    int lo = 0, hi = ngroups - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) / 2;
        if (__ldg(&gb[mid]) <= (int)blockIdx.x) lo = mid;
        else hi = mid - 1;
    }
    const int b0 = __ldg(&gb[lo]), nbk = __ldg(&gb[lo + 1]) - b0;
    const int i1 = __ldg(&gm[lo + 1]);
    __shared__ unsigned gen;
    for (int i = __ldg(&gm[lo]); i < i1; ++i) {
        const int m = __ldg(&order[i]);
        __syncthreads();   // nothing reads the previous member's arguments any more
        {
            const uint32_t *src = reinterpret_cast<const uint32_t *>(Pm + (size_t)m * stride);
            uint32_t *dst = reinterpret_cast<uint32_t *>(Ps);
            for (int w = tid; w < stride / 4; w += NTHREADS) dst[w] = __ldg(&src[w]);
        }
        __syncthreads();
        const PersistArgs &P = *Ps;
        const MixedPersist &X = *reinterpret_cast<const MixedPersist *>(reinterpret_cast<const char *>(Ps) +
                                                                        sizeof(PersistArgs));
        Scal *sc = P.a[0].sc;
        if (tid == 0) {
            s_stop = rdi(&sc->status) != 0;
            gen = 0u;
        }
        load_ctl(sc);
        __syncthreads();
        const Grp g{(int)blockIdx.x - b0, nbk, &gen, sc, P.spin_limit, nullptr, 0};
        if (!s_stop) {
            if (g.rank == 0 && tid == 0) sc->launches += 1;
            for (int s = 0; s < P.nsteps; ++s) {
                const int slot = (P.first_slot + s) & 1;
                const bool ok =
                    MX ? run_step_mixed(P, X, P.a[slot], g, sm, red) : run_step(P, P.a[slot], g, sm, red);
                if (!ok) break;
            }
            if (g.rank == 0 && tid == 0 && rdi(&sc->status)) sc->last_status = rdi(&sc->status);
        }
        leave(g);
    }
}

int ensemble_max_blocks(int mixed)
{
    int dev = 0, sms = 0, per_sm = 0;
    const void *k = mixed ? (const void *)k_ensemble<true> : (const void *)k_ensemble<false>;
    const size_t smem = mixed ? kPersistSmemMixed : kPersistSmem;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, NTHREADS, smem) != cudaSuccess) return 0;
    return per_sm * sms;
}

cudaError_t launch_ensemble(const void *Pm, int mixed, const int *groups, int ngroups, int blocks, cudaStream_t st)
{
    const char *P = static_cast<const char *>(Pm);
    int stride = (int)(mixed ? kArgsMixed : kArgsFp64);
    void *args[] = {&P, &stride, &groups, &ngroups};
    const void *k = mixed ? (const void *)k_ensemble<true> : (const void *)k_ensemble<false>;
    return cudaLaunchCooperativeKernel(k, dim3(blocks), dim3(BX, BZ), args,
                                       mixed ? kPersistSmemMixed : kPersistSmem, st);
}

int persistent_max_blocks()
{
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (cudaFuncSetAttribute(k_persistent, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kPersistSmem) != cudaSuccess)
        return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_persistent, NTHREADS, kPersistSmem) !=
        cudaSuccess)
        return 0;
    return per_sm * sms;
}

cudaError_t launch_persistent(const StepArgs a[2], const Level *L, int nlev, int n_corr,
                              int jac_maxit, int cg_maxit, int first_slot, int nsteps, int blocks,
                              long long wait_polls, cudaStream_t st)
{
    if (nlev < 1 || nlev > kMaxLevels) return cudaErrorInvalidValue;
    PersistArgs P;
    memset(&P, 0, sizeof(P));
    P.a[0] = a[0];
    P.a[1] = a[1];
    for (int l = 0; l < nlev; ++l) P.L[l] = L[l];
    P.nlev = nlev;
    P.nsteps = nsteps;
    P.first_slot = first_slot;
    P.n_corr = n_corr;
    P.jac_maxit = jac_maxit;
    P.cg_maxit = cg_maxit;
    P.spin_limit = spin_limit_of(wait_polls);
    void *args[] = {&P};
    return cudaLaunchCooperativeKernel((const void *)k_persistent, dim3(blocks), dim3(BX, BZ), args,
                                       kPersistSmem, st);
}

int persistent_mixed_max_blocks()
{
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (cudaFuncSetAttribute(k_persistent_mixed, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kPersistSmemMixed) != cudaSuccess)
        return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_persistent_mixed, NTHREADS, kPersistSmemMixed) !=
        cudaSuccess)
        return 0;
    return per_sm * sms;
}

cudaError_t launch_persistent_mixed(const StepArgs a[2], const Level &L0, const MixedArgs &m, const LevelF *Lf,
                                    int nlev, int n_corr, int jac_maxit, int cg_maxit,
                                    int first_slot, int nsteps, int blocks, long long wait_polls,
                                    cudaStream_t st)
{
    if (nlev < 1 || nlev > kMaxLevels) return cudaErrorInvalidValue;
    PersistArgs P;
    memset(&P, 0, sizeof(P));
    P.a[0] = a[0];
    P.a[1] = a[1];
    P.L[0] = L0;
    P.nlev = 1;
    P.nsteps = nsteps;
    P.first_slot = first_slot;
    P.n_corr = n_corr;
    P.jac_maxit = jac_maxit;
    P.cg_maxit = cg_maxit;
    P.spin_limit = spin_limit_of(wait_polls);
    MixedPersist X;
    memset(&X, 0, sizeof(X));
    X.m = m;
    for (int l = 0; l < nlev; ++l) X.Lf[l] = Lf[l];
    X.nlev = nlev;
    void *args[] = {&P, &X};
    return cudaLaunchCooperativeKernel((const void *)k_persistent_mixed, dim3(blocks), dim3(BX, BZ), args,
                                       kPersistSmemMixed, st);
}

}  // namespace

// the host entry points of this tile shape (external linkage: the shape
// table in gea_persistent.cu refers to it)
extern const PersistOps ops;
const PersistOps ops = {BX,
                        BZ,
                        persistent_max_blocks,
                        persistent_mixed_max_blocks,
                        ensemble_max_blocks,
                        launch_persistent,
                        launch_persistent_mixed,
                        launch_ensemble};
