// Complex128 stencil sweeps: the PML Helmholtz operator and one Taylor-Horner
// step of the exponential-integrator actions (Def. psi),
//     out = rho (y + sigma (A_s - mu) p + gamma v).
//
// GB300 issues about two FP64 operations per clock and SM (1.05 TFLOP/s measured),
// so an update costs what its FP64 instructions cost: the kernel is written for
// their number, and memory (64 B per update: p, y, the diagonal and the result;
// 2.7 TB/s at its rate) is far from a bound.  Everything is scaled by h^2, so that a
// neighbour outside the PML has coefficient 1 and costs an addition:
//   q = sum_d (wp_d p_{+d} + wm_d p_{-d}) + D p,   D = h^2 (kappa (1 + i s) - mu - sum_d wc_d + faces),
// with D read from a table that is made once per parameter set (k_diag64) and
// sigma = i tau folded into two multiply-adds with y.  An interior 2D update is
// then 6 additions + 4 + 2 multiply-adds = 12 FP64 instructions (3D: 16), where
// the general form needs 32 (3D: 42); an axis in its PML adds 4 to 6.
// Measured: 28.2 us a sweep of 1088^2 unknowns (42 G updates/s; 12 instructions at
// the measured 0.527 T/s would be 27 us), the general form 117 us; 2.4 us a sweep of
// 160^2, before 8.2 us; the psi_1 action on 128^3 127 ms, before 477 ms.
#include "mxp_internal.h"

namespace mxp {

// Scalars of a sweep, scaled: sig = sigma / h^2, (zx, zy) = h^2 (1 + i s), mu = h^2 mu.
struct Scal64 {
    double2 sig, gam, rho;
    double zx, zy, mu;
    int fast;        // sigma imaginary and rho = 1
    int nfaces;
    double h2;
    const double2 *face[6];
};

// Loads of the vectors.  A sweep may start before the previous one has ended
// (programmatic dependent launch), so they must stay behind the grid dependency
// wait: volatile asm keeps its order, a plain read-only load need not.
__device__ __forceinline__ double2 ldv(const double2 *p)
{
    double2 r;
    asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(r.x), "=d"(r.y) : "l"(p) : "memory");
    return r;
}

// Lets the next sweep's blocks start; they wait for this sweep's end before they read.
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <int DIM>
__device__ __forceinline__ double2 face_terms(const Geom &g, const Scal64 &sc, int i, int j, int k)
{
    // rows on a sound-hard or absorbing face: the ghost value is a multiple of
    // the row's own unknown, so its coefficient joins the diagonal
    double2 f = make_double2(0.0, 0.0);
    const int n0 = g.n[0], n1 = g.n[1];
    if (sc.face[0] && i == 0) f = cadd(f, sc.face[0][j + (int64_t)n1 * k]);
    if (sc.face[1] && i == n0 - 1) f = cadd(f, sc.face[1][j + (int64_t)n1 * k]);
    if (sc.face[2] && j == 0) f = cadd(f, sc.face[2][i + (int64_t)n0 * k]);
    if (sc.face[3] && j == n1 - 1) f = cadd(f, sc.face[3][i + (int64_t)n0 * k]);
    if (DIM >= 3) {
        if (sc.face[4] && k == 0) f = cadd(f, sc.face[4][i + (int64_t)n0 * j]);
        if (sc.face[5] && k == g.n[2] - 1) f = cadd(f, sc.face[5][i + (int64_t)n0 * j]);
    }
    return make_double2(f.x * sc.h2, f.y * sc.h2);
}

template <int DIM>
__device__ __forceinline__ double2 diag_of(const Geom &g, const double2 *coef, const double *kappa, const Scal64 &sc,
                                           int i, int j, int k, int64_t q)
{
    const int nm = g.nmax;
    double2 wcs = cadd(coef[2 * nm + i], coef[5 * nm + j]);
    if (DIM >= 3) wcs = cadd(wcs, coef[8 * nm + k]);
    const double kp = kappa[q];
    double2 d = make_double2(kp * sc.zx - sc.mu - wcs.x, kp * sc.zy - wcs.y);
    if (sc.nfaces) d = cadd(d, face_terms<DIM>(g, sc, i, j, k));
    return d;
}

__device__ __forceinline__ void fma_c(double2 &a, double2 c, double2 p)
{
    a.x = fma(c.x, p.x, a.x);
    a.x = fma(-c.y, p.y, a.x);
    a.y = fma(c.x, p.y, a.y);
    a.y = fma(c.y, p.x, a.y);
}

// One point, its axes inside (P = true) or outside their PML.  A body of its own
// for each combination: as branches inside one body the forms are short enough for
// the compiler to predicate, and a predicated-off FP64 instruction takes its 64
// cycles of the pipe all the same (28 instructions a point were issued instead of
// 14, 62.7 us a 1088^2 sweep).
template <int DIM, bool HAS_Y, bool HAS_V, bool FAST, int REL, bool PX, bool PY, bool PZ>
__device__ __forceinline__ void point64(const Geom &g, const double2 *__restrict__ coef,
                                        const double *__restrict__ kappa, const double2 *__restrict__ diag,
                                        const Scal64 &sc, const double2 *pin, const double2 *y, const double2 *v,
                                        double2 *pout, int i, int j, int k, int64_t q, bool act)
{
    const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2], nm = g.nmax;
    // tables of the problem: not written by a sweep
    const double2 d = diag ? diag[q] : diag_of<DIM>(g, coef, kappa, sc, i, j, k, q);
    double2 wpx, wmx, wpy, wmy, wpz, wmz;
    if (PX) { wpx = coef[i]; wmx = coef[nm + i]; }
    if (PY) { wpy = coef[3 * nm + j]; wmy = coef[4 * nm + j]; }
    if (PZ) { wpz = coef[6 * nm + k]; wmz = coef[7 * nm + k]; }
    if (REL == 0) let_next_start();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (REL == 1) let_next_start();
    const double2 zero = make_double2(0.0, 0.0);
    const double2 *pq = pin + q;
    const double2 pc = ldv(pq);
    const double2 xp = (i + 1 < n0) ? ldv(pq + 1) : zero;
    const double2 xm = (i > 0) ? ldv(pq - 1) : zero;
    const double2 yp = (j + 1 < n1) ? ldv(pq + g.s1) : zero;
    const double2 ym = (j > 0) ? ldv(pq - g.s1) : zero;
    double2 zp = zero, zm = zero, yv = zero, vv = zero;
    if (DIM >= 3) {
        if (k + 1 < n2) zp = ldv(pq + g.s2);
        if (k > 0) zm = ldv(pq - g.s2);
    }
    if (HAS_Y) yv = ldv(y + q);
    if (HAS_V) vv = ldv(v + q);

    // the additions first, then the multiply-adds onto them
    double2 a = zero;
    bool first = true;
    auto add = [&](double2 s) { a = first ? s : cadd(a, s); first = false; };
    if (!PX) add(cadd(xp, xm));
    if (!PY) add(cadd(yp, ym));
    if (DIM >= 3 && !PZ) add(cadd(zp, zm));
    auto mul = [&](double2 c, double2 p) {
        if (first) a = cmul(c, p);
        else fma_c(a, c, p);
        first = false;
    };
    if (PX) { mul(wpx, xp); mul(wmx, xm); }
    if (PY) { mul(wpy, yp); mul(wmy, ym); }
    if (DIM >= 3 && PZ) { mul(wpz, zp); mul(wmz, zm); }
    mul(d, pc);
    double2 o;
    if (FAST) {
        o = HAS_Y ? make_double2(fma(-sc.sig.y, a.y, yv.x), fma(sc.sig.y, a.x, yv.y))
                  : make_double2(-sc.sig.y * a.y, sc.sig.y * a.x);
    } else {
        o = yv;
        fma_c(o, sc.sig, a);
    }
    if (HAS_V) fma_c(o, sc.gam, vv);
    if (!FAST) o = cmul(sc.rho, o);
    if (REL == 2) let_next_start();
    if (act) pout[q] = o;
}

// One point per thread, a warp along x (so the PML of y and z is uniform over a
// warp, and a warp takes the general x form when any of its lanes needs it).
// FAST: sigma imaginary and rho = 1 (every sweep of an action but the last).  REL: see
// released_at (a template argument: tested at run time it costs 0.2 us a sweep).
template <int DIM, bool HAS_Y, bool HAS_V, bool FAST, int REL>
__global__ void __launch_bounds__(256) k_step64(Geom g, const double2 *__restrict__ coef,
                                                const double *__restrict__ kappa, const double2 *__restrict__ diag,
                                                const __grid_constant__ Scal64 sc, const double2 *pin,
                                                const double2 *y, const double2 *v, double2 *pout)
{
    const int i = blockIdx.x * 32 + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = DIM >= 3 ? blockIdx.z : 0;
    const bool act = i < g.n[0] && j < g.n[1];
    const int ic = min(i, g.n[0] - 1), jc = min(j, g.n[1] - 1);
    const int64_t q = ic + g.s1 * jc + g.s2 * k;
    const bool px = __any_sync(0xffffffffu, act && (i < g.in_lo[0] || i >= g.in_hi[0]));
    const bool py = jc < g.in_lo[1] || jc >= g.in_hi[1];
    const bool pz = DIM >= 3 && (k < g.in_lo[2] || k >= g.in_hi[2]);
#define MXP_POINT(X, Y, Z) \
    point64<DIM, HAS_Y, HAS_V, FAST, REL, X, Y, Z>(g, coef, kappa, diag, sc, pin, y, v, pout, ic, jc, k, q, act)
    switch ((px ? 1 : 0) | (py ? 2 : 0) | (pz ? 4 : 0)) {
    case 0: MXP_POINT(false, false, false); break;
    case 1: MXP_POINT(true, false, false); break;
    case 2: MXP_POINT(false, true, false); break;
    case 3: MXP_POINT(true, true, false); break;
    case 4: MXP_POINT(false, false, DIM >= 3); break;
    case 5: MXP_POINT(true, false, DIM >= 3); break;
    case 6: MXP_POINT(false, true, DIM >= 3); break;
    default: MXP_POINT(true, true, DIM >= 3); break;
    }
#undef MXP_POINT
}

template <int DIM>
__global__ void __launch_bounds__(256) k_diag64(Geom g, const double2 *__restrict__ coef,
                                                const double *__restrict__ kappa,
                                                const __grid_constant__ Scal64 sc, double2 *__restrict__ diag)
{
    const int i = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = DIM >= 3 ? blockIdx.z : 0;
    if (i >= g.n[0] || j >= g.n[1]) return;
    const int64_t q = i + g.s1 * j + g.s2 * k;
    diag[q] = diag_of<DIM>(g, coef, kappa, sc, i, j, k, q);
}

// Where a sweep lets the next one start: before its own wait (0), after it (1) or before
// its stores (2).  Released before the wait, a third and a fourth sweep start too while
// the first still runs: waiting blocks fill the SMs, and those of a later sweep go
// wherever some end, several to one SM and none to another (224^2: 6.3 us a sweep, 24^3
// 5.4 us).  After the wait there is at most one sweep ahead, evenly placed as long as
// two fit side by side (224^2 3.0, 24^3 2.6, but 352^2 7.2 us); before the stores it is
// placed on SMs that are about to be free (3.0, 2.8 and 5.0 us).  Up to four warps an
// SM the earlier start gains more; up to one, waiting blocks do no harm (24^2: 1.97,
// 2.17 and 2.21 us).  From some forty warps an SM on a sweep does not fit the SMs at
// once: its own blocks fill every gap, and the early release saves up to 3% (512^2: 8.2,
// 8.2 and 8.45 us).
static int released_at(const Geom &g)
{
    const int64_t warps = (int64_t)((g.n[0] + 31) / 32) * g.n[1] * g.n[2], sms = sm_count();
    return warps <= sms || warps > 40 * sms ? 0 : warps <= 4 * sms ? 1 : 2;
}

static Scal64 scaled(const Geom &g, const StepScalars<double2> &s)
{
    Scal64 r;
    const double h2 = 1.0 / g.ih2;
    r.sig = make_double2(s.sigma.x * g.ih2, s.sigma.y * g.ih2);
    r.gam = s.gamma;
    r.rho = s.rho;
    r.zx = s.zfac.x * h2;
    r.zy = s.zfac.y * h2;
    r.mu = s.mu * h2;
    r.fast = s.sigma.x == 0.0 && s.rho.x == 1.0 && s.rho.y == 0.0;
    r.nfaces = s.nfaces;
    r.h2 = h2;
    for (int f = 0; f < 6; ++f) r.face[f] = s.face[f];
    return r;
}

// Rows per block (a warp each): 4, one warp for each partition of an SM; 2 on grids
// too small to give every SM four such blocks, so that the last wave is not one block of
// a whole SM's work.  Blocks of 8 are no faster anywhere (us a sweep, 8 against 4 rows:
// 512^2 8.2 and 8.0, 56^3 10.6 and 9.9, 1088^2 28.6 and 28.3), blocks of 1 run out of
// block slots (1088^2 38, 320^2 5.1 against 4.5) and gain little on small grids (216^2
// 3.3 against 2.9, 28^3 2.9 and 2.9).
static void shape64(const Geom &g, dim3 *grid, dim3 *block)
{
    const int64_t bx = (g.n[0] + 31) / 32;
    const int by = bx * ((g.n[1] + 3) / 4) * g.n[2] < (int64_t)sm_count() * 4 ? 2 : 4;
    *block = dim3(32, by);
    *grid = dim3((unsigned)bx, (g.n[1] + by - 1) / by, g.n[2]);
}

template <int DIM, bool Y, bool V>
static void launch64(const Geom &g, const double2 *coef, const double *kappa, const double2 *diag, const Scal64 &sc,
                     const double2 *pin, const double2 *y, const double2 *v, double2 *pout, cudaStream_t st, bool chain)
{
    dim3 grid, block;
    shape64(g, &grid, &block);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = chain ? 1 : 0;
    // sweeps with y and the fast scalars are chained to one another; the others have
    // nothing behind them that is (an operator, a single step) or come once an action
    const int rel = Y && sc.fast ? released_at(g) : 2;
    if constexpr (Y) {
        if (rel == 0) {
            cudaLaunchKernelEx(&cfg, k_step64<DIM, Y, V, true, 0>, g, coef, kappa, diag, sc, pin, y, v, pout);
            return;
        }
        if (rel == 1) {
            cudaLaunchKernelEx(&cfg, k_step64<DIM, Y, V, true, 1>, g, coef, kappa, diag, sc, pin, y, v, pout);
            return;
        }
    }
    if (sc.fast) cudaLaunchKernelEx(&cfg, k_step64<DIM, Y, V, true, 2>, g, coef, kappa, diag, sc, pin, y, v, pout);
    else cudaLaunchKernelEx(&cfg, k_step64<DIM, Y, V, false, 2>, g, coef, kappa, diag, sc, pin, y, v, pout);
}

template <int DIM>
static void launch64_dim(const Geom &g, const double2 *coef, const double *kappa, const double2 *diag,
                         const Scal64 &sc, const double2 *pin, const double2 *y, const double2 *v, double2 *pout,
                         cudaStream_t st, bool chain)
{
    if (y && v) launch64<DIM, true, true>(g, coef, kappa, diag, sc, pin, y, v, pout, st, chain);
    else if (y) launch64<DIM, true, false>(g, coef, kappa, diag, sc, pin, y, v, pout, st, chain);
    else if (v) launch64<DIM, false, true>(g, coef, kappa, diag, sc, pin, y, v, pout, st, chain);
    else launch64<DIM, false, false>(g, coef, kappa, diag, sc, pin, y, v, pout, st, chain);
}

void launch_step64(const Geom &g, const double2 *coef, const double *kappa, const double2 *diag,
                   const StepScalars<double2> &sc, const double2 *pin, const double2 *y, const double2 *v,
                   double2 *pout, cudaStream_t st, bool chain)
{
    const Scal64 s = scaled(g, sc);
    count_launch();
    if (g.dim == 3) launch64_dim<3>(g, coef, kappa, diag, s, pin, y, v, pout, st, chain);
    else launch64_dim<2>(g, coef, kappa, diag, s, pin, y, v, pout, st, chain);
}

void make_diag64(const Geom &g, const double2 *coef, const double *kappa, const StepScalars<double2> &sc,
                 double2 *diag, cudaStream_t st)
{
    const Scal64 s = scaled(g, sc);
    dim3 grid, block;
    shape64(g, &grid, &block);
    count_launch();
    if (g.dim == 3) k_diag64<3><<<grid, block, 0, st>>>(g, coef, kappa, s, diag);
    else k_diag64<2><<<grid, block, 0, st>>>(g, coef, kappa, s, diag);
}

}  // namespace mxp
