// Two Taylor-Horner steps of a 3D exp action per launch (Def. psi on the operator of
// Eq. helmholtz, Eq. pml-1d-s and Sec. 3.4), complex64 and bfloat16 storage:
//   q = y + sigma1 (A_s - mu) p,   out = rho (y + sigma2 (A_s - mu) q).
//
// One step per launch moves 28 B (bf16 storage: 16 B) a point and step through HBM on
// grids beyond L2; two steps share the reads of p, y and kappa and the write.  A block
// marches along z over a region of RX x 16 columns, two adjacent columns per thread: at
// plane z it computes q(z) from p(z-1 .. z+1) and, from q(z-2 .. z), out(z-1) on the
// region without its edge (an output tile of (RX - 4) x 14: x starts stay multiples of
// 4 cells).  p, y and kappa of a plane arrive by cp.async.bulk.tensor in a ring of four
// stages, with the grid's surroundings filled with zeros; own-column values stay in
// registers, so a pair of points costs seven shared loads for q and four for out, and
// there is one block barrier per plane for both steps.  q is rounded to the storage
// type, as it is between launches of single steps: the results are those of the
// single-step sweeps to the last bit.
//
// Measured on 288^3, complex64: 200 us for two steps (230 us in single steps; 28 B a
// point and two steps would be 98 us of HBM), about 65% of the issue slots in use; the
// exp action 156 ms, before 180 ms.  In L2: 11.4 us a step of 129 x 102 x 115, before
// 14.4 us; 24.5 us of 160^3, before 28.7 us; 3.2 us of 56^3, before 10.3 us.
//
// The kernel is bound by its instructions, so a warp's row takes one of three bodies:
// all of it outside the PML (neighbours summed, real coefficient), in the PML in x
// only (complex coefficients on one axis; the points outside it run along with
// coefficients 1), or the general one.
//
// Every wait on an mbarrier is bounded: on timeout the kernel sets the error word, stops
// issuing loads, waits (bounded) for those in flight and returns.
#include "mxp_internal.h"
#include "tma3.h"

namespace mxp {

namespace {

constexpr int kRows = 16;            // region rows of a block
constexpr int kRing = 4;             // planes resident or in flight
constexpr int kThreads2 = 256;

template <typename S, int RX> struct Geo2 {
    static constexpr int W = RX + 4;                     // loaded columns, from x0 - 4
    static constexpr int al(int b) { return (b + 127) / 128 * 128; }
    static constexpr int PB = (kRows + 2) * W * (int)sizeof(S), YB = kRows * W * (int)sizeof(S), KB = kRows * W * 4;
    static constexpr int OY = al(PB), OK = OY + al(YB), STAGE = OK + al(KB), TX = PB + YB + KB;
    static constexpr int QB = kRows * RX * 8;            // one plane of q (float2)
    static constexpr size_t SMEM = (size_t)kRing * STAGE + 2 * QB + 128;
};

template <typename S> __device__ __forceinline__ float4 ld_pair(const S *p);
template <> __device__ __forceinline__ float4 ld_pair<float2>(const float2 *p) { return *reinterpret_cast<const float4 *>(p); }
template <> __device__ __forceinline__ float4 ld_pair<__nv_bfloat162>(const __nv_bfloat162 *p)
{
    const uint2 u = *reinterpret_cast<const uint2 *>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
// v rounded to the storage type
__device__ __forceinline__ float2 rounded(float2 v, float2) { return v; }
__device__ __forceinline__ float2 rounded(float2 v, __nv_bfloat162) { return __bfloat1622float2(__float22bfloat162_rn(v)); }

struct Point3 {
    float2 xp, xm, yp, ym, pp, pm, pc;
};

// The arithmetic of one step, written out as the single-step sweeps compute it: a
// complex product is one rounded product and one multiply-add per component (mul0 and
// mul1 differ in which), all other operations round on their own, in their order.
// The sums are packed pairs, one instruction for both components (215 -> 203 us); the
// products stay scalar, since the compiler contracts a packed product into the sum
// that follows it, which rounds once instead of twice.
__device__ __forceinline__ float2 add_rn(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 scale_rn(float s, float2 a) { return make_float2(__fmul_rn(s, a.x), __fmul_rn(s, a.y)); }
__device__ __forceinline__ float2 mul0(float2 a, float2 b)
{
    return make_float2(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x)));
}
__device__ __forceinline__ float2 mul1(float2 a, float2 b)
{
    return make_float2(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.y, b.x, __fmul_rn(a.x, b.y)));
}
// products with the x and z coefficients: the TMA-staged single step forms them as mul1,
// the register-marching one (rows that are no multiple of 4) as mul0
template <bool REG> __device__ __forceinline__ float2 mulxz(float2 a, float2 b) { return REG ? mul0(a, b) : mul1(a, b); }

// (A_s - mu) p without the diagonal, outside the PML: neighbours summed, one factor
__device__ __forceinline__ float2 lap_inner(const Point3 &n, float ih2)
{
    return scale_rn(ih2, add_rn(add_rn(add_rn(n.xp, n.xm), add_rn(n.yp, n.ym)), add_rn(n.pp, n.pm)));
}
// y and z outside their PML (coefficient m): in the x PML m = 1 / h^2 and f = 1; outside
// it the x coefficients and m are 1 and f = 1 / h^2
template <bool REG>
__device__ __forceinline__ float2 lap_x(const Point3 &n, float2 wp, float2 wm, float m, float f)
{
    float2 a = add_rn(mulxz<REG>(wp, n.xp), mulxz<REG>(wm, n.xm));
    a = add_rn(a, add_rn(scale_rn(m, n.yp), scale_rn(m, n.ym)));
    return scale_rn(f, add_rn(a, add_rn(scale_rn(m, n.pp), scale_rn(m, n.pm))));
}
struct Coef3 {
    float2 wpx, wmx, wpy, wmy, czp, czm;
};
template <bool REG> __device__ __forceinline__ float2 lap_general(const Point3 &n, const Coef3 &w)
{
    float2 a = add_rn(mulxz<REG>(w.wpx, n.xp), mulxz<REG>(w.wmx, n.xm));
    a = add_rn(a, add_rn(mul0(w.wpy, n.yp), mul0(w.wmy, n.ym)));
    return add_rn(a, add_rn(mulxz<REG>(w.czp, n.pp), mulxz<REG>(w.czm, n.pm)));
}
// y + i sig (lap + (kappa (1 + i s) - wcs) pc)
__device__ __forceinline__ float2 finish(float2 lap, float2 pc, float2 wcs, float kp, float zy, float sig, float2 y)
{
    const float2 d = make_float2(__fadd_rn(kp, -wcs.x), __fmaf_rn(kp, zy, -wcs.y));
    const float2 a = add_rn(lap, mul1(d, pc));
    return add_rn(make_float2(-__fmul_rn(sig, a.y), __fmul_rn(sig, a.x)), y);
}

__device__ __forceinline__ float2 half(int c, const float4 &f) { return c ? make_float2(f.z, f.w) : make_float2(f.x, f.y); }

// Store of a pair: both columns at once where both are in the grid.
__device__ __forceinline__ void st_pair(float2 *p, float2 a, float2 b, bool ina, bool inb)
{
    if (ina && inb) *reinterpret_cast<float4 *>(p) = make_float4(a.x, a.y, b.x, b.y);
    else if (ina) p[0] = a;
}
__device__ __forceinline__ void st_pair(__nv_bfloat162 *p, float2 a, float2 b, bool ina, bool inb)
{
    const __nv_bfloat162 ra = __float22bfloat162_rn(a), rb = __float22bfloat162_rn(b);
    if (ina && inb) {
        uint2 u;
        u.x = *reinterpret_cast<const unsigned *>(&ra);
        u.y = *reinterpret_cast<const unsigned *>(&rb);
        *reinterpret_cast<uint2 *>(p) = u;
    } else if (ina) {
        p[0] = ra;
    }
}

__device__ __forceinline__ bool is_real(float2 w, float ih2) { return w.x == ih2 && w.y == 0.f; }

struct Step2Args {
    float2 rho;
    float zy, sig1, sig2;        // shift s; sigma = i sig
    int rho_on;
};

template <typename S, int RX, bool REG>
__global__ void __launch_bounds__(kThreads2, 2) k_step3z2(Geom g, const float2 *__restrict__ coef, Step2Args sc,
                                                          const __grid_constant__ CUtensorMap mp,
                                                          const __grid_constant__ CUtensorMap my,
                                                          const __grid_constant__ CUtensorMap mk, S *pout, int64_t os1,
                                                          int64_t os2, int lz, unsigned *err)
{
    using G = Geo2<S, RX>;
    constexpr int L = RX / 2;                    // column pairs
    constexpr int TR = kThreads2 / L;            // thread rows
    constexpr int R = kRows / TR;                // rows per thread, TR apart
    constexpr int E = (int)sizeof(S) / 4;
    extern __shared__ unsigned char raw3[];
    __shared__ __align__(8) unsigned long long bar[kRing];
    unsigned char *stg = raw3 + ((128u - (smem_u32(raw3) & 127u)) & 127u);
    float2 *qb = reinterpret_cast<float2 *>(stg + kRing * G::STAGE);

    const int tid = threadIdx.x, lx = tid % L, ty = tid / L;
    const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2], nm = g.nmax;
    const int x0 = blockIdx.x * (RX - 4), y0 = blockIdx.y * (kRows - 2);    // output tile
    const int gx = x0 - 2 + 2 * lx;              // first of this thread's two columns
    const int z0 = blockIdx.z * lz, z1 = min(z0 + lz, n2);
    const int nload = z1 - z0 + 4;               // planes z0 - 2 .. z1 + 1

    auto issue = [&](int pi) {                   // plane z0 - 2 + pi into stage pi % kRing
        const int st = pi % kRing, z = z0 - 2 + pi;
        unsigned char *b = stg + st * G::STAGE;
        mbar_expect(&bar[st], (unsigned)G::TX);
        tma_load3(b, &mp, E * (x0 - 4), y0 - 2, z, &bar[st]);
        tma_load3(b + G::OY, &my, E * (x0 - 4), y0 - 1, z, &bar[st]);
        tma_load3(b + G::OK, &mk, x0 - 4, y0 - 1, z, &bar[st]);
    };
    if (tid == 0) {
        for (int s = 0; s < kRing; ++s)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bar[s])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    // per-column and per-row coefficients (constant along z)
    const int p0 = g.npml;
    const float ih2 = (float)g.ih2;
    float2 wpx[2], wmx[2], wcx[2], wpb[2], wmb[2], wpy[R], wmy[R], wxy[R][2];
    float mb[2], fb[2];
    bool xin[2], rowok[R], rowreal[R], yin[R], in[R][2];
    const bool xall = __all_sync(0xffffffffu, gx >= p0 && gx + 1 < n0 - p0);    // the warp outside the x PML
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int i = gx + c;
        xin[c] = i >= p0 && i < n0 - p0;
        wpx[c] = wmx[c] = wcx[c] = make_float2(0.f, 0.f);
        if (i >= 0 && i < n0) { wpx[c] = coef[i]; wmx[c] = coef[nm + i]; wcx[c] = coef[2 * nm + i]; }
        wpb[c] = xin[c] ? make_float2(1.f, 0.f) : wpx[c];
        wmb[c] = xin[c] ? make_float2(1.f, 0.f) : wmx[c];
        mb[c] = xin[c] ? 1.f : ih2;
        fb[c] = xin[c] ? ih2 : 1.f;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int j = y0 - 1 + ty + TR * r;
        const bool jin = j >= 0 && j < n1;
        float2 wcy = make_float2(0.f, 0.f);
        wpy[r] = wmy[r] = wcy;
        if (jin) { wpy[r] = coef[3 * nm + j]; wmy[r] = coef[4 * nm + j]; wcy = coef[5 * nm + j]; }
        yin[r] = j >= p0 && j < n1 - p0;
        rowok[r] = __all_sync(0xffffffffu, yin[r]);                             // the warp outside the y PML
        // its y coefficients are 1 / h^2 (the last one may keep a rounding error's imaginary part)
        rowreal[r] = __all_sync(0xffffffffu, yin[r] && is_real(wpy[r], ih2) && is_real(wmy[r], ih2));
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            in[r][c] = jin && gx + c >= 0 && gx + c < n0;
            wxy[r][c] = add_rn(wcx[c], wcy);
        }
    }
    // the next launch starts when this one no longer waits: released before the wait, a
    // third and a fourth would be resident too, unevenly spread (exp action on 24^3 3.66
    // and 3.44 ms, 28 x 14 x 12 3.55 and 3.43, 160^3 42.3 and 41.9)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (tid == 0)
        for (int pi = 0; pi < kRing && pi < nload; ++pi) issue(pi);

    // own columns: p(z-1), p(z), p(z+1); q(z-2), q(z-1); y and kappa of the previous plane
    float4 pm[R], pc[R], qm[R], qc[R], yprev[R];
    float2 kprev[R];
    bool ok = mbar_wait(&bar[0], 0) && mbar_wait(&bar[1], 0);
    const int own0 = (ty + 1) * G::W + 2 + 2 * lx, tile0 = ty * G::W + 2 + 2 * lx, q0 = ty * RX + 2 * lx;
    // edge threads of the region store no output: they read q in range and drop the result
    int qn[R];
    bool st0[R], st1[R];
    S *dst[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int row = ty + TR * r;
        pm[r] = ld_pair<S>(reinterpret_cast<const S *>(stg) + own0 + TR * r * G::W);
        pc[r] = ld_pair<S>(reinterpret_cast<const S *>(stg + G::STAGE) + own0 + TR * r * G::W);
        qm[r] = qc[r] = yprev[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        kprev[r] = make_float2(0.f, 0.f);
        const bool core = row >= 1 && row < kRows - 1 && lx >= 1 && lx < L - 1;
        qn[r] = core ? q0 + TR * r * RX : RX + 2;
        st0[r] = core && in[r][0];
        st1[r] = core && in[r][1];
        dst[r] = pout + gx + os1 * (y0 - 1 + row) + os2 * z0;
    }
    bool fail = __syncthreads_or(!ok) != 0;      // stage 0 is read
    int issued = min(nload, kRing);
    if (!fail && issued < nload) {
        if (tid == 0) issue(issued);
        ++issued;
    }
    // z coefficients of the plane before (for out) and of this one (for q)
    const float2 *cz = coef + 6 * nm;
    float2 bzp = make_float2(0.f, 0.f), bzm = bzp, bzc = bzp;
    bool zprev = false, zrprev = false;
    int cur = G::STAGE, nxt = 2 * G::STAGE;      // byte offsets of the stages of planes z and z + 1
    unsigned nbar = 2 % kRing, npar = 0;         // barrier and parity of plane z + 1
    int qcur = kRows * RX;                       // q(z) goes to qb + qcur, q(z - 1) is at the other half
    // twice: half of the register moves of the march (160^3: 24.5 us a step, rolled 27.1 us)
#pragma unroll 2
    for (int z = z0 - 1; z <= z1 && !fail; ++z) {
        ok = mbar_wait(&bar[nbar], npar);
        const S *ps = reinterpret_cast<const S *>(stg + cur) + own0, *pn = reinterpret_cast<const S *>(stg + nxt) + own0;
        const S *ys = reinterpret_cast<const S *>(stg + cur + G::OY) + tile0;
        const float *ks = reinterpret_cast<const float *>(stg + cur + G::OK) + tile0;
        float2 *qw = qb + qcur + q0;
        const float2 *qr = qb + (kRows * RX - qcur);
        const bool zok = z >= 0 && z < n2, zin = z >= p0 && z < n2 - p0, store = z > z0;
        const int zc = zok ? z : 0;
        const float2 czp = cz[zc], czm = cz[nm + zc], czc = cz[2 * nm + zc];
        const bool zreal = zin && is_real(czp, ih2) && is_real(czm, ih2);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int o = TR * r * G::W;
            const float4 pp = ld_pair<S>(pn + o), up = ld_pair<S>(ps + o + G::W), dn = ld_pair<S>(ps + o - G::W);
            const float2 lf = St<S>::ld(ps + o, -1), rt = St<S>::ld(ps + o, 2);
            const float4 yv = ld_pair<S>(ys + o);
            const float2 kv = *reinterpret_cast<const float2 *>(ks + o);
            // column c of the pair `mid` (own values), west / east: beyond the pair
            auto around = [](int c, const float4 &mid, float2 west, float2 east, const float4 &north, const float4 &south,
                             const float4 &above, const float4 &below) {
                Point3 n;
                n.pc = half(c, mid);
                n.xm = c ? half(0, mid) : west;
                n.xp = c ? east : half(1, mid);
                n.yp = half(c, north);
                n.ym = half(c, south);
                n.pp = half(c, above);
                n.pm = half(c, below);
                return n;
            };
            float2 q[2];
            if (xall && rowok[r] && zin) {
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const Point3 n = around(c, pc[r], lf, rt, up, dn, pp, pm[r]);
                    q[c] = rounded(finish(lap_inner(n, ih2), n.pc, add_rn(wxy[r][c], czc), c ? kv.y : kv.x, sc.zy, sc.sig1,
                                          half(c, yv)), S{});
                }
            } else if (rowreal[r] && zreal) {
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const Point3 n = around(c, pc[r], lf, rt, up, dn, pp, pm[r]);
                    q[c] = rounded(finish(lap_x<REG>(n, wpb[c], wmb[c], mb[c], fb[c]), n.pc, add_rn(wxy[r][c], czc),
                                          c ? kv.y : kv.x, sc.zy, sc.sig1, half(c, yv)), S{});
                    if (!in[r][c]) q[c] = make_float2(0.f, 0.f);
                }
            } else {
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const Point3 n = around(c, pc[r], lf, rt, up, dn, pp, pm[r]);
                    float2 lap = lap_general<REG>(n, Coef3{wpx[c], wmx[c], wpy[r], wmy[r], czp, czm});
                    if (zin && yin[r] && xin[c]) lap = lap_inner(n, ih2);
                    q[c] = rounded(finish(lap, n.pc, add_rn(wxy[r][c], czc), c ? kv.y : kv.x, sc.zy, sc.sig1, half(c, yv)),
                                   S{});
                    if (!(in[r][c] && zok)) q[c] = make_float2(0.f, 0.f);
                }
            }
            const float4 q4 = make_float4(q[0].x, q[0].y, q[1].x, q[1].y);
            *reinterpret_cast<float4 *>(qw + TR * r * RX) = q4;
            if (store) {                         // out(z - 1): the region without its edge
                const float2 *qs = qr + qn[r];
                const float4 qu = *reinterpret_cast<const float4 *>(qs + RX), qd = *reinterpret_cast<const float4 *>(qs - RX);
                const float2 ql = qs[-1], qe = qs[2];
                float2 v[2];
                if (xall && rowok[r] && zprev) {
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const Point3 n = around(c, qc[r], ql, qe, qu, qd, q4, qm[r]);
                        v[c] = finish(lap_inner(n, ih2), n.pc, add_rn(wxy[r][c], bzc), c ? kprev[r].y : kprev[r].x, sc.zy,
                                      sc.sig2, half(c, yprev[r]));
                    }
                } else if (rowreal[r] && zrprev) {
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const Point3 n = around(c, qc[r], ql, qe, qu, qd, q4, qm[r]);
                        v[c] = finish(lap_x<REG>(n, wpb[c], wmb[c], mb[c], fb[c]), n.pc, add_rn(wxy[r][c], bzc),
                                      c ? kprev[r].y : kprev[r].x, sc.zy, sc.sig2, half(c, yprev[r]));
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const Point3 n = around(c, qc[r], ql, qe, qu, qd, q4, qm[r]);
                        float2 lap = lap_general<REG>(n, Coef3{wpx[c], wmx[c], wpy[r], wmy[r], bzp, bzm});
                        if (zprev && yin[r] && xin[c]) lap = lap_inner(n, ih2);
                        v[c] = finish(lap, n.pc, add_rn(wxy[r][c], bzc), c ? kprev[r].y : kprev[r].x, sc.zy, sc.sig2,
                                      half(c, yprev[r]));
                    }
                }
                if (sc.rho_on) {
                    v[0] = mul0(sc.rho, v[0]);
                    v[1] = mul0(sc.rho, v[1]);
                }
                st_pair(dst[r], v[0], v[1], st0[r], st1[r]);
                dst[r] += os2;
            }
            qm[r] = qc[r];
            qc[r] = q4;
            pm[r] = pc[r];
            pc[r] = pp;
            yprev[r] = yv;
            kprev[r] = kv;
        }
        bzp = czp;
        bzm = czm;
        bzc = czc;
        zprev = zin;
        zrprev = zreal;
        fail = __syncthreads_or(!ok) != 0;       // q(z) is written, the stage of plane z is read
        if (!fail && issued < nload) {
            if (tid == 0) issue(issued);
            ++issued;
        }
        cur = nxt;
        nxt += G::STAGE;
        if (nxt == kRing * G::STAGE) nxt = 0;
        if (++nbar == kRing) {
            nbar = 0;
            npar ^= 1u;
        }
        qcur = kRows * RX - qcur;
    }
    // after a timeout: wait (bounded) for the loads still in flight
    if (fail && tid == 0) {
        atomicExch(err, 1u);
        for (int pi = max(0, issued - kRing); pi < issued; ++pi) mbar_wait(&bar[pi % kRing], (unsigned)(pi / kRing) & 1u);
    }
}

template <typename S, int RX, bool REG>
cudaError_t launch2(const Geom &g, const float2 *coef, const Step2Args &sc, const Tma3Maps &t, int ip, int iy, S *pout, int nseg, unsigned *err, cudaStream_t st, bool chain)
{
    using G = Geo2<S, RX>;
    constexpr int w = RX == 64;
    static std::atomic<bool> configured[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !configured[dev].load()) {
        const cudaError_t e = cudaFuncSetAttribute(k_step3z2<S, RX, REG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM);
        if (e != cudaSuccess) return e;
        configured[dev].store(true);
    }
    const int lz = (g.n[2] + nseg - 1) / nseg;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((g.n[0] + RX - 5) / (RX - 4), (g.n[1] + kRows - 3) / (kRows - 2), (g.n[2] + lz - 1) / lz);
    cfg.blockDim = dim3(kThreads2);
    cfg.dynamicSmemBytes = G::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = chain ? 1 : 0;
    count_launch();
    return cudaLaunchKernelEx(&cfg, k_step3z2<S, RX, REG>, g, coef, sc, t.p2[w][ip], t.y2[w][iy], t.k2[w], pout, (int64_t)t.pitch, (int64_t)t.pitch * g.n[1], lz, err);
}

// Region width and z segments that cost least: whole rounds of the blocks that are
// resident at once, each marching its segment plus four planes of lead-in, times the
// columns of a plane.
void shape2(const Geom &g, int *rx, int *nseg)
{
    double best = 1e300;
    for (int w : {32, 64}) {
        const int64_t bxy = (int64_t)((g.n[0] + w - 5) / (w - 4)) * ((g.n[1] + kRows - 3) / (kRows - 2));
        const int64_t slots = (int64_t)sm_count() * 2;
        for (int s = 1; s <= g.n[2] && s <= 64; ++s) {
            const int lz = (g.n[2] + s - 1) / s, segs = (g.n[2] + lz - 1) / lz;
            const double cost = (double)((bxy * segs + slots - 1) / slots) * (lz + 4) * w;
            if (cost < best) {
                best = cost;
                *rx = w;
                *nseg = segs;
            }
        }
    }
}

}  // namespace

template <typename S>
bool tma3_maps2(Tma3Maps *t, const Geom &g, void *const *bufs, const float *kappa)
{
    constexpr int E = TmaElt<S>::E;
    const int64_t row = (int64_t)t->pitch * E * 4, plane = row * g.n[1], krow = (int64_t)t->pitch * 4, kplane = krow * g.n[1];
    bool ok = true;
    for (int w = 0; w < 2 && ok; ++w) {
        const int cols = (w ? 64 : 32) + 4;
        for (int b = 0; b < 4 && ok; ++b)
            ok = tma3_encode(&t->p2[w][b], bufs[b], (int64_t)g.n[0] * E, g.n[1], g.n[2], row, plane, E * cols, kRows + 2) &&
                 tma3_encode(&t->y2[w][b], bufs[b], (int64_t)g.n[0] * E, g.n[1], g.n[2], row, plane, E * cols, kRows);
        ok = ok && tma3_encode(&t->k2[w], kappa, g.n[0], g.n[1], g.n[2], krow, kplane, cols, kRows);
    }
    return ok;
}

template <typename S>
cudaError_t launch_step3z2(const Geom &g, const float2 *coef, const StepScalars<float2> &s1, const StepScalars<float2> &s2,
                           const Tma3Maps *t, int ip, int iy, S *pout, unsigned *err, cudaStream_t st, bool chain)
{
    if (!t || !t->ok || ip < 0 || ip > 3 || iy < 0 || iy > 3) return cudaErrorInvalidValue;
    Step2Args sc;
    sc.rho = s2.rho;
    sc.zy = s1.zfac.y;
    sc.sig1 = s1.sigma.y;
    sc.sig2 = s2.sigma.y;
    sc.rho_on = !(s2.rho.x == 1.f && s2.rho.y == 0.f);
    int rx = 32, nseg = 1;
    shape2(g, &rx, &nseg);
    const bool reg = t->pitch != g.n[0];
    if (rx == 64)
        return reg ? launch2<S, 64, true>(g, coef, sc, *t, ip, iy, pout, nseg, err, st, chain)
                   : launch2<S, 64, false>(g, coef, sc, *t, ip, iy, pout, nseg, err, st, chain);
    return reg ? launch2<S, 32, true>(g, coef, sc, *t, ip, iy, pout, nseg, err, st, chain)
               : launch2<S, 32, false>(g, coef, sc, *t, ip, iy, pout, nseg, err, st, chain);
}

#define MXP_T2INST(S)                                                                                               \
    template bool tma3_maps2<S>(Tma3Maps *, const Geom &, void *const *, const float *);                            \
    template cudaError_t launch_step3z2<S>(const Geom &, const float2 *, const StepScalars<float2> &,               \
                                           const StepScalars<float2> &, const Tma3Maps *, int, int, S *,            \
                                           unsigned *, cudaStream_t, bool);
MXP_T2INST(float2)
MXP_T2INST(__nv_bfloat162)
#undef MXP_T2INST

}  // namespace mxp
