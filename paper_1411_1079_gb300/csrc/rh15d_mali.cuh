// rh15d_mali.cuh -- column-resident MALI kernel (Sect. 2.1-2.3, 3.1).
//
// One thread block owns one column at a time and runs all of that column's
// MALI iterations with the column's state in shared memory: populations
// (FP64), per-depth atmosphere scalars, and the rate accumulators.  When it takes a column, the block evaluates the line
// profiles of every line slot, ray and depth (they do not depend on the
// populations) into a per-block cache in global memory.  Per iteration:
//   1. warps take 32-wavelength tiles of the grid from a block-local queue;
//      each lane owns one wavelength and sweeps depth (linear short
//      characteristics; a tile and direction, all angles in one pass:
//      sweep_pairs in FP32, sweep_unit in FP64; with partial redistribution or
//      the Bezier solver a tile, one ray per pass: sweep_tile_k); at every
//      depth the lane forms its contributions to the preconditioned rate
//      matrix (Rybicki & Hummer 1992), the warp reduce-scatters them with
//      shuffles, and one lane per value holds the total for the tile's
//      accumulator;
//   2. the block sums the accumulators into each depth's rate matrix (FP64)
//      plus collisions, then one thread per depth solves the rate equations
//      (FP64, scaled unknowns, partial pivoting);
//   3. the block computes max |dn/n|, applies Ng order-2 acceleration
//      (history in global scratch) and tests convergence (Sect. 2.3).
// Columns come from a device work queue (pool mode, Sect. 3.1) or a static
// split over resident blocks (normal mode).  R is the precision of the
// formal solution and the rate terms (float or double); the rate matrix,
// the solve and Ng are always FP64.
#pragma once
#include <type_traits>

#include "rh15d_internal.h"
#include "rh15d_math64.h"

namespace rh {

namespace mali {

constexpr int kWarp = 32;
// Profile ring of the FP32 linear sweep with the profile cache: per warp, its
// tile's cached line profiles (every angle of the unit's direction) at
// kRingSlots depths -- the depth being swept and the next two -- copied from
// the cache by cp.async, so the HBM latency of a profile read is covered by
// two depth steps without holding the values in registers.
constexpr int kRingSlots = 3;
constexpr int kScratchUnit = 2304;              // granularity of the layout's scratch region, bytes
constexpr size_t kVtabBytes = sizeof(float4) * (RH_VT_N + 1);
constexpr int kNgLanes = 64;                    // fixed partition of the Ng dot products
constexpr int kRedDoubles = 5 * kNgLanes + 8;   // block reduction scratch

// constants of the packed sweep (fill_k2): operands of packed instructions
// come from the constant bank; as literals each use would be two moves
enum K2 { K2_ONE, K2_NEG, K2_WO, K2_E0 = K2_WO + 8, kNK2 = K2_E0 + 8 };

struct KParams {
    int64_t ncol;
    int N, L;
    const double *z, *T, *nH, *vz, *ne, *np, *nstar, *Crate;
    double *pops, *dmax;
    int32_t *iters;
    uint8_t *status;
    const void *lane;
    int npad;
    const float4 *vtab;
    double *nghist;
    int *queue;
    int persistent, maxiter, ng_order, ng_delay, ng_period, start;
    double tol, crsw, inv_nref;
    const int *colidx;         // work item -> column (nullptr: identity)
    int64_t nwork;
    const int *nwork_d;        // device count of work items (overrides nwork when set)
    // re-run ladder inside the kernel (Sect. 2.3): a column not converged
    // after its pass is restarted from LTE with switching factor rung_crsw[r],
    // Ng order rung_ng[r] and rung_maxiter iterations, r = 0 .. nrung-1
    int nrung, rung_maxiter;
    double rung_crsw[RH_MAX_RERUN];
    int rung_ng[RH_MAX_RERUN];
    int *rung_cols;                  // [nrung] columns entering each rung (nullptr: not counted)
    unsigned long long *rung_its;    // [1 + nrung] formal solutions of the pass and of each rung
    // partial redistribution
    double prd_eps0;
    int prd_hybrid;                  // 1: rho in the frame of the moving gas
    int formal;                      // formal solver: 0 linear, 1 quadratic Bezier short characteristics
    const int *lane_prd;
    const double *prd_nu, *prd_w;
    char *prd_scr;
    size_t prd_stride;               // bytes of scratch per block
    // profile cache (nullptr: the sweep evaluates the profiles itself)
    char *phic;
    size_t phic_stride;              // bytes of cache per block
    const double *tab64;             // FP64 function tables (rh15d_math64.h)
    // per-warp scratch of the sweep in the block's shared memory: piece bytes
    // a warp, the first nsp warps' in the accumulators' place (sweep_pairs with
    // the cache, which fills them after the sweep), the next nvp in the Voigt
    // table's place (only needed while the profiles are built), the others'
    // behind the layout
    int piece, nsp, nvp, scr[3];     // scr: byte offsets of the three places
    int slot_rows;                   // rows of the accumulator region
    int split;                       // 1: a tile's two directions are separate work items
    unsigned long long k2[kNK2];     // constants of the packed sweep, both halves alike (K2)
};

// Per-block PRD scratch: in R, the redistribution kernels K [sum np^2][N] (per
// line [k][j][i] = K_ij: transposed, so that the threads of a warp, which own
// consecutive points i, read consecutive addresses), then per PRD point
// [npp][N] the J-bar weights f, the mean intensity J, rho, D = dJ/drho (the
// derivative of J through the line's own emission) and the reduced frequency
// x of the point at each depth, per line [nprd][N] the damping a, then the
// plain-rate accumulators [pacc][N], the intensity of every ray at the PRD
// points [2 nmu][npp][N] (ray 2 m + d) followed by each ray's dI/drho there
// through the line's own emission [2 nmu][npp][N] (the hybrid scheme's
// gas-frame J and D are interpolated from them) and each ray's rho at the
// points [2 nmu][npp][N] (the hybrid scheme's gas-frame rho at the ray's
// gas-frame frequency, filled once per iteration), the hybrid scheme's
// interpolation tables of the column [2 nmu][npp][N] each (they depend on
// its velocities only; brackets as int in R-sized slots): for J_f at point
// i the bracket j and weight t of q_i + mu_z v_z and the weights e0, e1 of
// point i in the ray's rho at points j and j + 1, for the ray's rho at
// point p the bracket and weight of q_p - mu_z v_z; and the points'
// frequencies in velocity units c (nu - nu0) / nu0 [npp].  In FP64 the
// supply fraction F and J-bar per line [nprd][N], then the Ng history of rho
// [4][npp][N] (newest first).
template <typename R>
struct PrdScr {
    R *K, *f, *J, *rho, *D, *x, *a, *plain, *Iray, *ht, *he0, *he1, *rt, *q;
    int *hj, *rj;
    double *F, *Jbar, *hist;
};
template <typename R>
__host__ __device__ inline size_t prd_bytes(const DevAtom &A, int N)
{
    size_t r = sizeof(R) * ((size_t)A.prd_koff[A.nprd] * N + 5 * (size_t)A.npp * N + (size_t)A.nprd * N +
                            (size_t)A.pacc * N + 18 * (size_t)A.nmu * A.npp * N + (size_t)A.npp);
    r = (r + 255) & ~(size_t)255;
    r += sizeof(double) * (2 * (size_t)A.nprd * N + 4 * (size_t)A.npp * N) + 256;
    return (r + 255) & ~(size_t)255;   // every block's scratch 256-byte aligned (float4 loads of K)
}
// Per-block profile cache: the line profile phi (Voigt H(a, v) times its
// normalisation and 1/Doppler width, v including the ray's Doppler shift)
// of every line slot, direction (0 down, 1 up), depth, angle and lane in R
// (phi_block, phi_ray).  The profiles do
// not depend on the populations, so a column builds them once and every
// iteration reads them back instead of evaluating the Voigt function.
// Behind them, for the FP32 linear sweep, the warps' totals (pair_sums).
template <typename R>
__host__ __device__ inline size_t phic_bytes(const DevAtom &A, int N)
{
    const int even = (A.nmu + 1) / 2 * 2;        // FP32: pairs of angles
    size_t r = sizeof(R) * (size_t)A.nphi * 2 * (sizeof(R) == 4 ? even : A.nmu) * N * 32;
    if (sizeof(R) == 4 && !A.nprd) r += sizeof(R) * (size_t)even * A.macc * N;
    return (r + 255) & ~(size_t)255;
}

template <typename R>
__device__ inline PrdScr<R> prd_carve(char *base, const DevAtom &A, int N)
{
    PrdScr<R> q;
    R *r = reinterpret_cast<R *>(base);
    q.K = r;
    r += (size_t)A.prd_koff[A.nprd] * N;
    q.f = r;
    r += (size_t)A.npp * N;
    q.J = r;
    r += (size_t)A.npp * N;
    q.rho = r;
    r += (size_t)A.npp * N;
    q.D = r;
    r += (size_t)A.npp * N;
    q.x = r;
    r += (size_t)A.npp * N;
    q.a = r;
    r += (size_t)A.nprd * N;
    q.plain = r;
    r += (size_t)A.pacc * N;
    q.Iray = r;
    r += 6 * (size_t)A.nmu * A.npp * N;   // intensities, dI/drho, then rho per ray
    const size_t nt = 2 * (size_t)A.nmu * A.npp * N;
    q.hj = reinterpret_cast<int *>(r);
    r += nt;
    q.ht = r;
    r += nt;
    q.he0 = r;
    r += nt;
    q.he1 = r;
    r += nt;
    q.rj = reinterpret_cast<int *>(r);
    r += nt;
    q.rt = r;
    r += nt;
    q.q = r;
    r += (size_t)A.npp;
    size_t off = (reinterpret_cast<size_t>(r) + 255) & ~(size_t)255;
    q.F = reinterpret_cast<double *>(off);
    q.Jbar = q.F + (size_t)A.nprd * N;
    q.hist = q.Jbar + (size_t)A.nprd * N;
    return q;
}

template <typename R>
struct Smem {
    double *n, *nn;            // [L*N], [L*N]
    R *slot;                   // [macc][N] (x 2 with split directions)
    R *dz, *ivth, *vz;         // [N]
    R *bg;                     // [N][4]: h/kT, free-free, H- density, Thomson (one vector load per depth)
    R *Gc;                     // [ncont][N]
    R *ad;                     // [nline][N] damping
    R *nr;                     // [L][N] populations in R
    float4 *vtab;              // [RH_VT_N + 1] Voigt coefficient table
    double *red;               // reduction scratch [kRedDoubles]
    int *ibuf;                 // [8]
    char *base;                // of the whole layout (warp_scratch)
};

// Byte offsets of the regions of the block's dynamic shared memory.  The one
// function both sizes the allocation (host) and carves it (device), so the
// two cannot disagree: a layout whose carve ends past the allocated size
// (regions reserved by the carve but dropped from the size) writes outside
// the block's shared memory.
struct SmemLayout {
    size_t n, nn, Cr, red, slot, dz, ivth, vz, bg, Gc, ad, nr, vtab, ibuf, ring, end;
};
// ring_warps: units of kScratchUnit bytes of warp scratch behind the fixed regions
template <typename R>
__host__ __device__ inline SmemLayout smem_layout(int L, int N, int ntr, int ncont, int nline, int macc,
                                                  int ring_warps)
{
    SmemLayout o;
    size_t b = 0;
    o.n = b;
    b += sizeof(double) * (size_t)L * N;
    o.nn = b;
    b += sizeof(double) * (size_t)L * N;
    o.Cr = b;
    b += sizeof(double) * (size_t)N * 2 * ntr;
    o.red = b;
    b += sizeof(double) * kRedDoubles;
    o.slot = b;
    b += sizeof(R) * (size_t)macc * N;
    size_t *one[3] = {&o.dz, &o.ivth, &o.vz};
    for (int i = 0; i < 3; ++i) {
        *one[i] = b;
        b += sizeof(R) * (size_t)N;
    }
    b = (b + 15) & ~(size_t)15;                    // vector loads of the background block
    o.bg = b;
    b += sizeof(R) * 4 * (size_t)N;
    o.Gc = b;
    b += sizeof(R) * (size_t)ncont * N;
    o.ad = b;
    b += sizeof(R) * (size_t)nline * N;
    o.nr = b;
    b += sizeof(R) * (size_t)L * N;
    b = (b + 15) & ~(size_t)15;                    // float4 table: 16-byte aligned
    o.vtab = b;
    b += sizeof(float4) * (RH_VT_N + 1);
    o.ibuf = b;
    b += sizeof(int) * 8;
    b = (b + 15) & ~(size_t)15;
    o.ring = b;
    b += (size_t)kScratchUnit * ring_warps;
    o.end = b;
    return o;
}

template <typename R>
__host__ __device__ size_t smem_bytes(int L, int N, int ntr, int ncont, int nline, int macc, int ring_warps)
{
    return smem_layout<R>(L, N, ntr, ncont, nline, macc, ring_warps).end;
}

template <typename R>
__device__ Smem<R> carve(char *base, int L, int N, int ntr, int ncont, int nline, int macc, int ring_warps)
{
    const SmemLayout o = smem_layout<R>(L, N, ntr, ncont, nline, macc, ring_warps);
    Smem<R> s;
    s.n = reinterpret_cast<double *>(base + o.n);
    s.nn = reinterpret_cast<double *>(base + o.nn);
    s.red = reinterpret_cast<double *>(base + o.red);
    s.slot = reinterpret_cast<R *>(base + o.slot);
    s.dz = reinterpret_cast<R *>(base + o.dz);
    s.ivth = reinterpret_cast<R *>(base + o.ivth);
    s.vz = reinterpret_cast<R *>(base + o.vz);
    s.bg = reinterpret_cast<R *>(base + o.bg);
    s.Gc = reinterpret_cast<R *>(base + o.Gc);
    s.ad = reinterpret_cast<R *>(base + o.ad);
    s.nr = reinterpret_cast<R *>(base + o.nr);
    s.vtab = reinterpret_cast<float4 *>(base + o.vtab);
    s.ibuf = reinterpret_cast<int *>(base + o.ibuf);
    s.base = base;
    return s;
}

// warp w's scratch (KParams::piece), 16-byte aligned
template <typename R>
__device__ __forceinline__ char *warp_scratch(const Smem<R> &s, const KParams &p, int w)
{
    const int at = w < p.nsp ? p.scr[0] + w * p.piece
                   : w < p.nsp + p.nvp ? p.scr[1] + (w - p.nsp) * p.piece : p.scr[2] + (w - p.nsp - p.nvp) * p.piece;
    return s.base + at;
}

__device__ __forceinline__ float voigt(float a, float v, const float4 *tab, const double *) { return voigt_f32(a, v, tab); }
__device__ __forceinline__ double voigt(double a, double v, const float4 *, const double *tab64)
{
    double H, L;
    voigt64<false>(a, v, tab64, H, L);
    return H;
}

// 16-byte asynchronous global -> shared copy and its group fences (each
// thread waits for its own copies; __syncwarp makes them the warp's)
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Line profile phi(k, ray) of one wavelength: the Doppler shift of the ray,
// the Voigt function and the normalisation, with every rounding step fixed by
// intrinsics.  The cache build and the in-sweep evaluation both call this, and
// the compiler may not fuse or split its operations differently in the two
// places, so cached and uncached sweeps give the same bits.
__device__ __forceinline__ float line_phi(float q, float muz, float vz, float ivth, float a, float pn,
                                          const float4 *tab, const double *)
{
    const float v = __fmul_rn(__fmaf_rn(-muz, vz, q), ivth);
    return __fmul_rn(__fmul_rn(voigt_f32(a, v, tab), pn), ivth);
}
__device__ __forceinline__ double line_phi(double q, double muz, double vz, double ivth, double a, double pn,
                                           const float4 *, const double *tab64)
{
    const double v = __dmul_rn(__fma_rn(-muz, vz, q), ivth);
    return __dmul_rn(__dmul_rn(voigt(a, v, nullptr, tab64), pn), ivth);
}

template <typename R> __device__ __forceinline__ R rcp(R x);
template <> __device__ __forceinline__ float rcp<float>(float x) { return rcp_f32(x); }
template <> __device__ __forceinline__ double rcp<double>(double x) { return 1.0 / x; }

// 1 - exp(-x) for x > 0: FP32 uses 1 - __expf(-x) (x = h nu / kT > 0.1 on every grid here,
// relative error < 1e-6), FP64 expm1
template <typename R> __device__ __forceinline__ R one_m_exp(R x, R ex);
template <> __device__ __forceinline__ float one_m_exp<float>(float x, float ex) { return 1.0f - ex; }
template <> __device__ __forceinline__ double one_m_exp<double>(double x, double ex) { return -expm1(-x); }

template <typename R> __device__ __forceinline__ R rexp(R x);
template <> __device__ __forceinline__ float rexp<float>(float x) { return __expf(x); }
template <> __device__ __forceinline__ double rexp<double>(double x) { return exp(x); }

template <typename R> __device__ __forceinline__ R mu_of(const DevAtom &A, int m);
template <> __device__ __forceinline__ float mu_of<float>(const DevAtom &A, int m) { return A.muf[m]; }
template <> __device__ __forceinline__ double mu_of<double>(const DevAtom &A, int m) { return A.mu[m]; }
template <typename R> __device__ __forceinline__ R imu_of(const DevAtom &A, int m);
template <> __device__ __forceinline__ float imu_of<float>(const DevAtom &A, int m) { return A.imuf[m]; }
template <> __device__ __forceinline__ double imu_of<double>(const DevAtom &A, int m) { return A.imu[m]; }
// a product rounded on its own (never fused into a following addition)
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

template <typename R> __device__ __forceinline__ R wm2_of(const DevAtom &A, int m);
template <> __device__ __forceinline__ float wm2_of<float>(const DevAtom &A, int m) { return A.wm2f[m]; }
template <> __device__ __forceinline__ double wm2_of<double>(const DevAtom &A, int m) { return 0.5 * A.wmu[m]; }

// four consecutive values of a 16-byte aligned shared array
__device__ __forceinline__ void load4(const float *p, float &a, float &b, float &c, float &d)
{
    const float4 v = *reinterpret_cast<const float4 *>(p);
    a = v.x; b = v.y; c = v.z; d = v.w;
}
__device__ __forceinline__ void load4(const double *p, double &a, double &b, double &c, double &d)
{
    const double2 u = reinterpret_cast<const double2 *>(p)[0], v = reinterpret_cast<const double2 *>(p)[1];
    a = u.x; b = u.y; c = v.x; d = v.y;
}

// Per-lane constants of one tile with K transitions in its union.
template <typename R, int K>
struct LaneC {
    R c[K], Vc[K], Uc[K], E[K], q[K], pn[K], grat[K];
    int isline[K], lo[K], up[K], sub[K];
    R nu, nu3s, tw, hm;
};

// Depth-dependent, angle-independent quantities of one lane.
template <typename R, int K>
struct DepthC {
    R chibg, etabg, B, etac;
    R Rs[K], Xs[K], nu_[K], chc[K], Uct[K];
    R rf[K];                   // partial redistribution: psi/phi of the slot (1 otherwise)
};

template <typename R, int K, bool PRD = false>
__device__ __forceinline__ void depth_consts(const Smem<R> &s, const LaneC<R, K> &lc, int k, int N, DepthC<R, K> &d,
                                             R rho_k = (R)1, int prd_slot = -1)
{
    R hkT, kff, nhm, thom;
    load4(s.bg + 4 * k, hkT, kff, nhm, thom);
    R x = lc.nu * hkT;
    R ex = rexp<R>(-x);
    R omex = one_m_exp<R>(x, ex);
    d.chibg = (kff * lc.nu3s + nhm * lc.hm) * omex + thom;
    d.B = lc.tw * ex * rcp<R>(omex);
    d.etabg = d.chibg * d.B;
    d.etac = 0;
#pragma unroll
    for (int j = 0; j < K; ++j) {
        R nl = s.nr[lc.lo[j] * N + k];
        d.nu_[j] = s.nr[lc.up[j] * N + k];
        if (lc.isline[j]) {
            d.Rs[j] = lc.grat[j];
            if constexpr (PRD) {
                // psi = rho phi in stimulated and spontaneous emission
                d.rf[j] = j == prd_slot ? rho_k : (R)1;
                d.Rs[j] *= d.rf[j];
            }
            d.chc[j] = 0;
            d.Uct[j] = 0;
        } else {
            if constexpr (PRD) d.rf[j] = 1;
            d.Rs[j] = s.Gc[lc.sub[j] * N + k] * ex;
        }
        d.Xs[j] = nl - d.Rs[j] * d.nu_[j];
        if (!lc.isline[j]) {
            d.chc[j] = lc.Vc[j] * d.Xs[j];
            d.Uct[j] = lc.Uc[j] * d.Rs[j];
            d.etac += d.nu_[j] * d.Uct[j];
        }
    }
}

// Opacity and emissivity for one ray at one depth from the line profiles pc
// of its line slots; per-slot profile phi, opacity chj and emissivity per
// upper-level population U.
template <typename R, int K, bool PRD = false>
__device__ __forceinline__ void angle_vals(const LaneC<R, K> &lc, const DepthC<R, K> &d, const R (&pc)[K], R &chi,
                                           R &eta, R *phi, R *chj, R *U)
{
    chi = d.chibg;
    R ea = d.etac;
#pragma unroll
    for (int j = 0; j < K; ++j) {
        if (lc.isline[j]) {
            const R ph = pc[j];
            phi[j] = ph;
            chj[j] = lc.Vc[j] * ph * d.Xs[j];
            U[j] = lc.Uc[j] * ph;
            if constexpr (PRD) U[j] *= d.rf[j];
            ea += d.nu_[j] * U[j];
        } else {
            phi[j] = 1;
            chj[j] = d.chc[j];
            U[j] = d.Uct[j];
        }
        chi += chj[j];
    }
    eta = d.etabg + ea;
}

// Warp reduce-scatter of P values (P a power of two): afterwards every lane
// holds the warp total of value index lane >> (5 - log2 P).
template <int P, typename R>
__device__ __forceinline__ R reduce_scatter(R (&v)[P], int lane)
{
    int o = 16;
#pragma unroll
    for (int n = P; n > 1; n >>= 1) {
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
            R send = upper ? v[i] : v[i + n / 2];
            R keep = upper ? v[i + n / 2] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
        o >>= 1;
    }
    R r = v[0];
#pragma unroll
    for (; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
}

template <int M> struct Pow2 { static constexpr int v = M <= 1 ? 1 : (M <= 2 ? 2 : (M <= 4 ? 4 : (M <= 8 ? 8 : (M <= 16 ? 16 : 32)))); };
template <int P> struct Log2 { static constexpr int v = P <= 1 ? 0 : 1 + Log2<P / 2>::v; };
template <> struct Log2<1> { static constexpr int v = 0; };

// Planck terms of one wavelength at one depth: e^{-x}, 1 - e^{-x}
__device__ __forceinline__ void planck_terms(double x, const double *tab, double &ex, double &om)
{
    if (x < 0.5) {   // 1 - e^{-x} by expm1 where it would cancel
        om = -expm1(-x);
        ex = 1.0 - om;
    } else {
        ex = exp64(-x, tab);
        om = 1.0 - ex;
    }
}

// First element of the profile cache for cache row `row`, direction dir and
// depth k in the layout of sweep_unit, [row][dir][depth][angle][32 lanes].  (int: at most 288 rows x 2 x 4096 depths x 8 angles x 32
// lanes < 2^31)
__device__ __forceinline__ int phi_block(int nmu, int N, int row, int dir, int k)
{
    return ((row * 2 + dir) * N + k) * (nmu * kWarp);
}
// sweep_pairs: two angles interleaved, [row][dir][depth][pair][32 lanes][2], an
// odd last angle twice; first element of a row and direction.
__device__ __forceinline__ int phi_pairs(int np, int N, int row, int dir) { return (row * 2 + dir) * N * np * 2 * kWarp; }

// The kernels of sweep_tile_k walk one ray at a time and keep a ray's depths
// together: [row][dir][angle][depth][32 lanes]; first element of a ray.
__device__ __forceinline__ int phi_ray(int nmu, int N, int row, int dir, int m)
{
    return ((row * 2 + dir) * nmu + m) * N * kWarp;
}

// Depth-dependent, angle-independent quantities of one lane (NL lines first,
// then NC continua).
template <int K, int NL>
struct DepthV {
    static constexpr int NC = K - NL;
    double chi0, eta0, etabg, B;             // background + continua; background; Planck function
    double X[K], Rs[K];                      // n_l - R n_u, R
    double A[NL ? NL : 1], El[NL ? NL : 1];  // line opacity and emissivity per profile
    double Ut[NC ? NC : 1], oc[NC ? NC : 1]; // continuum U; opacity of the other continua and the background
};

template <int K, int NL>
__device__ __forceinline__ void depth_terms(const Smem<double> &s, const LaneC<double, K> &lc, const double *tab, int k,
                                            int N, DepthV<K, NL> &d)
{
    constexpr int NC = K - NL;
    double hkT, kff, nhm, thom, ex, om;
    load4(s.bg + 4 * k, hkT, kff, nhm, thom);
    planck_terms(lc.nu * hkT, tab, ex, om);
    const double chibg = (kff * lc.nu3s + nhm * lc.hm) * om + thom;
    d.B = lc.tw * ex * rcp64(om);
    d.etabg = chibg * d.B;
    d.chi0 = chibg;
    d.eta0 = d.etabg;
    double ch[NC ? NC : 1];
#pragma unroll
    for (int j = 0; j < K; ++j) {
        const double nl = s.nr[lc.lo[j] * N + k], nu = s.nr[lc.up[j] * N + k];
        if (j < NL) {
            d.Rs[j] = lc.grat[j];
            d.X[j] = nl - d.Rs[j] * nu;
            d.A[j] = lc.Vc[j] * d.X[j];
            d.El[j] = lc.Uc[j] * nu;
        } else {
            d.Rs[j] = s.Gc[lc.sub[j] * N + k] * ex;
            d.X[j] = nl - d.Rs[j] * nu;
            ch[j - NL] = lc.Vc[j] * d.X[j];
            d.Ut[j - NL] = lc.Uc[j] * d.Rs[j];
            d.chi0 += ch[j - NL];
            d.eta0 += nu * d.Ut[j - NL];
        }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        d.oc[c] = chibg;
#pragma unroll
        for (int c2 = 0; c2 < NC; ++c2)
            if (c2 != c) d.oc[c] += ch[c2];
    }
}

// Sums over the rays of one depth (w the ray's weight w_mu/2, phi 1 for a
// continuum, Psi = Psi* per unit emissivity, q = 1 - Psi* chi of the whole
// opacity, o_j the opacity of everything but transition j):
//   P_l = sum w phi_l I_eff, F_l = sum w phi_l (q + Psi o_l), S_l = sum w phi_l Psi (lines)
//   T_ll' = sum w Psi phi_l phi_l'   (pairs of lines)
//   Pc = sum w I_eff, Fc = sum w (q + Psi chi_lines), S0 = sum w Psi (shared by the continua:
//   o_c - chi_lines does not depend on the angle).
// The constants of the wavelength (c_j, R_j, E_j, X_j, U factors) multiply
// the sums once per depth instead of every ray's terms; with
//   up_j = c_j P_j, down_j = c_j R_j (E_j F_j + P_j), cross_jj' = c_j X_j U_j' (sum)
// all terms of the sums are positive, nothing nearly equal is subtracted.
// FP64 only: phi I_eff of a wing below a cold temperature minimum leaves the
// FP32 range before c_j brings it back.
template <int NL, int NC>
struct RaySums {
    static constexpr int NT = NL * (NL - 1) / 2;
    double P[NL ? NL : 1], F[NL ? NL : 1], S[NL ? NL : 1], T[NT ? NT : 1], Pc, Fc, S0;
};

// One unit of the FP64 sweep: tile b (K transitions in its union, the first NL
// of them lines) in one direction (dir 0 down, 1 up), every angle in one pass
// over depth, so the depth terms and the warp's reductions are paid once per
// depth and direction.  One lane = one wavelength.  At each depth the lane
// forms the rays' sums above and from them its contributions to the
// preconditioned rate matrix; the warp sums them over its wavelengths and
// lane a writes accumulator a.  The rays' states are in the warp's shared
// scratch (registers would not hold all rays).  Bound by the FP64 pipe (150
// columns x 3 iterations, profiles included: 371 -> 42 ms against one angle
// pair per pass with the library's exponentials and divisions).
template <int K, int NL, bool CACHE>
__device__ void sweep_unit(const DevAtom &A, const Smem<double> &s, const KParams &p, int b, int dir, double *slot,
                           bool add, int lane, const double *phc)
{
    constexpr int NC = K - NL;
    const int N = p.N, nmu = A.nmu, npad = p.npad, pi = b * kWarp + lane;
    const DevTile &tl = A.tile[b];
    const double *lt = reinterpret_cast<const double *>(p.lane);
    const double *tab = p.tab64;
    LaneC<double, K> lc;
    int poff[NL ? NL : 1];                       // first cache element of each line slot, this direction
#pragma unroll
    for (int j = 0; j < K; ++j) {
        const DevTrans &tr = A.tr[tl.t[j]];
        lc.c[j] = lt[(RH_NLANEF * j + 0) * npad + pi];
        lc.Vc[j] = lt[(RH_NLANEF * j + 1) * npad + pi];
        lc.Uc[j] = lt[(RH_NLANEF * j + 2) * npad + pi];
        lc.E[j] = lt[(RH_NLANEF * j + 3) * npad + pi];
        if (!CACHE) {
            lc.q[j] = lt[(RH_NLANEF * j + 4) * npad + pi];
            lc.pn[j] = lt[(RH_NLANEF * j + 5) * npad + pi];
        }
        if (j < NL) {
            lc.grat[j] = lt[(RH_NLANEF * j + 6) * npad + pi];
            poff[j] = CACHE ? phi_block(nmu, N, tl.phi[j], dir, 0) : 0;
        }
        lc.lo[j] = tr.l;
        lc.up[j] = tr.u;
        lc.sub[j] = tr.sub;
    }
    lc.nu = lt[kLaneNu * npad + pi];
    lc.hm = lt[kLaneHm * npad + pi];
    lc.nu3s = lt[kLaneNu3 * npad + pi];
    lc.tw = lt[kLaneTw * npad + pi];

    constexpr int M = K * (K + 1);
    constexpr int P = Pow2<M>::v;
    constexpr int SH = 5 - Log2<P>::v;
    const bool writer = (lane & ((1 << SH) - 1)) == 0;
    const int widx = lane >> SH;
    // ray m's I, chi and S of the upwind point at st[0], st[kWarp], st[2 kWarp]
    double *rays = reinterpret_cast<double *>(warp_scratch(s, p, threadIdx.x >> 5)) + lane;
    const int blk = nmu * kWarp;

    auto phi_at = [&](int j, int m, int k) -> double {
        if constexpr (CACHE) return phc[poff[j] + k * blk + m * kWarp + lane];
        else
            return line_phi(lc.q[j], dir ? A.mu[m] : -A.mu[m], s.vz[k], s.ivth[k], s.ad[lc.sub[j] * N + k], lc.pn[j],
                            s.vtab, tab);
    };
    RaySums<NL, NC> rs;
    auto zero = [&]() {
#pragma unroll
        for (int j = 0; j < NL; ++j) rs.P[j] = rs.F[j] = rs.S[j] = 0.0;
#pragma unroll
        for (int j = 0; j < RaySums<NL, NC>::NT; ++j) rs.T[j] = 0.0;
        rs.Pc = rs.Fc = rs.S0 = 0.0;
    };
    // opacity and emissivity of a ray; ls: the lines' part of the opacity
    auto opac = [&](const DepthV<K, NL> &d, const double (&ph)[NL ? NL : 1], double &chi, double &eta, double &ls) {
        eta = d.eta0;
        if constexpr (NL == 0) {
            chi = d.chi0;
        } else {
            if constexpr (NC > 0 || NL > 1) {
                ls = d.A[0] * ph[0];
#pragma unroll
                for (int j = 1; j < NL; ++j) ls = fma(d.A[j], ph[j], ls);
                chi = NL == 1 ? fma(d.A[0], ph[0], d.chi0) : d.chi0 + ls;
            } else {
                chi = fma(d.A[0], ph[0], d.chi0);
            }
#pragma unroll
            for (int j = 0; j < NL; ++j) eta = fma(d.El[j], ph[j], eta);
        }
    };
    // a ray's terms of the sums
    auto accumulate = [&](const DepthV<K, NL> &d, const double (&ph)[NL ? NL : 1], double w, double ls, double q,
                          double psi, double Ieff) {
        if constexpr (NC > 0) {
            rs.Pc = fma(w, Ieff, rs.Pc);
            rs.Fc = fma(w, NL > 0 ? fma(psi, ls, q) : q, rs.Fc);
            rs.S0 = fma(w, psi, rs.S0);
        }
#pragma unroll
        for (int j = 0; j < NL; ++j) {
            const double wp = w * ph[j];
            double o = d.chi0;
            int t = 0;
#pragma unroll
            for (int a = 0; a < NL; ++a)
#pragma unroll
                for (int c = a + 1; c < NL; ++c, ++t) {
                    if (a == j) o = fma(d.A[c], ph[c], o);
                    if (c == j) o = fma(d.A[a], ph[a], o);
                    if (a == j) rs.T[t] = fma(wp * psi, ph[c], rs.T[t]);
                }
            rs.P[j] = fma(wp, Ieff, rs.P[j]);
            rs.F[j] = fma(wp, fma(psi, o, q), rs.F[j]);
            if constexpr (NC > 0) rs.S[j] = fma(wp, psi, rs.S[j]);
        }
    };
    // the lane's contributions from the sums, summed over the warp
    auto flush = [&](const DepthV<K, NL> &d, int k) {
        double val[P], Pj[K];
#pragma unroll
        for (int a = M; a < P; ++a) val[a] = 0;
#pragma unroll
        for (int j = 0; j < K; ++j) {
            double Fj;
            if (j < NL) {
                Pj[j] = rs.P[j];
                Fj = rs.F[j];
            } else {
                Pj[j] = rs.Pc;
                Fj = rs.Fc + d.oc[j - NL] * rs.S0;
            }
            val[j] = lc.c[j] * Pj[j];
            val[K + j] = lc.c[j] * d.Rs[j] * (lc.E[j] * Fj + Pj[j]);
        }
#pragma unroll
        for (int j = 0; j < K; ++j)
#pragma unroll
            for (int j2 = 0; j2 < K; ++j2) {
                if (j2 == j) continue;
                const int lo = j < j2 ? j : j2, hi = j < j2 ? j2 : j;
                double x;
                if (hi < NL) x = rs.T[lo * NL - lo * (lo + 1) / 2 + hi - lo - 1];
                else if (lo < NL) x = rs.S[lo];
                else x = rs.S0;
                const double u = j2 < NL ? lc.Uc[j2] : d.Ut[j2 - NL < 0 ? 0 : j2 - NL];
                val[2 * K + j * (K - 1) + (j2 < j ? j2 : j2 - 1)] = lc.c[j] * x * d.X[j] * u;
            }
        const double t = reduce_scatter<P>(val, lane);
        if (writer && widx < M) {
            double *o = slot + widx * N + k;
            *o = add ? *o + t : t;
        }
    };
    // ---- boundary point: I = 0 at the top; at the bottom the diffusion
    // condition, which needs chi and B one point up
    const int k0 = dir == 0 ? 0 : N - 1;
    DepthV<K, NL> d2, d;
    if (dir == 1) depth_terms<K, NL>(s, lc, tab, N - 2, N, d2);
    depth_terms<K, NL>(s, lc, tab, k0, N, d);
    zero();
    for (int m = 0; m < nmu; ++m) {
        double ph[NL ? NL : 1], chi, eta, ls = 0.0, ch2 = 0.0, I = 0.0;
        if (dir == 1) {
#pragma unroll
            for (int j = 0; j < NL; ++j) ph[j] = phi_at(j, m, N - 2);
            opac(d2, ph, ch2, eta, ls);
        }
#pragma unroll
        for (int j = 0; j < NL; ++j) ph[j] = phi_at(j, m, k0);
        opac(d, ph, chi, eta, ls);
        if (dir == 1)   // B + mu (B - B2) / dtau = B + (B - B2) / (dtau / mu)
            I = fma(d.B - d2.B, rcp64((chi + ch2) * s.dz[N - 2] * (0.5 * A.imu[m])), d.B);
        double *st = rays + (size_t)m * 3 * kWarp;
        st[0] = I;
        st[kWarp] = chi;
        st[2 * kWarp] = eta * rcp64(chi);
        accumulate(d, ph, wm2_of<double>(A, m), ls, 1.0, 0.0, I);
    }
    flush(d, k0);
    for (int step = 1; step < N; ++step) {
        const int k = dir == 0 ? step : N - 1 - step;
        depth_terms<K, NL>(s, lc, tab, k, N, d);
        const double dzk = dir == 0 ? s.dz[k - 1] : s.dz[k];
        zero();
        for (int m = 0; m < nmu; ++m) {
            double ph[NL ? NL : 1];
#pragma unroll
            for (int j = 0; j < NL; ++j) ph[j] = phi_at(j, m, k);
            double *st = rays + (size_t)m * 3 * kWarp;
            double chi, eta, ls = 0.0, e, wu, wo, q;
            opac(d, ph, chi, eta, ls);
            const double ic = rcp64(chi), S = eta * ic;
            sc64((chi + st[kWarp]) * (0.5 * A.imu[m] * dzk), tab, e, wu, wo, q);
            const double base = fma(st[0], e, wu * st[2 * kWarp]), psi = wo * ic;
            st[0] = fma(wo, S, base);
            st[kWarp] = chi;
            st[2 * kWarp] = S;
            accumulate(d, ph, wm2_of<double>(A, m), ls, q, psi, fma(psi, d.etabg, base));
        }
        flush(d, k);
    }
}

// Rate contributions of one ray at one depth point (see sweep_pairs)
template <typename R, int K, int P>
__device__ __forceinline__ void ray_rates(const LaneC<R, K> &lc, const DepthC<R, K> &d, const R (&phi)[K],
                                          const R (&chj)[K], const R (&U)[K], R ichi, R wo, R omwo, R psi, R Ieff,
                                          R wm2, R (&val)[P])
{
#pragma unroll
    for (int j = 0; j < K; ++j) {
        R other = d.chibg;
#pragma unroll
        for (int j2 = 0; j2 < K; ++j2)
            if (j2 != j) other += chj[j2];
        const R f = omwo + wo * other * ichi;          // 1 - Psi* chi_j
        const R cw = lc.c[j] * wm2 * phi[j];
        val[j] = cw * Ieff;
        val[K + j] = cw * d.Rs[j] * (lc.E[j] * f + Ieff);
        const R cx = cw * d.Xs[j] * psi;
#pragma unroll
        for (int j2 = 0; j2 < K; ++j2)
            if (j2 != j) val[2 * K + j * (K - 1) + (j2 < j ? j2 : j2 - 1)] = cx * U[j2];
    }
}

// Per-lane constants of tile b
template <typename R, int K>
__device__ __forceinline__ void load_lane(const DevAtom &A, const KParams &p, int b, int lane, LaneC<R, K> &lc)
{
    const R *lt = reinterpret_cast<const R *>(p.lane);
    const int npad = p.npad, pi = b * kWarp + lane;
#pragma unroll
    for (int j = 0; j < K; ++j) {
        const DevTrans &tr = A.tr[A.tile[b].t[j]];
        lc.c[j] = lt[(RH_NLANEF * j + 0) * npad + pi];
        lc.Vc[j] = lt[(RH_NLANEF * j + 1) * npad + pi];
        lc.Uc[j] = lt[(RH_NLANEF * j + 2) * npad + pi];
        lc.E[j] = lt[(RH_NLANEF * j + 3) * npad + pi];
        lc.q[j] = lt[(RH_NLANEF * j + 4) * npad + pi];
        lc.pn[j] = lt[(RH_NLANEF * j + 5) * npad + pi];
        lc.grat[j] = lt[(RH_NLANEF * j + 6) * npad + pi];
        lc.isline[j] = tr.kind == 0;
        lc.lo[j] = tr.l;
        lc.up[j] = tr.u;
        lc.sub[j] = tr.sub;
    }
    lc.nu = lt[kLaneNu * npad + pi];
    lc.hm = lt[kLaneHm * npad + pi];
    lc.nu3s = lt[kLaneNu3 * npad + pi];
    lc.tw = lt[kLaneTw * npad + pi];
}

// ---- the FP32 linear sweep ---------------------------------------------------
// Two rays (two angles) in a register pair: one packed instruction does both,
// so the sweep, which is bound by instruction issue, issues half as many.
// Each half rounds as the scalar operation would.
struct f2 {
    unsigned long long u;
};
__device__ __forceinline__ f2 pk(float lo, float hi)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.u) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ f2 splat(float x) { return pk(x, x); }
__device__ __forceinline__ void upk(f2 a, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.u));
}
__device__ __forceinline__ f2 vfma(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.u) : "l"(a.u), "l"(b.u), "l"(c.u));
    return r;
}
__device__ __forceinline__ f2 vmul(f2 a, f2 b)
{
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u));
    return r;
}
__device__ __forceinline__ f2 vadd(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u));
    return r;
}
// A product that keeps its rounding: the assembler fuses a packed product into
// a packed sum that is its only use, in spite of both instructions' .rn; it
// leaves scalar products alone.
__device__ __forceinline__ f2 vmul_rn(f2 a, f2 b)
{
    float a0, a1, b0, b1;
    upk(a, a0, a1);
    upk(b, b0, b1);
    return pk(__fmul_rn(a0, b0), __fmul_rn(a1, b1));
}
__device__ __forceinline__ f2 vrcp(f2 a)
{
    float lo, hi;
    upk(a, lo, hi);
    return pk(rcp_f32(lo), rcp_f32(hi));
}

// Operations of both rays with one factor or term in common: two scalar
// instructions, since a packed one would need that value in both halves of a
// register pair first.
__device__ __forceinline__ f2 smul(float x, f2 a)
{
    float a0, a1;
    upk(a, a0, a1);
    return pk(__fmul_rn(a0, x), __fmul_rn(a1, x));
}
__device__ __forceinline__ f2 sadd(float x, f2 a)
{
    float a0, a1;
    upk(a, a0, a1);
    return pk(__fadd_rn(a0, x), __fadd_rn(a1, x));
}
__device__ __forceinline__ f2 sfma(float x, f2 a, f2 c)
{
    float a0, a1, c0, c1;
    upk(a, a0, a1);
    upk(c, c0, c1);
    return pk(__fmaf_rn(x, a0, c0), __fmaf_rn(x, a1, c1));
}
__device__ __forceinline__ f2 sfma(float x, f2 a, float c)
{
    float a0, a1;
    upk(a, a0, a1);
    return pk(__fmaf_rn(x, a0, c), __fmaf_rn(x, a1, c));
}

// x z of the first ray + x z of the second
__device__ __forceinline__ float vdot(f2 x, f2 z)
{
    float x0, x1, z0, z1;
    upk(x, x0, x1);
    upk(z, z0, z1);
    return __fmaf_rn(x1, z1, __fmul_rn(x0, z0));
}

// Linear short-characteristics weights of a pair, e^{-d}, w_u, w_o and 1 -
// w_o, to the bit those of sc_weights.  Both of its forms are evaluated and
// selected per ray, without a branch: the rays of a warp straddle d = 1/2 at
// most depths, and a straight line of packed instructions costs less than the
// divergent branch.
__device__ __forceinline__ void vsc(const KParams &kp, f2 d, f2 &e, f2 &wu, f2 &wo, f2 &omwo)
{
    auto C = [&](int i) { return f2{kp.k2[i]}; };
    const f2 one = C(K2_ONE), neg = C(K2_NEG), nd = vmul(d, neg);
    f2 w = C(K2_WO + 7), q = C(K2_E0 + 7);
#pragma unroll
    for (int i = 6; i >= 0; --i) {
        w = vfma(d, w, C(K2_WO + i));
        q = vfma(d, q, C(K2_E0 + i));
    }
    const f2 wos = vmul(w, d), nwo = vmul_rn(w, nd), wus = vfma(d, q, nwo), oms = vadd(nwo, one), es = vfma(nd, q, one);
    float d0, d1;
    upk(d, d0, d1);
    const f2 ex = pk(__expf(-d0), __expf(-d1));
    const f2 oml = vmul(vfma(ex, neg, one), pk(rcp_f32(d0), rcp_f32(d1)));
    const f2 wol = vfma(oml, neg, one), wul = vfma(ex, neg, oml);
    const bool s0 = d0 < 0.5f, s1 = d1 < 0.5f;
    auto sel = [&](f2 a, f2 b) {
        float a0, a1, b0, b1;
        upk(a, a0, a1);
        upk(b, b0, b1);
        return pk(s0 ? a0 : b0, s1 ? a1 : b1);
    };
    e = sel(es, ex);
    wu = sel(wus, wul);
    wo = sel(wos, wol);
    omwo = sel(oms, oml);
}

// Where the sums of opacities round a transition's opacity on its own (bit j:
// slot j) instead of fusing its last product into the sum: in chi and in the
// opacity of the other transitions at a depth step, in chi at the first point
// of a ray and at the point next to it that the diffusion condition reads; and
// whether the emissivity at the first point fuses chi_bg B.  Any choice is as
// accurate; these are kept because they have always been these kernels' (see
// sweep_pairs).
template <int K, int NL>
struct Unfused {
    static constexpr int step = K == 2 ? 2 : K == 3 && NL == 3 ? 6 : K == 3 && NL == 2 ? 2 : 0;
    static constexpr int other = K == 2 && NL == 0 ? 0 : step;
    static constexpr int first = K == 3 ? 6 : K == 2 ? 2 : 0;
    static constexpr int next = K == 2 && NL == 0 ? 0 : K == 3 && NL == 1 ? 6 : step;
    static constexpr bool eta_first = NL == 0;
};

// Depth-dependent, angle-independent quantities of one lane (the first NL
// transitions lines, the others continua)
template <int K>
struct DepthF {
    float chibg, etabg, B, etac;
    float Rs[K], X[K], nu[K], chc[K], Uct[K];   // R, n_l - R n_u, n_u, continuum opacity, continuum U
};
template <int K, int NL>
__device__ __forceinline__ void depth_f(const Smem<float> &s, const LaneC<float, K> &lc, int k, int N, DepthF<K> &d)
{
    float hkT, kff, nhm, thom;
    load4(s.bg + 4 * k, hkT, kff, nhm, thom);
    const float ex = __expf(-__fmul_rn(lc.nu, hkT)), om = __fsub_rn(1.0f, ex);   // h nu / kT > 0.1 on every grid
    d.chibg = __fmaf_rn(__fmaf_rn(kff, lc.nu3s, __fmul_rn(nhm, lc.hm)), om, thom);
    d.B = __fmul_rn(__fmul_rn(lc.tw, ex), rcp_f32(om));
    d.etabg = __fmul_rn(d.chibg, d.B);
    d.etac = 0.0f;
#pragma unroll
    for (int j = 0; j < K; ++j) {
        const float nl = s.nr[lc.lo[j] * N + k];
        d.nu[j] = s.nr[lc.up[j] * N + k];
        d.Rs[j] = j < NL ? lc.grat[j] : __fmul_rn(s.Gc[lc.sub[j] * N + k], ex);
        d.X[j] = __fmaf_rn(-d.Rs[j], d.nu[j], nl);
        if (j >= NL) {
            d.chc[j] = __fmul_rn(lc.Vc[j], d.X[j]);
            d.Uct[j] = __fmul_rn(lc.Uc[j], d.Rs[j]);
            d.etac = __fmaf_rn(d.nu[j], d.Uct[j], d.etac);
        }
    }
}

// Floats of a warp's scratch: the profile ring, [slot][line][pair][64] (CACHE),
// the rays' I, chi and S, [pair][3][64], and the pairs' weights and 1/mu.
__host__ __device__ inline int pairs_scratch(const DevAtom &A, bool cache)
{
    const int np = (A.nmu + 1) / 2;
    return (cache ? kRingSlots * A.maxnl * np * 2 * kWarp : 0) + np * 3 * 2 * kWarp + 16;
}

// The FP32 sweep of tile b (K transitions in its union, the first NL of them
// lines) in direction dir (0 down, 1 up), the angle pairs v0 .. v1 - 1 in one
// pass over depth, so the depth terms are paid once for all of them.  One lane
// = one wavelength.  At each depth the lane forms, without subtracting nearly
// equal numbers,
//   I_eff = I - Psi* eta_active = I_u e^{-dtau} + w_u S_u + w_o eta_bg/chi,
//   1 - Psi* chi_j = (1 - w_o) + w_o (chi - chi_j)/chi,
// and the contributions of a pair's two rays (weight w = w_mu/2):
//   up_j = (c_j w phi_j) I_eff,  down_j = (c_j w phi_j) R_j (E_j (1 - Psi* chi_j) + I_eff),
//   cross_{j,j'} = c_j X_j w phi_j Psi* U_j';
// the warp sums them over its wavelengths and gives the total of each of the
// M = K (K + 1) values, of every pair for itself, to one lane, which hands it
// on (out(total, value, pair, depth)).
// Every operation's rounding is spelled out, and the pairs' totals are added
// in the order (pair, direction).  Two reasons: c_j (1e23) meets phi_j (down
// to 1e-18) before I_eff (1e-30 below a cold temperature minimum) does, which
// keeps every term in the FP32 range; and a few columns in 65536 lie so near a
// singular rate matrix that another rounding of one iteration moves the
// iteration at which their populations fail.  The results are, to the bit,
// those of a pass per pair and direction with each term added to a tile's one
// accumulator, whatever the launch shape and with or without the cache.
// The loop over pairs is not unrolled (ray states in shared memory, the first
// point in the same loop): the blocks of an SM sweep tiles of different types
// side by side, and unrolled the nine bodies exceed the instruction cache.
// Per column-iteration (82 depths, 608 wavelengths, 5 angles; 16384 columns to
// 1e-3): scalar passes of two angles, both directions in one warp, 3.20 us;
// unrolled 3.80; rolled 2.97; with 128 depths 6.27 -> 4.09.  (Sums over all
// rays before the constants, one warp reduction per depth, took 1.79 us, but
// lose the up-rates of columns colder than 2450 K and move 12 of 65536
// columns: withdrawn.)  Bound by instruction issue and latency at 16 warps an
// SM: the reductions of every pair, both forms of the weights, index
// arithmetic.
template <int K, int NL, bool CACHE, typename Out>
__device__ __forceinline__ void sweep_pairs(const DevAtom &A, const Smem<float> &s, const KParams &p, int b, int dir,
                                            int v0, int v1, int lane, const float *phc, Out out)
{
    typedef Unfused<K, NL> UF;
    const int N = p.N, nmu = A.nmu, np = (nmu + 1) / 2;
    const DevTile &tl = A.tile[b];
    LaneC<float, K> lc;
    load_lane<float, K>(A, p, b, lane, lc);
    constexpr int NLA = NL ? NL : 1;
    constexpr int M = K * (K + 1), P = Pow2<M>::v, SH = 5 - Log2<P>::v;
    const bool writer = (lane & ((1 << SH) - 1)) == 0;
    const int widx = lane >> SH;
    constexpr bool RING = CACHE && NL > 0;
    const int blk = np * 2 * kWarp;              // floats of a line's profiles at one depth
    float *ring = reinterpret_cast<float *>(warp_scratch(s, p, threadIdx.x >> 5));
    float *rays = ring + (CACHE ? kRingSlots * A.maxnl * blk : 0) + 2 * lane;
    // weights and 1/mu of every pair (0 beyond an odd number of angles)
    unsigned long long *wi = reinterpret_cast<unsigned long long *>(rays - 2 * lane + np * 3 * 2 * kWarp);
    if (lane < np) {
        wi[2 * lane] = pk(A.wm2f[2 * lane], A.wm2f[2 * lane + 1]).u;
        wi[2 * lane + 1] = pk(A.imuf[2 * lane], A.imuf[2 * lane + 1]).u;
    }
    __syncwarp();
    struct Vals {
        f2 chi, eta, t[NLA], ch[NLA], U[NLA];    // opacity, emissivity; per line Vc phi, its opacity and U
    };
    auto vals = [&](const DepthF<K> &d, const f2 (&ph)[NLA], int mask, Vals &y, bool first) {
        if constexpr (NL == 0) {                 // the same for every ray
            float chi = d.chibg;
#pragma unroll
            for (int j = 0; j < K; ++j)
                chi = mask >> j & 1 ? __fadd_rn(chi, d.chc[j]) : __fmaf_rn(lc.Vc[j], d.X[j], chi);
            y.chi = splat(chi);
            y.eta = splat(first && UF::eta_first ? __fmaf_rn(d.chibg, d.B, d.etac) : __fadd_rn(d.etabg, d.etac));
        } else {
            f2 ea;
#pragma unroll
            for (int j = 0; j < K; ++j) {
                if (j < NL) {
                    const int l = j < NL ? j : 0;
                    y.t[l] = smul(lc.Vc[j], ph[l]);
                    y.ch[l] = smul(d.X[j], y.t[l]);
                    y.U[l] = smul(lc.Uc[j], ph[l]);
                    if (j == 0) {
                        ea = sfma(d.nu[j], y.U[l], d.etac);
                        y.chi = mask & 1 ? sadd(d.chibg, y.ch[l]) : sfma(d.X[j], y.t[l], d.chibg);
                    } else {
                        ea = sfma(d.nu[j], y.U[l], ea);
                        y.chi = mask >> j & 1 ? vadd(y.chi, y.ch[l]) : sfma(d.X[j], y.t[l], y.chi);
                    }
                } else {
                    float c0, c1;
                    upk(y.chi, c0, c1);
                    y.chi = mask >> j & 1 ? sadd(d.chc[j], y.chi)
                                          : pk(__fmaf_rn(lc.Vc[j], d.X[j], c0), __fmaf_rn(lc.Vc[j], d.X[j], c1));
                }
            }
            y.eta = sadd(d.etabg, ea);
        }
    };
    // contributions of a pair, summed over the warp
    auto rates = [&](const DepthF<K> &d, const f2 (&ph)[NLA], const Vals &y, f2 ichi, f2 wo, f2 omwo, f2 psi, f2 Ieff,
                     f2 wv) {
        float val[P];
#pragma unroll
        for (int a = M; a < P; ++a) val[a] = 0;
#pragma unroll
        for (int j = 0; j < K; ++j) {
            f2 other;
            float oc = d.chibg;                  // until a line comes in, the same for both rays
            bool vec = false;
#pragma unroll
            for (int q = 0; q < K; ++q) {
                if (q == j) continue;
                constexpr int mask = UF::other;
                const int l = q < NL ? q : 0;
                if (q < NL) {
                    if (!vec) other = mask >> q & 1 ? sadd(oc, y.ch[l]) : sfma(d.X[q], y.t[l], oc);
                    else other = mask >> q & 1 ? vadd(other, y.ch[l]) : sfma(d.X[q], y.t[l], other);
                    vec = true;
                } else if (vec) {
                    float c0, c1;
                    upk(other, c0, c1);
                    other = mask >> q & 1 ? sadd(d.chc[q], other)
                                          : pk(__fmaf_rn(lc.Vc[q], d.X[q], c0), __fmaf_rn(lc.Vc[q], d.X[q], c1));
                } else {
                    oc = mask >> q & 1 ? __fadd_rn(oc, d.chc[q]) : __fmaf_rn(lc.Vc[q], d.X[q], oc);
                }
            }
            const f2 f = vfma(vec ? vmul(wo, other) : smul(oc, wo), ichi, omwo);          // 1 - Psi* chi_j
            f2 cw = smul(lc.c[j], wv);
            if (j < NL) cw = vmul(cw, ph[j < NL ? j : 0]);
            const f2 cr = smul(d.Rs[j], cw), cx = vmul(smul(d.X[j], cw), psi);
            val[j] = vdot(cw, Ieff);
            val[K + j] = vdot(cr, sfma(lc.E[j], f, Ieff));
#pragma unroll
            for (int q = 0; q < K; ++q)
                if (q != j) {
                    float &o = val[2 * K + j * (K - 1) + (q < j ? q : q - 1)];
                    if (q < NL) {
                        o = vdot(cx, y.U[q < NL ? q : 0]);
                    } else {
                        float x0, x1;
                        upk(cx, x0, x1);
                        o = __fmaf_rn(x1, d.Uct[q], __fmul_rn(x0, d.Uct[q]));
                    }
                }
        }
        return reduce_scatter<P>(val, lane);
    };
    // The points in the order they are met: down 0, 1, .. N - 1; up N - 2 (for
    // the diffusion condition at the bottom, B and chi), N - 1, N - 2, .. 0.
    const int pts = N + dir, lead = dir;         // points before the ray's first one
    auto depth_of = [&](int st) { return dir == 0 ? st : (st == 0 ? N - 2 : N - st); };
    // profile ring: the copies of a point go into slot (point mod 3), issued two
    // points ahead (one commit group per point, empty past the end)
    int fst = 0, foff = 0, roff = 0;             // the next point to copy, its ring offset; the offset being read
    const int rstride = A.maxnl * blk, w16 = (v1 - v0) * 16;
    auto ring_fill = [&]() {
        if constexpr (RING) {
            if (fst < pts) {
                const int o = depth_of(fst) * blk + v0 * 2 * kWarp + 4 * lane;
                float *dst = ring + foff + v0 * 2 * kWarp + 4 * lane;
#pragma unroll
                for (int j = 0; j < NL; ++j) {   // pairs x 64 values: at most two 16-byte pieces a lane
                    const float *src = phc + phi_pairs(np, N, tl.phi[j], dir) + o;
                    if (lane < w16) cp_async16(dst + j * blk, src);
                    if (lane + kWarp < w16) cp_async16(dst + j * blk + 4 * kWarp, src + 4 * kWarp);
                }
            }
            cp_async_commit();
            ++fst;
            foff = foff == 2 * rstride ? 0 : foff + rstride;
        }
    };
    ring_fill();
    ring_fill();
    float B2 = 0.0f;
    for (int st = 0; st < pts; ++st) {
        const int k = depth_of(st);
        const float *rg = nullptr;
        if constexpr (RING) {
            cp_async_wait<1>();
            __syncwarp();
            rg = ring + roff + 2 * lane;
            ring_fill();   // into the slot read one point ago
            roff = roff == 2 * rstride ? 0 : roff + rstride;
        }
        DepthF<K> d;
        depth_f<K, NL>(s, lc, k, N, d);
        const float hz = 0.5f * (dir == 0 ? s.dz[k > 0 ? k - 1 : 0] : s.dz[k]);
#pragma unroll 1
        for (int v = v0; v < v1; ++v) {
            const int m = 2 * v;                 // beyond an odd number of angles: weight 0, mu 0, the profile of m
            f2 ph[NLA];
#pragma unroll
            for (int j = 0; j < NL; ++j) {
                if constexpr (RING) {
                    ph[j].u = *reinterpret_cast<const unsigned long long *>(rg + j * blk + v * 2 * kWarp);
                } else {
                    const int m2 = m + 1 < nmu ? m + 1 : m;
                    const float a = s.ad[lc.sub[j] * N + k];
                    ph[j] = pk(line_phi(lc.q[j], dir ? A.muf[m] : -A.muf[m], s.vz[k], s.ivth[k], a, lc.pn[j], s.vtab, p.tab64),
                               line_phi(lc.q[j], dir ? A.muf[m2] : -A.muf[m2], s.vz[k], s.ivth[k], a, lc.pn[j], s.vtab, p.tab64));
                }
            }
            f2 *r = reinterpret_cast<f2 *>(rays + v * 3 * 2 * kWarp);        // I, chi, S of the upwind point
            Vals y;
            f2 ichi, wo, omwo, psi, Ieff;
            if (st <= lead) {
                if (st < lead) {
                    vals(d, ph, UF::next, y, false);
                    r[kWarp] = y.chi;
                    B2 = d.B;
                    continue;
                }
                // the ray's first point: I = 0 at the top, the diffusion condition at the bottom
                vals(d, ph, UF::first, y, true);
                ichi = vrcp(y.chi);
                Ieff = splat(0.0f);
                if (dir == 1)
                    Ieff = vfma(vmul(pk(A.muf[m], A.muf[m + 1]), splat(__fsub_rn(d.B, B2))),
                                vrcp(vmul(vmul(splat(0.5f), vadd(y.chi, r[kWarp])), splat(s.dz[N - 2]))), splat(d.B));
                wo = psi = splat(0.0f);
                omwo = splat(1.0f);
                r[0] = Ieff;
                r[2 * kWarp] = vmul(y.eta, ichi);
            } else {
                f2 e, wu;
                vals(d, ph, UF::step, y, false);
                ichi = vrcp(y.chi);
                const f2 S = vmul(y.eta, ichi);
                vsc(p, vmul(smul(hz, vadd(y.chi, r[kWarp])), f2{wi[2 * v + 1]}), e, wu, wo, omwo);
                const f2 base = vfma(wu, r[2 * kWarp], vmul(r[0], e));
                r[0] = vfma(wo, S, base);
                r[2 * kWarp] = S;
                psi = vmul(wo, ichi);
                Ieff = vfma(wo, smul(d.etabg, ichi), base);
            }
            r[kWarp] = y.chi;
            const float t = rates(d, ph, y, ichi, wo, omwo, psi, Ieff, f2{wi[2 * v]});
            if (writer && widx < M) out(t, widx, v, k);
        }
    }
    if constexpr (RING) {
        cp_async_wait<0>();
        __syncwarp();
    }
}

// The sweep with partial redistribution (PRD) or the Bezier solver (BEZ): one
// tile (K transitions in its union, their kinds read at run time), downward
// and upward, one angle per pass over depth; the contributions are those of
// sweep_pairs.
// PRD: the tile's PRD slot emits with psi = rho phi (rho of the lane's point
// and depth from the block's scratch), PRD lanes accumulate the angle-averaged
// mean intensity J, and every slot also accumulates its plain rates (actual
// intensity) cw I and cw R (E + I), for the PRD update.
// prd_I (hybrid PRD only, else nullptr): the rays' intensities at the PRD
// points and then their dI/drho, written here, and then the rays' rho,
// read here.
template <typename R, int K, bool PRD, bool BEZ>
__device__ void sweep_tile_k(const DevAtom &A, const Smem<R> &s, const KParams &p, int b, R *slot, int lane,
                             R *prd_rho, R *prd_J, R *prd_D, R *prd_plain, R *prd_I, const R *phc)
{
    const int N = p.N;
    const DevTile &tl = A.tile[b];
    const int nmu = A.nmu;
    const int pi = b * kWarp + lane;
    LaneC<R, K> lc;
    load_lane<R, K>(A, p, b, lane, lc);
    // cached line profiles of the current ray at depth k for the tile's line
    // slots (0 elsewhere)
    int pb[K];                                     // the ray's first element of each line slot's cache rows
    auto load_ph = [&](int k, R (&o)[K]) {
#pragma unroll
        for (int j = 0; j < K; ++j) {
            if (!lc.isline[j]) o[j] = 0;
            else o[j] = phc[pb[j] + k * kWarp];
        }
    };
    constexpr int M = K * (K + 1);
    constexpr int MP = PRD ? M + 2 * K : M;        // with the plain rates
    constexpr int P = Pow2<MP>::v;
    constexpr int SH = 5 - Log2<P>::v;
    const bool writer = (lane & ((1 << SH) - 1)) == 0;
    const int widx = lane >> SH;
    int pp = -1;                                   // PRD point of the lane
    const R *rho_lane = nullptr;
    R *plain = nullptr;
    constexpr bool bez = BEZ;                      // quadratic Bezier formal solver
    bool hyb = false;                              // hybrid PRD at this lane
    if constexpr (PRD) {
        pp = tl.prd_slot >= 0 ? p.lane_prd[pi] : -1;
        rho_lane = pp >= 0 ? prd_rho + (size_t)pp * N : nullptr;
        plain = prd_plain + (size_t)tl.pacc_off * N;
        hyb = prd_I != nullptr && pp >= 0;
    }

    // contributions of one depth point to the tile's accumulators
    auto emit = [&](int k, const DepthC<R, K> &d, const R (&phi)[K], const R (&chj)[K], const R (&U)[K], R ichi,
                    R wo, R omwo, R psi, R Ieff, R Ik, R wm2, int ray) {
        R val[P];
        ray_rates<R, K, P>(lc, d, phi, chj, U, ichi, wo, omwo, psi, Ieff, wm2, val);
        if constexpr (PRD) {
#pragma unroll
            for (int j = 0; j < K; ++j) {
                const R cw = lc.c[j] * wm2 * phi[j];
                val[M + 2 * j] = cw * Ik;
                val[M + 2 * j + 1] = cw * d.Rs[j] * (lc.E[j] + Ik);
            }
            // fire-and-forget reductions (zeroed before the sweep): one lane per
            // location, adding in program order, so the sum is deterministic;
            // D = dJ/drho through the PRD line's own emission, Psi* n_u U0.
            // Hybrid PRD: the ray's I and dI/drho at the point instead, for
            // the gas-frame J and D of the rho update
            if (pp >= 0) {
                R e0 = 0;
#pragma unroll
                for (int j = 0; j < K; ++j)
                    if (j == tl.prd_slot) e0 = d.nu_[j] * lc.Uc[j] * phi[j];
                if (hyb) {
                    const size_t ri = ((size_t)ray * A.npp + pp) * N + k;
                    prd_I[ri] = Ik;
                    prd_I[ri + 2 * (size_t)A.nmu * A.npp * N] = psi * e0;
                } else {
                    atomicAdd(prd_J + (size_t)pp * N + k, wm2 * Ik);
                    atomicAdd(prd_D + (size_t)pp * N + k, wm2 * (psi * e0));
                }
            }
        }
#pragma unroll
        for (int a = MP; a < P; ++a) val[a] = 0;
        const R t = reduce_scatter<P>(val, lane);
        if (writer && widx < M) slot[widx * N + k] += t;   // zeroed before the sweep
        if constexpr (PRD) {
            if (writer && widx >= M && widx < MP) atomicAdd(plain + (widx - M) * N + k, t);
        }
    };

    for (int m = 0; m < nmu; ++m) {
        const R mu = mu_of<R>(A, m), imu = imu_of<R>(A, m), wm2 = wm2_of<R>(A, m);
        for (int dir = 0; dir < 2; ++dir) {
            const R muz = dir == 0 ? -mu : mu;
            const int ray = 2 * m + dir;
#pragma unroll
            for (int j = 0; j < K; ++j)
                pb[j] = lc.isline[j] ? phi_ray(nmu, N, tl.phi[j], dir, m) + lane : 0;
            R I, chip = 0, Sp;
            // rho of the lane's PRD point: the static-frame ratio, or (hybrid)
            // this ray's interpolated gas-frame ratio
            const R *rl = hyb ? prd_I + ((4 * (size_t)A.nmu + ray) * A.npp + pp) * N : rho_lane;
            {
                R pc[K];
                // boundary point: I = 0 at the top; at the bottom the diffusion
                // condition, which needs chi and B one point up
                const int k0 = dir == 0 ? 0 : N - 1;
                R B2 = 0;
                if (dir == 1) {
                    DepthC<R, K> d2;
                    depth_consts<R, K, PRD>(s, lc, N - 2, N, d2, rl ? rl[N - 2] : (R)1, tl.prd_slot);
                    B2 = d2.B;
                    R phi[K], chj[K], U[K], eta;
                    load_ph(N - 2, pc);
                    angle_vals<R, K, PRD>(lc, d2, pc, chip, eta, phi, chj, U);
                }
                DepthC<R, K> d;
                depth_consts<R, K, PRD>(s, lc, k0, N, d, rl ? rl[k0] : (R)1, tl.prd_slot);
                R chi, eta, phi[K], chj[K], U[K];
                load_ph(k0, pc);
                angle_vals<R, K, PRD>(lc, d, pc, chi, eta, phi, chj, U);
                const R ichi = rcp<R>(chi);
                if (dir == 0) {
                    I = 0;
                } else {
                    R dtv = (R)0.5 * (chi + chip) * s.dz[N - 2];
                    I = d.B + mu * (d.B - B2) * rcp<R>(dtv);
                }
                chip = chi;
                Sp = eta * ichi;
                emit(k0, d, phi, chj, U, ichi, (R)0, (R)1, (R)0, I, I, wm2, ray);
            }
            // rho of the lane's PRD point (global scratch) loaded one depth step ahead
            R rho_nx = (PRD && rl) ? rl[dir == 0 ? 1 : N - 2] : (R)1;
            // cached profiles, like rho, loaded one depth step ahead
            R pa[K];
            load_ph(dir == 0 ? 1 : N - 2, pa);
            for (int step = 1; step < N; ++step) {
                const int k = dir == 0 ? step : N - 1 - step;
                const bool has_d = step + 1 < N;   // a downwind point
                const R rho_k = rho_nx;
                if (PRD && rl && has_d) rho_nx = rl[dir == 0 ? step + 1 : N - 2 - step];
                R na[K];
                load_ph(has_d ? (dir == 0 ? k + 1 : k - 1) : k, na);
                // the profiles three depths on into L1: one step of look-ahead
                // does not cover their HBM latency
                if (BEZ && step + 3 < N) {
#pragma unroll
                    for (int j = 0; j < K; ++j)
                        if (lc.isline[j])
                            asm volatile("prefetch.global.L1 [%0];" ::"l"(phc + pb[j] + (dir == 0 ? k + 3 : k - 3) * kWarp));
                }
                // quadratic Bezier step: the downwind point's opacity and source
                // function first (its profiles and rho are the ones loaded for
                // the next step), so that its depth terms are dead before the
                // point's own are formed
                R chid = 0, Sd = 0;
                if (bez && has_d) {   // BEZ kernels only
                    DepthC<R, K> dd;
                    depth_consts<R, K, PRD>(s, lc, dir == 0 ? k + 1 : k - 1, N, dd, rho_nx, tl.prd_slot);
                    R etad, phid[K], chjd[K], Ud[K];
                    angle_vals<R, K, PRD>(lc, dd, na, chid, etad, phid, chjd, Ud);
                    Sd = etad * rcp<R>(chid);
                }
                DepthC<R, K> d;
                depth_consts<R, K, PRD>(s, lc, k, N, d, rho_k, tl.prd_slot);
                R chi, eta, phi[K], chj[K], U[K];
                angle_vals<R, K, PRD>(lc, d, pa, chi, eta, phi, chj, U);
                const R ichi = rcp<R>(chi);
                const R S = eta * ichi;
                const R dzk = dir == 0 ? s.dz[k - 1] : s.dz[k];
                const R dtau = (R)0.5 * (chi + chip) * dzk * imu;
                R Ieff, psi, wo, omwo;
                if (bez) {
                    const R dtd = has_d ? (R)0.5 * (chid + chi) * (dir == 0 ? s.dz[k] : s.dz[k - 1]) * imu : (R)1;
                    R ex, wu, wob, wc, omp;
                    bez_weights(dtau, ex, wu, wob, wc, omp);
                    const R C = bez_control<R>(Sp, S, Sd, dtau, dtd, has_d);
                    const R base = I * ex + wu * Sp + wc * (C - S);
                    wo = wob + wc;                 // Psi* = w_o + w_c
                    omwo = omp;
                    I = base + wo * S;
                    Ieff = base + wo * (d.etabg * ichi);
                } else {
                    R ome, wu;
                    sc_weights(dtau, ome, wu, wo, omwo);
                    const R base = I * ome + wu * Sp;
                    I = base + wo * S;
                    Ieff = base + wo * (d.etabg * ichi);
                }
                psi = wo * ichi;
#pragma unroll
                for (int j = 0; j < K; ++j) pa[j] = na[j];
                chip = chi;
                Sp = S;
                emit(k, d, phi, chj, U, ichi, wo, omwo, psi, Ieff, I, wm2, ray);
            }
        }
    }
}

// The warps' totals of the FP32 linear sweep (with the profile cache), behind
// the block's profiles: [pair][direction][depth][accumulator].  Kept apart, the
// tiles' directions are independent work items (20 tiles on 8 warps: 5 rounds
// of one direction instead of 3 of both) and all angles go in one pass, and
// still the sum is taken in the order of a pass per pair and direction.
__device__ __forceinline__ float *pair_sums(const DevAtom &A, const KParams &p, float *phc)
{
    return phc + (size_t)A.nphi * 2 * ((A.nmu + 1) / 2 * 2) * p.N * kWarp;
}
__device__ __forceinline__ void sum_pairs(const DevAtom &A, const KParams &p, const float *g, float *slot)
{
    const int n = A.macc * p.N, nq = (A.nmu + 1) / 2 * 2;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        float s = g[i];
#pragma unroll 4
        for (int q = 1; q < nq; ++q) s = __fadd_rn(s, g[(size_t)q * n + i]);
        slot[i % A.macc * p.N + i / A.macc] = s;
    }
}

// Work item q of the sweep: a tile, in one direction (split: sweep_unit and
// the cached sweep_pairs) or in both.
template <typename R, bool PRD, bool CACHE, bool BEZ>
__device__ __forceinline__ void sweep_item(const DevAtom &A, const Smem<R> &s, const KParams &p, int q, int lane,
                                           R *prd_rho, R *prd_J, R *prd_D, R *prd_plain, R *prd_I, R *phc)
{
    const int b = A.order[p.split ? q >> 1 : q];
    const DevTile &tl = A.tile[b];
    const int d0 = p.split ? q & 1 : 0, d1 = p.split ? d0 + 1 : 2;
    R *slot = s.slot + (size_t)tl.acc_off * p.N;
    if constexpr (PRD || BEZ) {
        // (with the kinds at compile time the nine tile bodies of the PRD
        // kernels cost more in instruction fetches than they save, 3.2 -> 4.8
        // ms an iteration of 304 columns)
        switch (tl.K) {
        case 1: sweep_tile_k<R, 1, PRD, BEZ>(A, s, p, b, slot, lane, prd_rho, prd_J, prd_D, prd_plain, prd_I, phc); break;
        case 2: sweep_tile_k<R, 2, PRD, BEZ>(A, s, p, b, slot, lane, prd_rho, prd_J, prd_D, prd_plain, prd_I, phc); break;
        default: sweep_tile_k<R, 3, PRD, BEZ>(A, s, p, b, slot, lane, prd_rho, prd_J, prd_D, prd_plain, prd_I, phc); break;
        }
    } else {
        auto tile = [&](auto k_, auto nl_) {
            constexpr int K = decltype(k_)::value, NL = decltype(nl_)::value;
            if constexpr (sizeof(R) == 8) {
                for (int dir = d0; dir < d1; ++dir)
                    sweep_unit<K, NL, CACHE>(A, s, p, b, dir, slot + (p.split && dir ? (size_t)A.macc * p.N : 0),
                                             !p.split && dir, lane, phc);
            } else if constexpr (CACHE) {
                // a pass's totals, kept apart until every unit is done (sum_pairs)
                float *g = pair_sums(A, p, phc) + tl.acc_off;
                sweep_pairs<K, NL, CACHE>(A, s, p, b, d0, 0, (A.nmu + 1) / 2, lane, phc,
                                          [&](float t, int a, int v, int k) {
                    g[((2 * v + d0) * p.N + k) * A.macc + a] = t;
                });
            } else {
                for (int v = 0; 2 * v < A.nmu; ++v)
                    for (int dir = 0; dir < 2; ++dir)
                        sweep_pairs<K, NL, CACHE>(A, s, p, b, dir, v, v + 1, lane, phc, [&](float t, int a, int, int k) {
                            slot[a * p.N + k] = __fadd_rn(slot[a * p.N + k], t);   // zeroed before the sweep
                        });
            }
        };
#define RH_TILE(K_, NL_) tile(std::integral_constant<int, K_>(), std::integral_constant<int, NL_>())
        switch (tl.K * 4 + tl.nl) {
        case 4: RH_TILE(1, 0); break;
        case 5: RH_TILE(1, 1); break;
        case 8: RH_TILE(2, 0); break;
        case 9: RH_TILE(2, 1); break;
        case 10: RH_TILE(2, 2); break;
        case 12: RH_TILE(3, 0); break;
        case 13: RH_TILE(3, 1); break;
        case 14: RH_TILE(3, 2); break;
        default: RH_TILE(3, 3); break;
        }
#undef RH_TILE
    }
}

// Hybrid PRD tables.  Interpolation over PRD line [off, last] (points sorted
// by frequency q, velocity units) at x: the bracket j in [off, last - 1] and
// weight t on point j + 1, value (1 - t) v_j + t v_{j+1}; beyond the ends
// the end value, (off, 0) or (last - 1, 1).
template <typename R>
__device__ __forceinline__ void prd_bracket(const R *qv, int off, int last, R x, int &j, R &t)
{
    if (x <= qv[off]) {
        j = off;
        t = 0;
    } else if (x >= qv[last]) {
        j = last - 1;
        t = 1;
    } else {
        int lo = off, hi = last;                   // qv[lo] <= x < qv[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (qv[mid] <= x) lo = mid;
            else hi = mid;
        }
        j = lo;
        t = (x - qv[lo]) / (qv[lo + 1] - qv[lo]);
    }
}

// weight of point i in the interpolation at x
template <typename R>
__device__ __forceinline__ R prd_weight(const R *qv, int off, int last, int i, R x)
{
    int j;
    R t;
    prd_bracket<R>(qv, off, last, x, j, t);
    return (j == i ? (R)1 - t : (R)0) + (j + 1 == i ? t : (R)0);
}

// the column's tables: threads take (ray, point, depth)
template <typename R>
__device__ void build_hybrid_tables(const DevAtom &A, const Smem<R> &s, const PrdScr<R> &ps, int N)
{
    const int nw = 2 * A.nmu * A.npp * N;
    for (int e = threadIdx.x; e < nw; e += blockDim.x) {
        const int k = e % N, rp = e / N, pt = rp % A.npp, ray = rp / A.npp;
        int q = 0;
        while (pt >= A.prd_off[q + 1]) ++q;
        const int off = A.prd_off[q], last = A.prd_off[q + 1] - 1;
        const R mu = mu_of<R>(A, ray >> 1), muz = (ray & 1) ? mu : -mu, sh = muz * s.vz[k];
        int j;
        R t;
        prd_bracket<R>(ps.q, off, last, ps.q[pt] + sh, j, t);
        ps.hj[e] = j;
        ps.ht[e] = t;
        ps.he0[e] = prd_weight<R>(ps.q, off, last, pt, ps.q[j] - sh);
        ps.he1[e] = prd_weight<R>(ps.q, off, last, pt, ps.q[j + 1] - sh);
        prd_bracket<R>(ps.q, off, last, ps.q[pt] - sh, j, t);
        ps.rj[e] = j;
        ps.rt[e] = t;
    }
}

// Hybrid PRD: each ray's rho at the PRD points, the gas-frame rho_f at the
// ray's gas-frame frequency q_p - mu_z v_z, for the sweep to read like the
// static-frame rho; threads take (ray, point, depth)
template <typename R>
__device__ void fill_rho_ray(const DevAtom &A, const PrdScr<R> &ps, int N)
{
    const int nw = 2 * A.nmu * A.npp * N;
    R *out = ps.Iray + 4 * (size_t)A.nmu * A.npp * N;
    for (int e = threadIdx.x; e < nw; e += blockDim.x) {
        const int k = e % N, j = ps.rj[e];
        const R t = ps.rt[e];
        out[e] = ((R)1 - t) * ps.rho[(size_t)j * N + k] + t * ps.rho[(size_t)(j + 1) * N + k];
    }
}

// Hybrid PRD: the gas-frame mean intensity and its local derivative at every
// PRD point and depth (threads take (point, depth)),
//   J_f(i) = sum over rays (w_mu/2) [(1 - t) I_j + t I_{j+1}],
//   D_f(i) = sum over rays (w_mu/2) [(1 - t) dI_j e0 + t dI_{j+1} e1],
// rays in the order the sweep adds the static-frame J, each product rounded
// before its sum as the sweep's accumulation does
template <typename R>
__device__ void hybrid_JD(const DevAtom &A, const PrdScr<R> &ps, int N)
{
    const size_t nt = (size_t)A.npp * N, nr = 2 * (size_t)A.nmu;
    for (int e = threadIdx.x; e < (int)nt; e += blockDim.x) {
        const int k = e % N;
        R J = 0, D = 0;
        for (int ray = 0; ray < (int)nr; ++ray) {
            const R w = wm2_of<R>(A, ray >> 1);
            const size_t x = (size_t)ray * nt + e;
            const int j = ps.hj[x];
            const R t = ps.ht[x];
            const R *Ir = ps.Iray + (size_t)ray * nt + k, *Dr = Ir + nr * nt;
            const R v = ((R)1 - t) * Ir[(size_t)j * N] + t * Ir[(size_t)(j + 1) * N];
            const R dv = ((R)1 - t) * Dr[(size_t)j * N] * ps.he0[x] + t * Dr[(size_t)(j + 1) * N] * ps.he1[x];
            J += mul_rn(w, v);
            D += mul_rn(w, dv);
        }
        ps.J[e] = J;
        ps.D[e] = D;
    }
}

// Fill the column's profile cache: warps take (row, direction, quarter of the
// depths), lanes their wavelengths (the same arithmetic as the uncached sweep).
template <typename R, bool RAYS, bool PAIRS>
__device__ void build_profiles(const DevAtom &A, const Smem<R> &s, const KParams &p, R *phc)
{
    const int N = p.N, nmu = A.nmu;
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const R *lt = reinterpret_cast<const R *>(p.lane);
    for (int w = threadIdx.x >> 5; w < A.nphi * 8; w += nw) {
        const int row = w >> 3, dir = (w >> 2) & 1, part = w & 3;
        const int b = A.phi_tile[row], j = A.phi_j[row];
        const int pi = b * kWarp + lane;
        const R q = lt[(RH_NLANEF * j + 4) * p.npad + pi];
        const R pn = lt[(RH_NLANEF * j + 5) * p.npad + pi];
        const R *ad = s.ad + (size_t)A.tr[A.tile[b].t[j]].sub * N;
        for (int k = N * part / 4; k < N * (part + 1) / 4; ++k) {
            const R vz = s.vz[k], iv = s.ivth[k], a = ad[k];
            auto at = [&](int m) {
                const R mu = mu_of<R>(A, m);
                return line_phi(q, dir ? mu : -mu, vz, iv, a, pn, s.vtab, p.tab64);
            };
            if constexpr (PAIRS) {
                const int np = (nmu + 1) / 2;
                float2 *o = reinterpret_cast<float2 *>(phc + phi_pairs(np, N, row, dir)) + k * np * kWarp + lane;
                for (int v = 0; v < np; ++v) {
                    const R lo = at(2 * v), hi = 2 * v + 1 < nmu ? at(2 * v + 1) : lo;
                    o[v * kWarp] = make_float2(lo, hi);
                }
            } else {
                R *o = phc + (RAYS ? phi_ray(nmu, N, row, dir, 0) + k * kWarp : phi_block(nmu, N, row, dir, k)) + lane;
                for (int m = 0; m < nmu; ++m) o[RAYS ? m * N * kWarp : m * kWarp] = at(m);
            }
        }
    }
}

__device__ __forceinline__ double block_max(double v, double *red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    double t = -1.0e308;
    for (int i = 0; i < nw; ++i) t = fmax(t, red[i]);
    __syncthreads();
    return t;
}

// ---- rate equations ----------------------------------------------------------
// Off-diagonal rate-matrix entries (DevAtom::ent_*), summed in FP64 over the
// tiles' accumulators and the collisional rates by the whole block: a thread
// takes (entry, depth) items, holds their sums in registers until every
// accumulator of their depths has been read, and puts them in the
// accumulators' place: entry e of depth k in row e (FP64) or split over rows
// 2e and 2e + 1 (FP32), so a depth's sums only displace its own accumulators.
// Chunks of depths keep the held items at kHeld a thread.  (One thread per
// depth doing all of this and the solve with its matrix in local memory took
// 118 us an iteration, a quarter of the iteration.)
constexpr int kHeld = 8;
__device__ __forceinline__ void put_entry(float *slot, int e, int N, int k, double v)
{
    slot[(2 * e) * N + k] = __int_as_float(__double2loint(v));
    slot[(2 * e + 1) * N + k] = __int_as_float(__double2hiint(v));
}
__device__ __forceinline__ void put_entry(double *slot, int e, int N, int k, double v) { slot[e * N + k] = v; }
__device__ __forceinline__ double get_entry(const float *slot, int e, int N, int k)
{
    return __hiloint2double(__float_as_int(slot[(2 * e + 1) * N + k]), __float_as_int(slot[(2 * e) * N + k]));
}
__device__ __forceinline__ double get_entry(const double *slot, int e, int N, int k) { return slot[e * N + k]; }

template <typename R>
__device__ void assemble_rates(const DevAtom &A, R *slot, const R *slot2, int N, const double *Cr, double fcr)
{
    const int nt = blockDim.x, kc = min(N, kHeld * nt / A.nent);
    const R one = slot2 == slot ? (R)0 : (R)1;   // 0: no second set of accumulators
    for (int k0 = 0; k0 < N; k0 += kc) {
        const int nk = min(kc, N - k0);
        double g[kHeld];
#pragma unroll
        for (int h = 0; h < kHeld; ++h) {
            const int it = threadIdx.x + h * nt, e = it / nk, k = k0 + it % nk;
            double s = 0.0;
            if (e < A.nent) {
#pragma unroll 2
                for (int i = A.ent_off[e]; i < A.ent_off[e + 1]; ++i) {
                    const int m = A.ent_acc[i], o = (m >> 1) * N + k;   // accumulator, sign in bit 0
                    const R v = slot[o] + one * slot2[o];
                    s += (double)(m & 1 ? -v : v);
                }
                for (int i = A.cx_off[e]; i < A.cx_off[e + 1]; ++i) s += Cr[(size_t)k * 2 * A.ntr + A.cx_idx[i]] * fcr;
            }
            g[h] = s;
        }
        __syncthreads();
#pragma unroll
        for (int h = 0; h < kHeld; ++h) {
            const int it = threadIdx.x + h * nt, e = it / nk, k = k0 + it % nk;
            if (e < A.nent) put_entry(slot, e, N, k, g[h]);
        }
    }
    __syncthreads();
}

// Scaled LU solve of one depth's rate equations (the row of the most
// populated level replaced by particle conservation, unknowns scaled by the
// old populations, rows equilibrated) for the new populations.  Returns 0 on
// success.  One thread holds the system in registers: LM >= L is a
// compile-time size (levels beyond L are rows of the identity), every index is
// static, and a pivot is brought up by conditional row exchanges.
template <int LM, typename R>
__device__ __noinline__ int solve_lu(const DevAtom &A, const R *slot, int N, int k, const double *n, double nHk,
                                     double *nn)
{
    const int L = A.nlev;
    double G[LM][LM], sc[LM], b[LM];
#pragma unroll
    for (int p = 0; p < LM; ++p)
#pragma unroll
        for (int q = 0; q < LM; ++q) {
            const int e = p < L && q < L ? A.ent_id[p * RH_MAXLEV + q] : -1;
            G[p][q] = e >= 0 ? get_entry(slot, e, N, k) : 0.0;
        }
    int r = 0;
    double top = -1.0;
#pragma unroll
    for (int q = 0; q < LM; ++q) {
        double s = 0.0;
#pragma unroll
        for (int p = 0; p < LM; ++p)
            if (p != q) s += G[p][q];
        G[q][q] = q < L ? -s : 1.0;
        sc[q] = q < L ? n[q * N + k] : 1.0;
        b[q] = 0.0;
        if (q < L && sc[q] > top) {
            top = sc[q];
            r = q;
        }
    }
    int bad = 0;
#pragma unroll
    for (int p = 0; p < LM; ++p) {
        double mx = 0.0;
#pragma unroll
        for (int q = 0; q < LM; ++q) {
            if (p == r) G[p][q] = q < L ? 1.0 : 0.0;
            G[p][q] *= sc[q];
            mx = fmax(mx, fabs(G[p][q]));
        }
        if (!(mx > 0.0)) bad = 1;
        const double im = 1.0 / mx;
#pragma unroll
        for (int q = 0; q < LM; ++q) G[p][q] *= im;
        if (p == r) b[p] = nHk * im;
    }
#pragma unroll
    for (int c = 0; c < LM; ++c) {
#pragma unroll
        for (int rr = c + 1; rr < LM; ++rr) {
            const bool sw = fabs(G[rr][c]) > fabs(G[c][c]);
#pragma unroll
            for (int q = c; q < LM; ++q) {
                const double u = G[c][q], v = G[rr][q];
                G[c][q] = sw ? v : u;
                G[rr][q] = sw ? u : v;
            }
            const double u = b[c], v = b[rr];
            b[c] = sw ? v : u;
            b[rr] = sw ? u : v;
        }
        if (G[c][c] == 0.0) bad = 1;
        // one reciprocal per pivot (kept for the back substitution)
        const double ip = 1.0 / G[c][c];
        G[c][c] = ip;
#pragma unroll
        for (int rr = c + 1; rr < LM; ++rr) {
            const double f = G[rr][c] * ip;
#pragma unroll
            for (int q = c + 1; q < LM; ++q) G[rr][q] -= f * G[c][q];
            b[rr] -= f * b[c];
        }
    }
    if (bad) return 1;
#pragma unroll
    for (int c = LM - 1; c >= 0; --c) {
        double s = b[c];
#pragma unroll
        for (int q = c + 1; q < LM; ++q) s -= G[c][q] * b[q];
        b[c] = s * G[c][c];
    }
#pragma unroll
    for (int l = 0; l < LM; ++l)
        if (l < L) nn[l * N + k] = b[l] * sc[l];
    return 0;
}

template <typename R>
__device__ __forceinline__ int solve_depth(const DevAtom &A, const R *slot, int N, int k, const double *n, double nHk,
                                           double *nn)
{
    if (A.nlev <= 4) return solve_lu<4, R>(A, slot, N, k, n, nHk, nn);
    if (A.nlev <= 6) return solve_lu<6, R>(A, slot, N, k, n, nHk, nn);
    return solve_lu<RH_MAXLEV, R>(A, slot, N, k, n, nHk, nn);
}

// CACHE: line profiles from the per-block cache (p.phic, nullptr only for an
// atom without lines); otherwise evaluated in the sweep.  BEZ: the quadratic
// Bezier formal solver (its own instantiations, so that the linear kernels
// keep their registers).  FP32: 128 registers, two resident blocks of 256
// threads, or (linear solver, complete redistribution) one of 512.  (Three
// blocks of 256 at 80 registers: 3.92 instead of 3.11 us per column-iteration.)
template <typename R, bool PRD, bool CACHE, bool BEZ>
__global__ void __launch_bounds__(sizeof(R) == 4 && !PRD && !BEZ ? 512 : 256, sizeof(R) == 4 && (PRD || BEZ) ? 2 : 1) mali_kernel(const __grid_constant__ DevAtom A, const __grid_constant__ KParams p)
{
    extern __shared__ __align__(16) char smem_raw[];
    const int N = p.N, L = A.nlev;
    constexpr bool RAYS = PRD || BEZ;                        // sweep_tile_k, which adds to its accumulators
    constexpr bool UNITS = sizeof(R) == 8 && !RAYS;          // sweep_unit, which writes them
    constexpr bool SUMS = sizeof(R) == 4 && !RAYS && CACHE;  // sweep_pairs, totals kept apart
    Smem<R> s = carve<R>(smem_raw, L, N, 0, A.ncont, A.nline, p.slot_rows, 0);
    const int tid = threadIdx.x, lane = tid & 31;
    const int LN = L * N;
    double *hist = p.nghist + (size_t)blockIdx.x * 4 * LN;

    const int64_t nwork = p.nwork_d ? (int64_t)*p.nwork_d : p.nwork;
    PrdScr<R> ps{};
    if constexpr (PRD) ps = prd_carve<R>(p.prd_scr + (size_t)blockIdx.x * p.prd_stride, A, N);
    R *phc = (CACHE && p.phic) ? reinterpret_cast<R *>(p.phic + (size_t)blockIdx.x * p.phic_stride) : nullptr;
    int64_t done = 0;
    for (;;) {
        __syncthreads();
        if (tid == 0) {
            int64_t q;
            if (p.persistent) q = atomicAdd(p.queue, 1);
            else q = (int64_t)blockIdx.x + done * gridDim.x;
            s.ibuf[0] = q < nwork ? (p.colidx ? p.colidx[q] : (int)q) : -1;
        }
        __syncthreads();
        const int col = s.ibuf[0];
        if (col < 0) break;
        ++done;
        const size_t cN = (size_t)col * N;
        // ---- load the column (and the Voigt table, whose place the sweep's scratch takes)
        if (sizeof(R) == 4)
            for (int i = tid; i <= RH_VT_N; i += blockDim.x) s.vtab[i] = p.vtab[i];
        for (int k = tid; k < N; k += blockDim.x) {
            double T = p.T[cN + k];
            double ne = p.ne[cN + k];
            s.dz[k] = (R)(k < N - 1 ? fabs(p.z[cN + k] - p.z[cN + k + 1]) : 0.0);
            double vth = sqrt(2.0 * kK * T / A.mass);
            s.ivth[k] = (R)(1.0 / vth);
            s.vz[k] = (R)p.vz[cN + k];
            s.bg[4 * k + 0] = (R)(kH / (kK * T));
            double e2 = kQ * kQ / (4.0 * kPi * kEps0);
            double Cff = e2 * e2 * e2 * 4.0 / (3.0 * kMe * kH * kC) * sqrt(2.0 * kPi / (3.0 * kK * kMe));
            s.bg[4 * k + 1] = (R)(Cff * ne * p.np[cN + k] / sqrt(T) / kNuRef3);
            double n1 = p.nstar[((size_t)col * L + 0) * N + k];
            double lam3 = pow(kH * kH / (2.0 * kPi * kMe * kK * T), 1.5);
            s.bg[4 * k + 2] = (R)(0.25 * n1 * ne * lam3 * exp(0.754 * kQ / (kK * T)));
            s.bg[4 * k + 3] = (R)(kSigmaT * ne);
            double sk = N > 1 ? (double)k / (N - 1) : 0.0;
            for (int t = 0; t < A.ntr; ++t) {
                const DevTrans &tr = A.tr[t];
                if (tr.kind == 0) {
                    s.ad[tr.sub * N + k] = (R)exp((1.0 - sk) * tr.ln_atop + sk * tr.ln_abot);
                } else {
                    s.Gc[tr.sub * N + k] = (R)(p.nstar[((size_t)col * L + tr.l) * N + k] /
                                               p.nstar[((size_t)col * L + tr.u) * N + k]);
                }
            }
        }
        const double *Cr = p.Crate + cN * 2 * A.ntr;
        if (phc) {
            __syncthreads();   // the column's Doppler widths, velocities and damping
            build_profiles<R, RAYS, sizeof(R) == 4 && !RAYS>(A, s, p, phc);
        }
        if constexpr (PRD) {
            // redistribution kernels of the column: K_ij = R(x_j, x_i) w_j / sum_j (.),
            // x in Doppler units of the depth (static frame), and the J-bar weights
            // f_j = H(a, x_j) w_j / sum_j (.); x and a per point and depth first
            for (int e = tid; e < A.npp * N; e += blockDim.x) {
                const int pp = e / N, k = e % N;
                int q = 0;
                while (pp >= A.prd_off[q + 1]) ++q;
                const DevTrans &tr = A.tr[A.prd_t[q]];
                const double dnuD = tr.nu0 / kC * sqrt(2.0 * kK * p.T[cN + k] / A.mass);
                ps.x[e] = (R)((p.prd_nu[pp] - tr.nu0) / dnuD);
            }
            for (int pp = tid; pp < A.npp; pp += blockDim.x) {
                int q = 0;
                while (pp >= A.prd_off[q + 1]) ++q;
                const double nu0 = A.tr[A.prd_t[q]].nu0;
                ps.q[pp] = (R)(kC * (p.prd_nu[pp] - nu0) / nu0);
            }
            for (int e = tid; e < A.nprd * N; e += blockDim.x) {
                const int q = e / N, k = e % N;
                const DevTrans &tr = A.tr[A.prd_t[q]];
                const double sk = N > 1 ? (double)k / (N - 1) : 0.0;
                ps.a[e] = (R)exp((1.0 - sk) * tr.ln_atop + sk * tr.ln_abot);
            }
            __syncthreads();
            if (p.prd_hybrid) build_hybrid_tables<R>(A, s, ps, N);   // read after later barriers
            for (int q = 0; q < A.nprd; ++q) {
                const int off = A.prd_off[q], np = A.prd_off[q + 1] - off, npair = np * (np + 1) / 2;
                R *Kq = ps.K + (size_t)A.prd_koff[q] * N;
                // R is symmetric: one evaluation per unordered pair (i <= j), pairs
                // numbered row by row, p = i np - i (i - 1) / 2 + (j - i)
                for (int e = tid; e < npair * N; e += blockDim.x) {
                    const int k = e / npair, pr = e % npair;
                    int i = (int)((2.0f * np + 1.0f - sqrtf((2.0f * np + 1.0f) * (2.0f * np + 1.0f) - 8.0f * pr)) * 0.5f);
                    while (i > 0 && i * np - i * (i - 1) / 2 > pr) --i;
                    while ((i + 1) * np - (i + 1) * i / 2 <= pr) ++i;
                    const int j = i + pr - (i * np - i * (i - 1) / 2);
                    const R ak = ps.a[q * N + k];
                    const R rv = r2a_dev<R>(ak, ps.x[(size_t)(off + j) * N + k], ps.x[(size_t)(off + i) * N + k]);
                    Kq[((size_t)k * np + j) * np + i] = rv * (R)p.prd_w[off + j];     // K_ij
                    Kq[((size_t)k * np + i) * np + j] = rv * (R)p.prd_w[off + i];     // K_ji
                }
            }
            __syncthreads();
            for (int q = 0; q < A.nprd; ++q) {
                const int off = A.prd_off[q], np = A.prd_off[q + 1] - off;
                R *Kq = ps.K + (size_t)A.prd_koff[q] * N;
                for (int e = tid; e < np * N; e += blockDim.x) {
                    const int k = e / np, i = e % np;
                    R *col = Kq + (size_t)k * np * np + i;                    // K_ij at col[j np]
                    R sr = 0;
                    for (int j = 0; j < np; ++j) sr += col[(size_t)j * np];
                    const R inv = (R)1 / sr;
                    for (int j = 0; j < np; ++j) col[(size_t)j * np] *= inv;
                }
                for (int k = tid; k < N; k += blockDim.x) {
                    const R ak = ps.a[q * N + k];
                    R fs = 0;
                    for (int j = 0; j < np; ++j) {
                        const R v = voigt(ak, ps.x[(size_t)(off + j) * N + k], s.vtab, p.tab64) * (R)p.prd_w[off + j];
                        ps.f[(size_t)(off + j) * N + k] = v;
                        fs += v;
                    }
                    const R inv = (R)1 / fs;
                    for (int j = 0; j < np; ++j) ps.f[(size_t)(off + j) * N + k] *= inv;
                }
            }
        }
        int start = p.start, ng_order = p.ng_order, maxiter = p.maxiter, rung = 0;
        double crsw = p.crsw;
        int it = 0, status = RH_COL_MAXITER;
        double dmax = 1e300;
      restart:
        if constexpr (PRD) {
            for (int i = tid; i < A.npp * N; i += blockDim.x) ps.rho[i] = 1;   // PRD starts as CRD
            if (p.prd_hybrid) {
                __syncthreads();
                fill_rho_ray<R>(A, ps, N);
            }
        }
        for (int i = tid; i < LN; i += blockDim.x) {
            double v = start == 0 ? p.nstar[(size_t)col * LN + i] : p.pops[(size_t)col * LN + i];
            s.n[i] = v;
        }
        int hcount = 0, hpos = 0, rcount = 0, rpos = 0;
        status = RH_COL_MAXITER;
        dmax = 1e300;
        for (it = 1; it <= maxiter; ++it) {
            double fcr = crsw > 1.0 ? fmax(1.0, crsw * pow(10.0, -(double)(it - 1))) : 1.0;
            for (int i = tid; i < LN; i += blockDim.x) s.nr[i] = (R)(s.n[i] * p.inv_nref);
            if (!UNITS && !SUMS)
                for (int i = tid; i < A.macc * N; i += blockDim.x) s.slot[i] = 0;
            if constexpr (PRD) {
                for (int i = tid; i < A.npp * N; i += blockDim.x) {
                    ps.J[i] = 0;
                    ps.D[i] = 0;
                }
                for (int i = tid; i < A.pacc * N; i += blockDim.x) ps.plain[i] = 0;
            }
            if (tid == 0) s.ibuf[1] = 0;
            __syncthreads();
            // ---- formal solution and rate accumulation: warps take tiles from a
            // block-local queue, most expensive tiles first
            for (;;) {
                int q = 0;
                if (lane == 0) q = atomicAdd(&s.ibuf[1], 1);
                q = __shfl_sync(0xffffffffu, q, 0);
                if (q >= (p.split ? 2 * A.ntile : A.ntile)) break;
                sweep_item<R, PRD, CACHE, BEZ>(A, s, p, q, lane, ps.rho, ps.J, ps.D, ps.plain,
                                               p.prd_hybrid ? ps.Iray : nullptr, phc);
            }
            __syncthreads();
            if constexpr (SUMS) {
                sum_pairs(A, p, pair_sums(A, p, phc), s.slot);
                __syncthreads();
            }
            // ---- rate equations: the matrices by the whole block, then one thread per depth
            assemble_rates<R>(A, s.slot, UNITS && p.split ? s.slot + (size_t)A.macc * N : s.slot, N, Cr, fcr);
            int bad = 0;
            double dloc = 0.0;
            for (int k = tid; k < N; k += blockDim.x) {
                int e = solve_depth<R>(A, s.slot, N, k, s.n, p.nH[cN + k], s.nn);
                if (e) bad = 2;
                for (int l = 0; l < L && !e; ++l) {
                    double a = s.nn[l * N + k];
                    if (!(isfinite(a) && a > 0.0)) {
                        bad = bad ? bad : 1;
                        break;
                    }
                    dloc = fmax(dloc, fabs(a - s.n[l * N + k]) / a);
                }
            }
            double badg = block_max((double)bad, s.red);
            dmax = block_max(dloc, s.red);
            if (badg > 0) {
                status = badg > 1.5 ? RH_COL_SINGULAR : RH_COL_NONFINITE;
                break;
            }
            const bool conv = dmax < p.tol && fcr == 1.0;
            // ---- Ng history (newest first, ring of 4)
            hpos = (hpos + 3) & 3;
            for (int i = tid; i < LN; i += blockDim.x) hist[(size_t)hpos * LN + i] = s.nn[i];
            __syncthreads();
            if (hcount < 4) ++hcount;
            if (!conv && ng_order == 2 && it >= p.ng_delay && hcount >= 4 &&
                (it - p.ng_delay) % p.ng_period == 0) {
                const double *x0 = hist + (size_t)hpos * LN, *x1 = hist + (size_t)((hpos + 1) & 3) * LN,
                             *x2 = hist + (size_t)((hpos + 2) & 3) * LN, *x3 = hist + (size_t)((hpos + 3) & 3) * LN;
                // dot products over a fixed partition of kNgLanes partial sums,
                // added in a fixed order: the result does not depend on the
                // block size
                for (int v = tid; v < kNgLanes; v += blockDim.x) {
                    double q[5] = {0, 0, 0, 0, 0};
                    for (int i = v; i < LN; i += kNgLanes) {
                        double d0 = x0[i] - x1[i], d1 = x1[i] - x2[i], d2 = x2[i] - x3[i];
                        double pp = d0 - d1, qq = d0 - d2;
                        q[0] += pp * pp;
                        q[1] += pp * qq;
                        q[2] += qq * qq;
                        q[3] += d0 * pp;
                        q[4] += d0 * qq;
                    }
                    for (int j = 0; j < 5; ++j) s.red[j * kNgLanes + v] = q[j];
                }
                __syncthreads();
                if (tid < 5) {
                    double t = 0.0;
                    for (int i = 0; i < kNgLanes; ++i) t += s.red[tid * kNgLanes + i];
                    s.red[5 * kNgLanes + tid] = t;
                }
                __syncthreads();
                const double a11 = s.red[5 * kNgLanes + 0], a12 = s.red[5 * kNgLanes + 1],
                             a22 = s.red[5 * kNgLanes + 2], b1 = s.red[5 * kNgLanes + 3],
                             b2 = s.red[5 * kNgLanes + 4];
                __syncthreads();
                double det = a11 * a22 - a12 * a12;
                if (fabs(det) > 0.0 && isfinite(det)) {
                    double ca = (b1 * a22 - b2 * a12) / det, cb = (a11 * b2 - a12 * b1) / det;
                    int okl = 1;
                    for (int i = tid; i < LN; i += blockDim.x) {
                        double v = (1.0 - ca - cb) * x0[i] + ca * x1[i] + cb * x2[i];
                        if (!(isfinite(v) && v > 0.0)) okl = 0;
                    }
                    double ok = -block_max(-(double)okl, s.red);
                    if (ok > 0.5) {
                        for (int i = tid; i < LN; i += blockDim.x) {
                            double v = (1.0 - ca - cb) * x0[i] + ca * x1[i] + cb * x2[i];
                            s.nn[i] = v;
                        }
                        __syncthreads();
                        for (int i = tid; i < LN; i += blockDim.x) hist[(size_t)hpos * LN + i] = s.nn[i];
                        hcount = 1;
                    }
                }
            }
            __syncthreads();
            for (int i = tid; i < LN; i += blockDim.x) s.n[i] = s.nn[i];
            __syncthreads();
            if (conv) {
                status = RH_COL_CONVERGED;
                break;
            }
            if constexpr (PRD) {
                // rho for the next iteration (Uitenbroek 2001, Eq. 14, angle-averaged,
                // gamma = 1): r = 1 + F (sum_j K_ij J_j / Jbar - 1), F = n_l R_lu /
                // (supply of the upper level) with the plain rates of this formal
                // solution and the collisions, n the next iteration's populations;
                // PRD switching (Eq. 1) r' = eps r + (1 - eps), eps = min(1, eps0
                // it^2) of the iteration that uses it
                const double eps =
                    p.prd_eps0 > 0.0 ? fmin(1.0, p.prd_eps0 * (double)(it + 1) * (double)(it + 1)) : 1.0;
                if (p.prd_hybrid) {
                    hybrid_JD<R>(A, ps, N);   // the gas-frame J and D in place of the sweep's
                    __syncthreads();
                }
                for (int e = tid; e < A.nprd * N; e += blockDim.x) {
                    const int q = e / N, k = e % N, tq = A.prd_t[q];
                    const int u = A.tr[tq].u, l = A.tr[tq].l;
                    double in = 0.0, up_line = 0.0;
                    for (int b = 0; b < A.ntile; ++b) {
                        const DevTile &tb = A.tile[b];
                        for (int j = 0; j < tb.K; ++j) {
                            const DevTrans &t2 = A.tr[tb.t[j]];
                            const double pu = (double)ps.plain[(size_t)(tb.pacc_off + 2 * j) * N + k];
                            const double pd = (double)ps.plain[(size_t)(tb.pacc_off + 2 * j + 1) * N + k];
                            if (t2.u == u) in += s.n[t2.l * N + k] * pu;
                            if (t2.l == u) in += s.n[t2.u * N + k] * pd;
                            if (tb.t[j] == tq) up_line += pu;
                        }
                    }
                    const double *Ck = Cr + (size_t)k * 2 * A.ntr;
                    for (int t = 0; t < A.ntr; ++t) {
                        if (A.tr[t].u == u) in += s.n[A.tr[t].l * N + k] * Ck[2 * t] * fcr;
                        if (A.tr[t].l == u) in += s.n[A.tr[t].u * N + k] * Ck[2 * t + 1] * fcr;
                    }
                    ps.F[e] = s.n[l * N + k] * up_line / in;
                    const int off = A.prd_off[q], np = A.prd_off[q + 1] - off;
                    R jb = 0;
                    for (int j = 0; j < np; ++j) jb += ps.f[(size_t)(off + j) * N + k] * ps.J[(size_t)(off + j) * N + k];
                    ps.Jbar[e] = (double)jb;
                }
                __syncthreads();
                // with Ng: one Jacobi step rho += (r' - rho) / max(1 - eps g_ii, 0.02),
                // g_ii = dr_i/drho_i = F D_i (K_ii - f_i sum_j K_ij J_j / Jbar) / Jbar,
                // and Ng on the rho sequence; without Ng: rho = (rho + r') / 2
                const bool jac = ng_order == 2;
                rpos = (rpos + 3) & 3;
                double *rh0 = ps.hist + (size_t)rpos * A.npp * N;
                // threads own (depth, point) with the point fastest: K_ij of
                // consecutive points i at consecutive addresses, J_j shared.  In
                // FP32, with np a multiple of 4, a thread owns four consecutive
                // points and streams K as float4 with eight rows in flight (the
                // sum is memory-latency-bound otherwise); the sums run over j in
                // the same order either way.
                for (int q = 0; q < A.nprd; ++q) {
                    const int off = A.prd_off[q], np = A.prd_off[q + 1] - off;
                    const R *Kq = ps.K + (size_t)A.prd_koff[q] * N;
                    const bool vec = sizeof(R) == 4 && (np & 3) == 0 && (A.prd_koff[q] & 3) == 0;
                    const int G = vec ? 4 : 1, ng = np / G;
                    for (int e = tid; e < ng * N; e += blockDim.x) {
                        const int k = e / ng, i0 = (e % ng) * G;
                        const R *col = Kq + (size_t)k * np * np + i0;
                        const R *Jk = ps.J + (size_t)off * N + k;
                        R sr[4] = {0, 0, 0, 0};
                        if constexpr (sizeof(R) == 4) {
                            if (vec) {
                                float4 acc[2] = {make_float4(0, 0, 0, 0), make_float4(0, 0, 0, 0)};
                                int j = 0;
                                for (; j + 8 <= np; j += 8) {
                                    float4 kv[8];
                                    float jv[8];
#pragma unroll
                                    for (int u = 0; u < 8; ++u) {
                                        kv[u] = *reinterpret_cast<const float4 *>(col + (size_t)(j + u) * np);
                                        jv[u] = Jk[(size_t)(j + u) * N];
                                    }
#pragma unroll
                                    for (int u = 0; u < 8; ++u) {
                                        float4 &a4 = acc[u & 1];
                                        a4.x += kv[u].x * jv[u];
                                        a4.y += kv[u].y * jv[u];
                                        a4.z += kv[u].z * jv[u];
                                        a4.w += kv[u].w * jv[u];
                                    }
                                }
                                for (; j < np; ++j) {
                                    const float4 kv = *reinterpret_cast<const float4 *>(col + (size_t)j * np);
                                    const float jv = Jk[(size_t)j * N];
                                    acc[0].x += kv.x * jv;
                                    acc[0].y += kv.y * jv;
                                    acc[0].z += kv.z * jv;
                                    acc[0].w += kv.w * jv;
                                }
                                sr[0] = acc[0].x + acc[1].x;
                                sr[1] = acc[0].y + acc[1].y;
                                sr[2] = acc[0].z + acc[1].z;
                                sr[3] = acc[0].w + acc[1].w;
                            }
                        }
                        if (!vec) {
                            // eight independent partial sums, added in a fixed order
                            R part[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                            int j = 0;
                            for (; j + 8 <= np; j += 8) {
#pragma unroll
                                for (int u = 0; u < 8; ++u)
                                    part[u] += col[(size_t)(j + u) * np] * Jk[(size_t)(j + u) * N];
                            }
                            for (; j < np; ++j) part[0] += col[(size_t)j * np] * Jk[(size_t)j * N];
                            sr[0] = ((part[0] + part[1]) + (part[2] + part[3])) + ((part[4] + part[5]) + (part[6] + part[7]));
                        }
                        const R jb = (R)ps.Jbar[q * N + k], F = (R)ps.F[q * N + k], ep = (R)eps;
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            if (g >= G) break;
                            const int i = i0 + g, pe = (off + i) * N + k;
                            const R r = (R)1 + F * (sr[g] / jb - (R)1);
                            R den = 2;
                            if (jac) {
                                const R gi = F * (Kq[((size_t)k * np + i) * np + i] - ps.f[pe] * sr[g] / jb) * ps.D[pe] / jb;
                                den = (R)1 - ep * gi;
                                den = den > (R)0.02 ? den : (R)0.02;
                            }
                            ps.rho[pe] += ((ep * r + ((R)1 - ep)) - ps.rho[pe]) / den;
                            rh0[pe] = (double)ps.rho[pe];
                        }
                    }
                }
                __syncthreads();
                if (rcount < 4) ++rcount;
                if (jac && it >= p.ng_delay && rcount >= 4 && (it - p.ng_delay) % p.ng_period == 0) {
                    const int RV = A.npp * N;
                    const double *x0 = rh0, *x1 = ps.hist + (size_t)((rpos + 1) & 3) * RV,
                                 *x2 = ps.hist + (size_t)((rpos + 2) & 3) * RV,
                                 *x3 = ps.hist + (size_t)((rpos + 3) & 3) * RV;
                    for (int v = tid; v < kNgLanes; v += blockDim.x) {
                        double q5[5] = {0, 0, 0, 0, 0};
                        for (int i = v; i < RV; i += kNgLanes) {
                            double d0 = x0[i] - x1[i], d1 = x1[i] - x2[i], d2 = x2[i] - x3[i];
                            double pq = d0 - d1, qq = d0 - d2;
                            q5[0] += pq * pq;
                            q5[1] += pq * qq;
                            q5[2] += qq * qq;
                            q5[3] += d0 * pq;
                            q5[4] += d0 * qq;
                        }
                        for (int j = 0; j < 5; ++j) s.red[j * kNgLanes + v] = q5[j];
                    }
                    __syncthreads();
                    if (tid < 5) {
                        double t = 0.0;
                        for (int i = 0; i < kNgLanes; ++i) t += s.red[tid * kNgLanes + i];
                        s.red[5 * kNgLanes + tid] = t;
                    }
                    __syncthreads();
                    const double a11 = s.red[5 * kNgLanes + 0], a12 = s.red[5 * kNgLanes + 1],
                                 a22 = s.red[5 * kNgLanes + 2], b1 = s.red[5 * kNgLanes + 3],
                                 b2 = s.red[5 * kNgLanes + 4];
                    __syncthreads();
                    const double det = a11 * a22 - a12 * a12;
                    if (fabs(det) > 0.0 && isfinite(det)) {
                        const double ca = (b1 * a22 - b2 * a12) / det, cb = (a11 * b2 - a12 * b1) / det;
                        int okl = 1;
                        for (int i = tid; i < RV; i += blockDim.x) {
                            const double v = (1.0 - ca - cb) * x0[i] + ca * x1[i] + cb * x2[i];
                            if (!(isfinite(v) && v >= 0.0)) okl = 0;
                        }
                        const double ok = -block_max(-(double)okl, s.red);
                        if (ok > 0.5) {
                            for (int i = tid; i < RV; i += blockDim.x) {
                                const double v = (1.0 - ca - cb) * x0[i] + ca * x1[i] + cb * x2[i];
                                ps.rho[i] = (R)v;
                                rh0[i] = (double)ps.rho[i];
                            }
                            rcount = 1;
                        }
                    }
                }
                __syncthreads();
                if (p.prd_hybrid) fill_rho_ray<R>(A, ps, N);   // read after the next barrier
            }
        }
        if (it > maxiter) it = maxiter;
        if (tid == 0 && p.rung_its) atomicAdd(&p.rung_its[rung], (unsigned long long)it);
        if (status != RH_COL_CONVERGED && rung < p.nrung) {
            // next rung of the re-run ladder: from LTE, its own switching and Ng
            start = 0;
            ng_order = p.rung_ng[rung];
            crsw = p.rung_crsw[rung];
            maxiter = p.rung_maxiter;
            ++rung;
            if (tid == 0 && p.rung_cols) atomicAdd(&p.rung_cols[rung - 1], 1);
            __syncthreads();
            goto restart;
        }
        for (int i = tid; i < LN; i += blockDim.x) p.pops[(size_t)col * LN + i] = s.n[i];
        if (tid == 0) {
            p.iters[col] = it;
            p.status[col] = (uint8_t)status;
            p.dmax[col] = dmax;
        }
    }
}


}  // namespace mali

// the column kernels' addresses (one translation unit per family, compiled in
// parallel)
const void *mali_kernel_crd32(bool cache);
const void *mali_kernel_crd64(bool cache);
const void *mali_kernel_bez(int precision);
const void *mali_kernel_prd32();
const void *mali_kernel_prd32_bez();
const void *mali_kernel_prd64(bool bez);

}  // namespace rh
