// rh15d_mali.cu -- launches of the column kernel: which kernel, its launch
// shape and shared memory, its parameters.
#include <algorithm>
#include <cstdio>
#include <cstring>

#include "rh15d_mali.cuh"

namespace rh {

using namespace mali;

size_t mali_nghist_bytes_per_block(const DevAtom &A, int ndep) { return sizeof(double) * 4 * A.nlev * ndep; }

// the column kernel's shared-memory layout for the given sizes: its byte
// offsets in carve order and the allocated size (host computation only)
int mali_smem_layout(int precision, int L, int N, int ntr, int ncont, int nline, int macc, int ring_warps,
                     size_t *offsets, int noff, size_t *bytes)
{
    const SmemLayout o = precision == 1 ? smem_layout<float>(L, N, ntr, ncont, nline, macc, ring_warps)
                                        : smem_layout<double>(L, N, ntr, ncont, nline, macc, ring_warps);
    const size_t v[16] = {o.n,  o.nn, o.Cr, o.red,  o.slot, o.dz,   o.ivth, o.vz,
                          o.bg, o.Gc, o.ad, o.nr,   o.vtab, o.ibuf, o.ring, o.end};
    for (int i = 0; i < noff && i < 16; ++i) offsets[i] = v[i];
    *bytes = precision == 1 ? smem_bytes<float>(L, N, ntr, ncont, nline, macc, ring_warps)
                            : smem_bytes<double>(L, N, ntr, ncont, nline, macc, ring_warps);
    return 16;
}

size_t mali_phic_bytes_per_block(const DevAtom &A, int ndep, int precision)
{
    return precision == 1 ? phic_bytes<float>(A, ndep) : phic_bytes<double>(A, ndep);
}

size_t mali_prd_bytes_per_block(const DevAtom &A, int ndep, int precision)
{
    if (!A.nprd) return 0;
    return precision == 1 ? prd_bytes<float>(A, ndep) : prd_bytes<double>(A, ndep);
}

namespace {

// What a launch of the column kernel needs besides its parameters.
struct Shape {
    const void *fn = nullptr;
    size_t sm = 0;
    int per_sm = 0;      // resident blocks per SM (0: does not fit)
    int split = 0, piece = 0, nsp = 0, nvp = 0, slot_rows = 0;
};

// The kernel for the atom and options, its shared memory with bw warps and
// its resident blocks.  The linear sweeps of complete redistribution take a
// tile's two directions as separate work items: twice the items balance the
// warps (20 tiles on 8 warps: 3 rounds of both directions, 5 of one).  FP32
// with the cache always (the totals are kept apart in global memory and summed
// in a fixed order); FP64, whose directions then have accumulators of their
// own, where those cost no resident block (43.0 -> 42.4 ms; an accumulator
// is the downward sum plus the upward one either way).  So no result depends
// on the launch shape.
cudaError_t shape_of(const DevAtom &A, int N, int precision, bool cache, bool bez, int bw, Shape &s)
{
    const bool f32 = precision == 1, crd = !A.nprd && !bez;
    if (A.nprd) s.fn = f32 ? (bez ? mali_kernel_prd32_bez() : mali_kernel_prd32()) : mali_kernel_prd64(bez);
    else if (bez) s.fn = mali_kernel_bez(precision);
    else if (f32) s.fn = mali_kernel_crd32(cache);
    else s.fn = mali_kernel_crd64(cache);
    if (crd)   // ray states, and (FP32 with the cache) the profile ring, per warp
        s.piece = f32 ? pairs_scratch(A, cache) * (int)sizeof(float) : 3 * A.nmu * kWarp * (int)sizeof(double);
    for (int split = 0; split <= (crd && !f32 ? 1 : 0); ++split) {
        // accumulators (of both directions), or the rate-matrix entries summed in their place
        const int macc = std::max(split ? 2 * A.macc : A.macc, (f32 ? 2 : 1) * A.nent);
        // warps whose scratch lies in the accumulators' and in the Voigt table's place (warp_scratch)
        const int slot = macc * N * (int)sizeof(float) - 16;
        const int nsp = s.piece && f32 && cache && slot > 0 ? slot / s.piece : 0;
        const int nvp = s.piece && !(f32 && !cache) ? (int)(kVtabBytes / s.piece) : 0;
        const int behind = s.piece ? std::max(0, bw - nsp - nvp) : 0;
        const int extra = (behind * s.piece + kScratchUnit - 1) / kScratchUnit;
        const size_t sm = f32 ? smem_bytes<float>(A.nlev, N, 0, A.ncont, A.nline, macc, extra)
                              : smem_bytes<double>(A.nlev, N, 0, A.ncont, A.nline, macc, extra);
        int per = 0;
        if (sm > 227 * 1024) {
            if (split) break;
            s.sm = sm;
            return cudaSuccess;   // per_sm 0
        }
        cudaError_t e = cudaFuncSetAttribute(s.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, s.fn, bw * kWarp, sm);
        if (e != cudaSuccess) return e;
        if (split && per < s.per_sm) break;
        s.sm = sm;
        s.per_sm = per;
        s.split = crd && f32 ? cache : split;
        s.nsp = nsp;
        s.nvp = nvp;
        s.slot_rows = macc;
    }
    return cudaSuccess;
}

// warps per block where the caller leaves the choice: 8, and 16 (FP32, the
// register limit) while every column has an SM of its own, where the second
// resident block would stay empty (12 iterations of one column 6.8 -> 5.4 ms,
// of 150 7.1 -> 5.6 ms; of 200, with 8, 10.0 ms)
int default_warps(const DevAtom &A, const IterLaunch &o, bool bez)
{
    if (o.block_warps > 0) return o.block_warps;
    if (A.nprd || bez) return o.precision ? 8 : 4;
    return o.precision == 1 && !o.nwork_d && o.nwork <= o.nsm ? 16 : 8;
}

// The warps, kernel and layout a launch takes: the caller's warps, or the
// default, halved (to 4 at least) until a column fits the block's shared
// memory (many depths, angles or overlapping lines: fewer warps' scratch).
cudaError_t pick_shape(const DevAtom &A, int N, const IterLaunch &o, bool cache, bool bez, int &bw, Shape &s)
{
    bw = default_warps(A, o, bez);
    for (;;) {
        s = Shape();
        const cudaError_t e = shape_of(A, N, o.precision, cache, bez, bw, s);
        if (e != cudaSuccess || s.per_sm > 0 || o.block_warps > 0 || bw <= 4) return e;
        bw /= 2;
    }
}

void fill_k2(KParams &p)
{
    // 1, -1; w_o / d and (1 - e^{-d}) / d as polynomials in d (sc_weights)
    const float c[kNK2] = {1.0f,        -1.0f,        0.5f,        -1.0f / 6,   1.0f / 24,    -1.0f / 120,
                           1.0f / 720,  -1.0f / 5040, 1.0f / 40320, -1.0f / 362880, 1.0f,     -0.5f,
                           1.0f / 6,    -1.0f / 24,   1.0f / 120,  -1.0f / 720, 1.0f / 5040,  -1.0f / 40320};
    for (int i = 0; i < kNK2; ++i) {
        uint32_t u;
        memcpy(&u, &c[i], 4);
        p.k2[i] = (unsigned long long)u << 32 | u;
    }
}

KParams make_params(const DevAtom &A, const ColumnArrays &c, const void *lane_tab, int npad, const float4 *vtab,
                    double nref, double *nghist, int *queue, const IterLaunch &o)
{
    KParams p;
    p.ncol = c.ncol;
    p.N = c.ndep;
    p.L = A.nlev;
    p.z = c.z;
    p.T = c.T;
    p.nH = c.nH;
    p.vz = c.vz;
    p.ne = c.ne;
    p.np = c.np;
    p.nstar = c.nstar;
    p.Crate = c.Crate;
    p.pops = c.pops;
    p.dmax = c.dmax;
    p.iters = c.iters;
    p.status = c.status;
    p.lane = lane_tab;
    p.npad = npad;
    p.vtab = vtab;
    p.nghist = nghist;
    p.queue = queue;
    p.persistent = o.persistent;
    p.maxiter = o.maxiter;
    p.ng_order = o.ng_order;
    p.ng_delay = o.ng_delay;
    p.ng_period = o.ng_period;
    p.start = o.start;
    p.tol = o.tol;
    p.crsw = o.crsw;
    p.inv_nref = 1.0 / nref;
    p.colidx = o.colidx;
    p.nwork = o.nwork;
    p.nwork_d = o.nwork_d;
    p.nrung = o.nrung;
    p.rung_maxiter = o.rung_maxiter;
    for (int r = 0; r < RH_MAX_RERUN; ++r) {
        p.rung_crsw[r] = o.rung_crsw[r];
        p.rung_ng[r] = o.rung_ng[r];
    }
    p.rung_cols = o.rung_cols;
    p.rung_its = o.rung_its;
    p.prd_eps0 = o.prd_eps0;
    p.prd_hybrid = o.prd_hybrid;
    p.formal = o.formal;
    p.lane_prd = o.lane_prd;
    p.prd_nu = o.prd_nu;
    p.prd_w = o.prd_w;
    p.prd_scr = reinterpret_cast<char *>(o.prd_scr);
    p.prd_stride = A.nprd ? (o.precision == 1 ? prd_bytes<float>(A, c.ndep) : prd_bytes<double>(A, c.ndep)) : 0;
    p.tab64 = o.tab64;
    p.piece = p.nsp = p.nvp = p.split = p.slot_rows = p.scr[0] = p.scr[1] = p.scr[2] = 0;
    fill_k2(p);
    p.phic_stride = o.precision == 1 ? phic_bytes<float>(A, c.ndep) : phic_bytes<double>(A, c.ndep);
    p.phic = (o.phic && p.phic_stride && p.phic_stride <= o.phic_cap) ? reinterpret_cast<char *>(o.phic) : nullptr;
    return p;
}

// grid of the persistent launch, bounded by the scratch the caller has
int64_t grid_of(const DevAtom &A, const KParams &p, const IterLaunch &o, const Shape &s, size_t hist_cap)
{
    const int per_sm = o.ctas_per_sm > 0 ? std::min(o.ctas_per_sm, s.per_sm) : s.per_sm;
    int64_t grid = (int64_t)per_sm * o.nsm;
    if (!p.nwork_d && grid > p.nwork) grid = p.nwork;
    grid = std::min<int64_t>(grid, (int64_t)(hist_cap / mali_nghist_bytes_per_block(A, p.N)));
    if (A.nprd) grid = std::min<int64_t>(grid, (int64_t)(o.prd_cap / p.prd_stride));
    if (p.phic) grid = std::min<int64_t>(grid, (int64_t)(o.phic_cap / p.phic_stride));
    return grid;
}

}  // namespace

// resident blocks per SM of the linear solver's kernel (a launch with the
// Bezier solver takes its own kernel's occupancy)
int mali_max_ctas_per_sm(const DevAtom &A, int ndep, int precision, int block_warps)
{
    Shape s;
    return shape_of(A, ndep, precision, true, false, block_warps, s) == cudaSuccess ? s.per_sm : 0;
}

// warps per block and resident blocks per SM of a launch with the profile cache
void mali_launch_shape(const DevAtom &A, int ndep, const IterLaunch &o, int *warps, int *ctas)
{
    Shape s;
    *warps = *ctas = 0;
    if (pick_shape(A, ndep, o, true, o.formal == 1, *warps, s) != cudaSuccess) return;
    *ctas = o.ctas_per_sm > 0 ? std::min(o.ctas_per_sm, s.per_sm) : s.per_sm;
}

cudaError_t launch_mali(const DevAtom &A, const ColumnArrays &c, const void *lane_tab, int npad, const float4 *vtab,
                        double nref, double *nghist, size_t nghist_cap, int *queue, const IterLaunch &o,
                        cudaStream_t st, float *ms_out, int *grid_out, char *err, size_t errn)
{
    if (A.nphi && !(o.phic && mali_phic_bytes_per_block(A, c.ndep, o.precision) <= o.phic_cap)) {
        snprintf(err, errn, "no profile cache");
        return cudaErrorInvalidValue;
    }
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, st);
    cudaError_t e = launch_mali_prealloc(A, c, lane_tab, npad, vtab, nref, nghist, nghist_cap, queue, o, st, grid_out,
                                         err, errn);
    cudaEventRecord(e1, st);
    if (e == cudaSuccess) e = cudaEventSynchronize(e1);
    if (e == cudaSuccess && ms_out) cudaEventElapsedTime(ms_out, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return e;
}

// The launch itself: no timing events (event objects are driver
// allocations), scratch pointers supplied by the caller, no wait.
cudaError_t launch_mali_prealloc(const DevAtom &A, const ColumnArrays &c, const void *lane_tab, int npad,
                                 const float4 *vtab, double nref, double *nghist, size_t nghist_cap, int *queue,
                                 const IterLaunch &o, cudaStream_t st, int *grid_out, char *err, size_t errn)
{
    KParams p = make_params(A, c, lane_tab, npad, vtab, nref, nghist, queue, o);
    // without a profile cache (callers that cannot allocate) the sweep
    // evaluates the profiles; partial redistribution always has the cache
    // (the FP32 linear sweep keeps its totals there too, also of an atom without lines)
    const bool bez = o.formal == 1, cache = p.phic || (!A.nphi && (o.precision == 0 || A.nprd || bez));
    if (!cache && A.nprd) {
        snprintf(err, errn, "the partial-redistribution kernel needs the profile cache");
        return cudaErrorInvalidValue;
    }
    if (bez && !cache) {
        snprintf(err, errn, "the Bezier formal solver needs the profile cache (an earlier rh_iterate or rh_solve)");
        return cudaErrorInvalidValue;
    }
    int bw = 0;
    Shape s;
    cudaError_t e = pick_shape(A, p.N, o, cache, bez, bw, s);
    if (e != cudaSuccess) return e;
    if (s.per_sm < 1) {
        snprintf(err, errn, "column kernel does not fit: %zu B shared memory, %d threads", s.sm, bw * kWarp);
        return cudaErrorInvalidConfiguration;
    }
    p.split = s.split;
    p.slot_rows = s.slot_rows;
    p.piece = s.piece;
    p.nsp = s.nsp;
    p.nvp = s.nvp;
    const SmemLayout lo = o.precision == 1 ? smem_layout<float>(A.nlev, p.N, 0, A.ncont, A.nline, s.slot_rows, 0)
                                           : smem_layout<double>(A.nlev, p.N, 0, A.ncont, A.nline, s.slot_rows, 0);
    p.scr[0] = (int)((lo.slot + 15) & ~(size_t)15);
    p.scr[1] = (int)lo.vtab;
    p.scr[2] = (int)lo.ring;
    const int64_t grid = grid_of(A, p, o, s, nghist_cap);
    if (grid < 1) {
        snprintf(err, errn, "scratch of one column (Ng history %zu B) exceeds the capacity (%zu B)",
                 mali_nghist_bytes_per_block(A, p.N), nghist_cap);
        return cudaErrorInvalidValue;
    }
    *grid_out = (int)grid;
    if (o.persistent) {
        e = cudaMemsetAsync(queue, 0, sizeof(int), st);
        if (e != cudaSuccess) return e;
    }
    void *args[] = {(void *)&A, (void *)&p};
    return cudaLaunchKernel(s.fn, dim3((unsigned)grid), dim3(bw * kWarp), args, s.sm, st);
}

}  // namespace rh
