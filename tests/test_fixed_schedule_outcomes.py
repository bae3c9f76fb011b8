"""Fixed numbers of FP32 iterations end the same way whatever the launch shape, and as they always have.  About one
column in a thousand of a cube loses a positive population in its first iterations, and a few in 65536 lie so near
that edge that any other rounding of the sweep's contributions, or another order of their sums, moves the iteration
at which they fail or saves them.  OUTCOMES holds such columns -- (seed, column): (status, iterations) of
`chromosphere_cube(nx=8192, ny=1, ndep=82, seed)` (4096 columns with partial redistribution) -- as the sweeps that add
ray after ray (c w phi) I to a tile's accumulators end them, with R_II-A integrated term by term (status 1: all
iterations done, 2: a population not positive)."""
import numpy as np
import pytest

import rh_synth

pytestmark = pytest.mark.gpu

LINEAR = {(100, 5310): (2, 9), (101, 1553): (2, 5), (103, 130): (2, 7), (104, 4245): (2, 6), (104, 6040): (2, 7),
          (105, 3242): (2, 10), (105, 5477): (1, 12), (106, 492): (1, 12), (106, 2110): (1, 12), (106, 3667): (1, 12),
          (106, 5066): (1, 12)}
BEZIER = {(100, 3994): (2, 6), (101, 1985): (1, 8), (103, 5184): (2, 6), (104, 8125): (2, 6), (106, 3648): (1, 8),
          (106, 7772): (2, 2), (107, 1628): (1, 8), (107, 3834): (2, 2)}
PRD = {(301, 1207): (1, 8), (301, 3232): (1, 8), (305, 3136): (1, 8)}
HYBRID = {(301, 1847): (1, 8), (303, 2398): (1, 8), (303, 2474): (1, 8), (303, 3128): (2, 6), (303, 3745): (2, 6),
          (304, 4066): (1, 8)}


def _context(rh, atom, cols):
    ctx = rh.Context(0)
    ctx.setup_atom(atom)
    ctx.load_columns(cols)
    return ctx


@pytest.fixture(scope="module")
def rh():
    import paper_1411_1079_gb300 as m
    m.build()
    return m


CRD_ATOM = rh_synth.hydrogen_like_atom()
PRD_ATOM = rh_synth.hydrogen_like_atom(prd_lines=((1, 2), (1, 3)), prd_nlambda=64)


@pytest.mark.parametrize("atom,ncol,kw,outcomes", [
    (CRD_ATOM, 8192, dict(formal=0, maxiter=12), LINEAR), (CRD_ATOM, 8192, dict(formal=1, maxiter=8), BEZIER),
    (PRD_ATOM, 4096, dict(maxiter=8, prd_eps0=0.05, prd_hybrid=0), PRD),
    (PRD_ATOM, 4096, dict(maxiter=8, prd_eps0=0.05, prd_hybrid=1), HYBRID)], ids=["linear", "bezier", "prd", "hybrid"])
def test_nearly_singular_columns_end_as_recorded(rh, atom, ncol, kw, outcomes):
    parts = []
    for seed in sorted({s for s, _ in outcomes}):
        cube = rh_synth.chromosphere_cube(nx=ncol, ny=1, ndep=82, seed=seed)
        parts.append(rh_synth.subset(cube, [c for s, c in sorted(outcomes) if s == seed]))
    cols = {k: np.concatenate([p[k] for p in parts]) for k in parts[0]}
    ctx = _context(rh, atom, cols)
    ctx.iterate(tol=0.0, precision=1, **kw)
    _, iters, status, _ = ctx.populations()
    got = {k: (int(status[i]), int(iters[i])) for i, k in enumerate(sorted(outcomes))}
    assert got == outcomes


# 8 angles and 82 depths: the largest accumulators and profiles per block, the most passes over the angles
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("formal", [0, 1])
@pytest.mark.parametrize("nmu", [2, 8])
def test_results_do_not_depend_on_the_launch_shape(rh, precision, formal, nmu):
    atom = rh_synth.hydrogen_like_atom(nmu=nmu)
    cube = rh_synth.chromosphere_cube(nx=400, ny=1, ndep=82, seed=21)
    few = rh_synth.subset(cube, slice(0, 3))
    ref = None
    for cols, warps in ((few, 0), (few, 4), (few, 8), (few, 1)) + (((cube, 0),) if precision else ()):
        ctx = _context(rh, atom, cols)
        ctx.iterate(maxiter=3, tol=0.0, ng_order=0, precision=precision, formal=formal, block_warps=warps)
        n = ctx.populations()[0][:3]
        ref = n if ref is None else ref
        assert np.array_equal(n, ref), warps


def _iterate_uncached(ctx, shape, **kw):
    """rh_iterate_noalloc on a context without a profile cache: the sweep evaluates the profiles itself."""
    import torch
    out = (torch.zeros(shape, dtype=torch.float64, device="cuda"),
           torch.zeros(shape[0], dtype=torch.int32, device="cuda"),
           torch.zeros(shape[0], dtype=torch.uint8, device="cuda"),
           torch.zeros(shape[0], dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    ctx.iterate_noalloc(*out, **kw)
    torch.cuda.synchronize()
    return out[0].cpu().numpy()


# Below a cold temperature minimum the intensities of the Lyman lines are 1e-26 and less, their profiles 1e-18 in the
# wings: the up-rates need the FP32 terms in an order that stays in range.  Tolerance: some 150 roundings of 2^-24
# between a contribution and the populations.
@pytest.mark.parametrize("nmu", [1, 2, 3, 5, 8])
@pytest.mark.parametrize("tmin", [3000.0, 2450.0, 2000.0, 1700.0])
def test_cold_temperature_minimum(rh, tmin, nmu):
    atom = rh_synth.hydrogen_like_atom(nmu=nmu)
    cols = rh_synth.chromosphere_cube(nx=8, ny=1, ndep=82, seed=7)
    T, low = cols["T"], cols["T"].min(axis=1, keepdims=True)
    cols["T"] = np.ascontiguousarray(np.where(T < 7000.0, 7000.0 - (7000.0 - T) * (7000.0 - tmin) / (7000.0 - low), T))
    kw = dict(maxiter=12, tol=0.0, ng_order=0, precision=1)
    n32 = _iterate_uncached(_context(rh, atom, cols), (8, atom["nlev"], 82), **kw)
    ctx = _context(rh, atom, cols)
    ctx.iterate(**dict(kw, precision=0))
    n64 = ctx.populations()[0]
    ctx.iterate(**kw)
    assert np.array_equal(ctx.populations()[0], n32)      # with and without the cache, to the bit
    assert np.max(np.abs(n32 / n64 - 1)) < 1e-5
