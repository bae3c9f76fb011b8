"""rh_solve reports the launch shape that ran: the library's default warps per block (FP32 linear: 16 while every column
has an SM of its own, 8 beyond; FP64 linear: 8; FP64 with the Bezier solver: 4), halved where a column does not fit."""
import pytest

import rh_synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rh():
    import paper_1411_1079_gb300 as m
    m.build()
    return m


def _stats(rh, ncol, ndep, atom=None, **kw):
    ctx = rh.Context(0)
    ctx.setup_atom(atom or rh_synth.hydrogen_like_atom())
    ctx.load_columns(rh_synth.chromosphere_cube(nx=ncol, ny=1, ndep=ndep, seed=4))
    return ctx.solve(maxiter=1, rescue=False, autotune=0, **kw)


@pytest.mark.parametrize("ncol,kw,warps", [(2, dict(precision=1), 16), (400, dict(precision=1), 8),
                                           (2, dict(precision=0), 8), (2, dict(precision=0, formal=1), 4),
                                           (2, dict(precision=1, formal=1), 8), (2, dict(precision=1, block_warps=6), 6)])
def test_reported_shape_is_the_default(rh, ncol, kw, warps):
    s = _stats(rh, ncol, 32, **kw)
    assert s["block_warps"] == warps and s["ctas_per_sm"] >= 1


def test_scratch_that_does_not_fit_halves_the_warps(rh):
    # three lines per tile and eight angles: 16 warps' profile rings fill the block at some depths, 8 warps' do not
    atom = rh_synth.hydrogen_like_atom(qwing=1000.0, nmu=8)
    seen = {n: _stats(rh, 1, n, atom, precision=1)["block_warps"] for n in (20, 60, 82, 100, 128, 160)}
    assert set(seen.values()) == {16, 8}, seen
