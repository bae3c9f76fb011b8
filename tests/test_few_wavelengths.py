"""Emergent spectra of many columns at fewer wavelengths than a warp has lanes: several columns share a block.  The
same wavelengths within a call of 64 (a column a block, compared with the oracle elsewhere) give the same bits."""
import numpy as np
import pytest

import rh_synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ncol,ndep", [(2501, 2), (2501, 13), (1300, 82), (9001, 33)])
def test_few_wavelengths_of_many_columns(ncol, ndep, precision):
    import paper_1411_1079_gb300 as rh
    rh.build()
    ctx = rh.Context(0)
    ctx.setup_atom(rh_synth.hydrogen_like_atom())
    ctx.load_columns(rh_synth.chromosphere_cube(nx=ncol, ny=1, ndep=ndep, seed=9))
    ns = ctx.lte()[0]
    ctx.set_populations(ns * np.exp(np.random.default_rng(ndep).uniform(-0.5, 0.5, ns.shape)))
    lam = np.concatenate([np.linspace(121.35e-9, 121.85e-9, 20), np.linspace(655.9e-9, 657.1e-9, 24),
                          np.geomspace(85e-9, 60e-6, 20)])
    ref = ctx.emergent_spectrum(0.8, lam, precision=precision)
    for n in (1, 2, 5, 8, 16, 17, 31):
        pick = np.linspace(3, 60, n).astype(int)
        got = ctx.emergent_spectrum(0.8, lam[pick], precision=precision)
        assert np.array_equal(got, ref[:, pick]), n
