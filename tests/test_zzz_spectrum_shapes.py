"""Emergent spectra at the edges of the spectrum kernel's split: wavelength counts around a warp and a block, few
columns (depths split over threads) and many, two depths, more depths than one shared-memory table holds, and the
FP64 Voigt function over its branches (|v| below and above 8, 10, 14, 24).  Against the FP64 oracle on given
populations; tolerances as in the parity tests (1e-10 FP64, 1e-4 FP32 opacities rounded once per depth)."""
import numpy as np
import pytest

import rh_synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ncol,ndep,nlam", [(1, 2, 1), (1, 13, 33), (3, 82, 31), (2, 300, 40), (40, 82, 257),
                                            (90, 17, 64)])
def test_spectrum_shapes_match_oracle(orc, ncol, ndep, nlam):
    import paper_1411_1079_gb300 as rh
    rh.build()
    atom = rh_synth.hydrogen_like_atom()
    cols = rh_synth.chromosphere_cube(nx=ncol, ny=1, ndep=ndep, seed=8)
    g = rh.Context(0)
    g.setup_atom(atom)
    g.load_columns(cols)
    o = orc.Oracle()
    o.setup_atom(atom)
    o.load_columns(cols)
    rng = np.random.default_rng(ndep)
    n = o.lte()[0] * np.exp(rng.uniform(-0.5, 0.5, (ncol, atom["nlev"], ndep)))
    g.set_populations(n)
    o.set_populations(n)
    # line core to far wing of Lyman alpha and H alpha, continua, and a long wavelength (small h nu / kT)
    lam = np.concatenate([np.linspace(121.35e-9, 121.85e-9, nlam // 2), np.linspace(655.9e-9, 657.1e-9, nlam // 3)])
    lam = np.concatenate([lam, np.geomspace(85e-9, 60e-6, nlam - lam.size)])
    for mu in (1.0, 0.35):
        Io = o.emergent_spectrum(mu, lam)
        assert np.max(np.abs(g.emergent_spectrum(mu, lam, precision=0) / Io - 1)) < 1e-10
        assert np.max(np.abs(g.emergent_spectrum(mu, lam, precision=1) / Io - 1)) < 1e-4
