"""The FP64 Voigt function on both sides of its branches (|v| = 16: Taylor polynomials of Dawson's integral or the
asymptotic series; |v| = 24 and 60: 10, 8 or 6 terms of it), through emergent spectra of columns at one temperature and
at rest, whose |v| at a wavelength is the same at every depth.  Against the FP64 oracle, as in the parity tests."""
import numpy as np
import pytest

import rh_synth

pytestmark = pytest.mark.gpu

C, K_B, AMU = 2.99792458e8, 1.380649e-23, 1.66053906660e-27


@pytest.mark.parametrize("line", [0, 4])
@pytest.mark.parametrize("T", [4000.0, 9000.0])
def test_both_sides_of_every_branch(orc, line, T):
    import paper_1411_1079_gb300 as rh
    rh.build()
    atom = rh_synth.hydrogen_like_atom()
    cols = rh_synth.chromosphere_cube(nx=2, ny=1, ndep=24, seed=3)
    cols["T"] = np.full_like(cols["T"], T)
    cols["vz"] = np.zeros_like(cols["vz"])
    E = np.asarray(atom["E_J"])
    nu0 = (E[atom["line_u"][line]] - E[atom["line_l"][line]]) / 6.62607015e-34
    vth = np.sqrt(2.0 * K_B * T / (atom["mass_amu"] * AMU))
    v = np.array([0.01, 3.0, 15.9, 15.999, 16.001, 16.1, 23.99, 24.01, 59.99, 60.01, 70.0])
    lam = C / (nu0 * (1.0 + np.concatenate([-v, v]) * vth / C))
    g = rh.Context(0)
    g.setup_atom(atom)
    g.load_columns(cols)
    o = orc.Oracle()
    o.setup_atom(atom)
    o.load_columns(cols)
    n = o.lte()[0] * np.exp(np.random.default_rng(1).uniform(-0.5, 0.5, (2, atom["nlev"], 24)))
    g.set_populations(n)
    o.set_populations(n)
    Io = o.emergent_spectrum(1.0, lam)
    assert np.max(np.abs(g.emergent_spectrum(1.0, lam, precision=0) / Io - 1)) < 1e-10
