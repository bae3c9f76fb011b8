"""Kernels at the edges of their tilings: training GEMMs at sizes that select each copy width and leave remainders of
every tile dimension, the column kernel over angle counts (vectors of rays per pass) and level counts (sizes of the
rate-equation solve), and Stokes spectra around a round of a block.  Tolerances are those of the parity tests:
gradients of the BF16 network to cosine 0.999 and relative L2 2e-2 per tensor against the FP64 reference; FP64
populations of a fixed schedule to 1e-9, the FP32 sweep to 1e-3; FP64 Stokes to 1e-9 of I, FP32 to 1e-4."""
import numpy as np
import pytest

import rh_synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rh():
    import paper_1411_1079_gb300 as m
    m.build()
    return m


# (levels, depths, hidden, rows): 16-byte copies; 8-byte (outputs 4 x 13 = 52); element copies (outputs 5 x 13 = 65)
@pytest.mark.parametrize("nbound,ndep,hidden,rows", [(3, 16, 64, 130), (3, 13, 40, 33), (4, 13, 50, 70), (3, 2, 8, 1)])
def test_training_gradients_at_odd_sizes(rh, nbound, ndep, hidden, rows):
    from oracle import mlp
    atom = rh_synth.small_atom(nbound=nbound)
    cols = rh_synth.chromosphere_cube(nx=rows, ny=1, ndep=ndep, seed=5)
    g = rh.Context(0)
    g.setup_atom(atom)
    g.load_columns(cols)
    rng = np.random.default_rng(1)
    ns, ne = g.lte()
    n = ns * np.exp(rng.uniform(-0.5, 0.5, ns.shape))
    g.set_populations(n)
    X = mlp.features(cols["T"], ne, cols["nH"], cols["vz"])
    Y = np.log(n / ns).reshape(rows, -1)
    dims = (X.shape[1], hidden, 2, Y.shape[1])
    parts = []
    for di, do in mlp.layer_dims(*dims):
        parts += [rng.standard_normal(do * di) * np.sqrt(2.0 / di), 0.1 * rng.standard_normal(do)]
    scale = np.maximum(np.abs(X).max(axis=0), 1.0)
    state = np.concatenate(parts + [0.5 * scale, 1.0 / scale]).astype(np.float32)
    g.surrogate_init(hidden=hidden, nhidden=2, seed=0)
    g.surrogate_set_state(state)
    loss, grad = g.surrogate_loss_grad(np.arange(rows))
    loss_o, grad_o = mlp.loss_grad(state.astype(np.float64), dims, X, Y)
    assert loss == pytest.approx(loss_o, rel=1e-2)
    off = 0
    for di, do in mlp.layer_dims(*dims):
        for size in (di * do, do):
            a, b = grad[off:off + size].astype(np.float64), grad_o[off:off + size]
            off += size
            assert np.linalg.norm(a - b) < 2e-2 * np.linalg.norm(b) + 1e-12
            assert a @ b > 0.999 * np.linalg.norm(a) * np.linalg.norm(b) - 1e-24


@pytest.mark.parametrize("nmu", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("nbound,ndep", [(2, 2), (3, 33), (6, 12)])
def test_column_kernel_over_angles_and_levels(rh, orc, nmu, nbound, ndep):
    atom = rh_synth.small_atom(nbound=nbound, nmu=nmu)
    cols = rh_synth.chromosphere_cube(nx=5, ny=1, ndep=ndep, seed=3)
    g = rh.Context(0)
    g.setup_atom(atom)
    o = orc.Oracle()
    o.setup_atom(atom)
    for formal in (0, 1):
        g.load_columns(cols)
        o.load_columns(cols)
        o.iterate(maxiter=4, tol=0.0, ng_order=0, formal=formal)
        no = o.populations()[0]
        for prec, tol in ((0, 1e-9), (1, 1e-3)):
            g.iterate(maxiter=4, tol=0.0, ng_order=0, precision=prec, formal=formal)
            assert np.max(np.abs(g.populations()[0] / no - 1)) < tol, (formal, prec)


@pytest.mark.parametrize("nlam", [1, 31, 224, 225, 401])
def test_stokes_wavelength_counts(rh, orc, nlam):
    atom = rh_synth.hydrogen_like_atom()
    cols = rh_synth.chromosphere_cube(nx=3, ny=1, ndep=21, seed=6)
    g = rh.Context(0)
    g.setup_atom(atom)
    g.load_columns(cols)
    o = orc.Oracle()
    o.setup_atom(atom)
    o.load_columns(cols)
    n = o.lte()[0] * np.exp(np.random.default_rng(2).uniform(-0.5, 0.5, (3, atom["nlev"], 21)))
    g.set_populations(n)
    o.set_populations(n)
    fld = (np.full((3, 21), 0.15), np.full((3, 21), 0.9), np.full((3, 21), 2.1))
    lam = 656.46e-9 + np.linspace(-0.4e-9, 0.4e-9, nlam)
    ref = o.emergent_stokes(4, 1.5, *fld, lam)
    for prec, tol in ((0, 1e-9), (1, 1e-4)):
        got = g.emergent_stokes(4, 1.5, *fld, lam, precision=prec)
        assert np.max(np.abs(got - ref) / ref[..., :1]) < tol
