"""The forest kernel's intervals and Chebyshev nodes against the FP64 oracle, element by element
(1e-5 relative, the bound of the other forest tests): bin counts on both sides of where the
number of intervals, the coarse level and the two bins per lane change, column lengths
around the staged chunk, and sightline counts that split a column over several CTAs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_11603_gb300 import thor
    c = thor.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n_bins,nz,dv", [(2, 3, 9.0), (63, 40, 4.0), (64, 64, 2.0), (65, 33, 8.0), (128, 200, 1.0),
                                          (129, 200, 1.0), (512, 300, 2.5), (513, 300, 2.5), (1024, 1023, 2.0),
                                          (1025, 1025, 2.0), (2047, 700, 3.0), (2048, 1024, 2.0), (2048, 60, 1.5)])
def test_intervals_against_oracle(ctx, orc, n_bins, nz, dv):
    from paper_2507_11603_gb300 import synth
    n, T, v = synth.forest_fields_numpy((nz, 2, 3), seed=n_bins)
    kw = dict(ds_cm=synth.forest_scale(2.0, dv), dv_cell=dv, n_bins=n_bins, dv_bin=nz * dv / n_bins)
    got = ctx.forest(n, T, v, **kw).astype(np.float64)
    sel = np.arange(6)
    ref = orc.forest(n, T, v, sel % 3, sel // 3, **kw)
    assert (np.abs(got - ref) / ref).max() < 1e-5


@pytest.mark.parametrize("nxy", [(1, 1), (40, 8)])
def test_cells_of_extreme_width(ctx, orc, nxy):
    """Cells from 30 K to 3e7 K in one column: cores narrower than a bin and wider than half the
    box, next to one another."""
    rng = np.random.default_rng(3)
    shape = (256,) + nxy
    n = (1e-10 * np.exp(rng.standard_normal(shape))).astype(np.float32)
    T = (10.0 ** rng.uniform(1.5, 7.5, shape)).astype(np.float32)
    v = (200.0 * rng.standard_normal(shape)).astype(np.float32)
    kw = dict(ds_cm=3e22, dv_cell=2.0, n_bins=1000, dv_bin=0.512)
    got = ctx.forest(n, T, v, **kw).astype(np.float64)
    sel = np.arange(0, nxy[0] * nxy[1], 40)
    ref = orc.forest(n, T, v, sel % nxy[1], sel // nxy[1], **kw)
    assert (np.abs(got[sel] - ref) / ref).max() < 1e-5


def test_an_infinite_cell_reaches_every_bin(ctx):
    n = np.full((128, 1, 2), 1e-10, np.float32)
    n[5, 0, 1] = np.inf
    T = np.full_like(n, 1e4)
    v = np.zeros_like(n)
    tau = ctx.forest(n, T, v, ds_cm=3e22, dv_cell=8.0, n_bins=1024, dv_bin=1.0)
    assert np.isfinite(tau[0]).all() and np.isinf(tau[1]).all()
