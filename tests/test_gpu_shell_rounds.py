"""The shell loop's core events in rounds (thor_ctx_set_bursts) against its general event, photon
by photon and bit by bit, where a round's shape changes: packets per warp from one to 32
(events per packet and round from 32 down to 4) and scattering caps around the depth of a
round."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
GEOS = [dict(T=1e4, tau0=3e3, phase="isotropic"),
        dict(R_in=0.9, N_HI=1e18, T=1e4, v_max=120.0, tau_dust=0.5, phase="dipole"),
        dict(R_in=0.5, N_HI=1e19, T=2e4, v_max=60.0, tau_dust=0.2, phase="dipole", core_skip=True)]


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_11603_gb300 import thor
    c = thor.Context(0)
    c.set_launch(32, 1)  # 152 warps: few photons already fill lanes
    yield c
    c.close()


@pytest.mark.parametrize("geo", GEOS)
@pytest.mark.parametrize("per_warp,cap", [(1, 0), (1, 33), (3, 17), (5, 16), (9, 15), (17, 5), (32, 4), (32, 1)])
def test_rounds_equal_general_events(ctx, geo, per_warp, cap):
    g = ctx.shell(**geo)
    kw = dict(n_photons=152 * per_warp - 1, seed=17, sigma=30.0, n_bins=64, X_min=-800.0, X_max=800.0, raw=True,
              max_scat=cap or 3000)
    ctx.set_bursts(0, 0)
    a = ctx.run(g, **kw)
    ctx.set_bursts(32, 1)
    b = ctx.run(g, **kw)
    assert np.array_equal(a.spectrum, b.spectrum)
    assert np.array_equal(a.raw_nscat, b.raw_nscat) and np.array_equal(a.raw_status, b.raw_status)
    assert np.array_equal(np.asarray(a.raw_X).view(np.uint32), np.asarray(b.raw_X).view(np.uint32))
    for k in ("n_scat", "n_dust_scat", "n_upar_iters", "n_steps", "n_escaped", "n_absorbed", "n_capped"):
        assert a.stats[k] == b.stats[k], k
