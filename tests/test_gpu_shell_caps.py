"""Photons stopped at a scattering cap, in flight, in the core or in the wing, have the same records
bit by bit whichever kernel finished them: in one launch, with packets given away in its tail,
re-packed between launches (tail compaction) and resumed there."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
GEOS = [dict(R_in=0.2, N_HI=1e17, T=1e4, v_max=400.0, tau_dust=0.1, phase="dipole"),
        dict(R_in=0.5, N_HI=1e18, T=1e4, v_max=100.0, tau_dust=1.0, albedo=0.5, phase="mixed"),
        dict(R_in=0.9, N_HI=1e19, T=1e4, v_max=200.0, phase="dipole")]


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_11603_gb300 import thor
    c = thor.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("geo", GEOS)
@pytest.mark.parametrize("cap", [3, 60, 2000])
def test_capped_photons_do_not_depend_on_the_launch(ctx, geo, cap):
    g = ctx.shell(**geo)
    kw = dict(n_photons=40000, seed=9, sigma=60.0, n_bins=50, X_min=-800.0, X_max=800.0, raw=True, max_scat=cap)
    ctx.set_tail_share(False)
    a = ctx.run(g, **kw)
    ctx.set_tail_share(True)
    out = [ctx.run(g, **kw)]
    for spill, phases in ((16, 24), (24, 4)):
        ctx.set_tail(spill, phases)
        out.append(ctx.run(g, **kw))
    ctx.set_tail(0, 24)
    assert a.stats["n_capped"] > 10
    for b in out:
        assert np.array_equal(np.asarray(a.raw_X).view(np.uint32), np.asarray(b.raw_X).view(np.uint32))
        assert np.array_equal(a.raw_nscat, b.raw_nscat) and np.array_equal(a.raw_status, b.raw_status)
        for k in ("n_escaped", "n_absorbed", "n_capped", "n_scat", "n_dust_scat", "n_upar_iters", "n_steps"):
            assert a.stats[k] == b.stats[k], k
