"""Power-law shells, H I and Mg II: packets saved in mid-flight and resumed -- given away in the tail
of a launch, re-packed between launches, or sliced by a server's rounds -- carry their whole state
(the interrupted flight, the pending safety distance, the column), so per-photon records are the
same bit by bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
GEOS = {"HI": (dict(R_in=0.2, N_HI=10 ** 17.5, T=1e4, v_max=150.0, alpha_rho=-1.0, alpha_v=0.8, tau_dust=0.3), 20000),
        "HI mixed": (dict(R_in=0.1, N_HI=10 ** 18.2, T=1e4, v_max=120.0, alpha_rho=-1.5, alpha_v=0.5, phase="mixed"), 6000),
        "MgII": (dict(species="MgII", R_in=1e-3, N_HI=10 ** 14.2, T=1e4, v_max=200.0, alpha_rho=0.0, alpha_v=1.0), 40000),
        "MgII thick": (dict(species="MgII", R_in=0.1, N_HI=10 ** 15.0, T=2e4, v_max=100.0, alpha_rho=-1.0, alpha_v=0.8,
                            tau_dust=0.4), 20000)}


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_11603_gb300 import thor
    c = thor.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("name", GEOS)
def test_resumed_packets_equal_uninterrupted_ones(ctx, name):
    geo, n = GEOS[name]
    g = ctx.shell(profile="power_law", **{"phase": "dipole", **geo})
    kw = dict(n_photons=n, seed=41, sigma=150.0, ew=500.0, C_cont=900.0, n_bins=60, X_min=-1500.0, X_max=1500.0, raw=True,
              raw_sweep=True)
    ctx.set_tail_share(False)
    a = ctx.run(g, **kw)
    ctx.set_tail_share(True)
    out = [ctx.run(g, **kw)]
    for launch in ((32, 1), (256, 0)):  # few warps: nearly every packet of the tail is given away
        ctx.set_launch(*launch)
        out.append(ctx.run(g, **kw))
    ctx.set_launch(128, 0)
    for spill, phases in ((16, 24), (24, 4)):
        ctx.set_tail(spill, phases)
        out.append(ctx.run(g, **kw))
    ctx.set_tail(0, 24)
    assert a.stats["n_steps"] > 128 * n / 4  # flights of more than one slice
    for b in out:
        assert np.array_equal(a.spectrum, b.spectrum)
        for k in ("raw_X", "raw_X0", "raw_col"):
            assert np.array_equal(np.asarray(getattr(a, k)).view(np.uint32), np.asarray(getattr(b, k)).view(np.uint32)), k
        assert np.array_equal(a.raw_nscat, b.raw_nscat) and np.array_equal(a.raw_status, b.raw_status)
        for k in ("n_escaped", "n_absorbed", "n_capped", "n_scat", "n_upar_iters", "n_steps"):
            assert a.stats[k] == b.stats[k], k


@pytest.mark.parametrize("events", [3, 64])
def test_served_slices_equal_one_launch(ctx, events):
    geo, n = dict(GEOS["HI"][0]), 3000
    common = dict(n_bins=60, X_min=-1500.0, X_max=1500.0, sigma=150.0, phase="dipole")
    one = ctx.run(ctx.shell(profile="power_law", phase="dipole", **geo), n_photons=n, seed=7,
                  **{k: v for k, v in common.items() if k != "phase"})
    srv = ctx.server(max_requests=2, events_per_round=events, n_slots=1024)
    r = srv.wait(srv.submit(profile="power_law", n_photons=n, seed=7, **geo, **common), timeout_ms=120000)
    srv.close()
    assert np.array_equal(one.spectrum, r.spectrum)
    for k in ("n_escaped", "n_absorbed", "n_scat", "n_upar_iters", "n_steps"):
        assert one.stats[k] == r.stats[k], k
