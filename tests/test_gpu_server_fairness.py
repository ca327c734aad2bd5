"""A request whose packets need general events keeps its share of a served round when they share a
warp with packets trapped in the line core: counted in rounds, on a server of one warp.  While a
general event waits at most four core events run before it, so a round that holds B general events
without the trapped packets holds at least B / 5 with them (16 core events to one: B / 17)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_11603_gb300 import thor
    c = thor.Context(0)
    yield c
    c.close()


def test_trapped_packets_do_not_starve_general_events(ctx):
    # far in the wing of thin gas, scattered by dust alone: tau_dust^2 / 2 general events
    thin = dict(R_in=0.5, N_HI=1e12, T=1e4, v_max=10.0, tau_dust=40.0, albedo=1.0, g_hg=0.0, phase="isotropic",
                X0=1000.0, n_photons=8, seed=5, n_bins=16)
    trapped = dict(R_in=0.0, tau0=1e7, T=1e4, phase="dipole", n_photons=16, seed=6, n_bins=16)
    rounds, got = [], []
    for with_trapped in (False, True):
        srv = ctx.server(max_requests=4, events_per_round=64, n_slots=32, block_size=32, priority=False)
        if with_trapped:
            first = srv.submit(**trapped)
            while srv.stats()["rounds"] < 8:  # its packets are in flight
                pass
        before = srv.stats()["rounds"]
        r = srv.wait(srv.submit(**thin), timeout_ms=120000)
        rounds.append(srv.stats()["rounds"] - before)
        if with_trapped:
            assert not srv.poll(first)  # it was in flight all the while
            srv.cancel(first)
        got.append(r)
        srv.close()
    assert rounds[0] >= 8  # the thin request takes many rounds by itself
    assert rounds[1] <= 6 * rounds[0] + 4, rounds
    assert np.array_equal(got[0].spectrum, got[1].spectrum)
    assert got[0].stats["n_dust_scat"] == got[1].stats["n_dust_scat"] > 1000
