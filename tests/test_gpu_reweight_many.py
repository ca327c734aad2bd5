"""Reweighting of many photons for few targets against FP64, element by element (1e-5 relative, the
bound of the other reweighting tests): photon counts and target counts on both sides of the lines
between the kernels, bins on both sides of FP32 sums, all photons in one bin, a column that is
not a number."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
SAMPLE = (800.0, 740.0, 2500.0)


def pdf(p, X):
    sigma, ew, C = p
    pl = ew / (ew + 2 * C)
    g = pl / (np.sqrt(2 * np.pi) * sigma) * np.exp(-0.5 * (X / sigma) ** 2)
    return np.where(np.abs(X) <= C, g + (1 - pl) / (2 * C), g)


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_11603_gb300 import thor
    c = thor.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n,K,nb,width", [(524288, 1, 60, 700.0), (524289, 1, 60, 700.0), (524289, 1, 1, 700.0),
                                          (600001, 2, 4096, 700.0), (1048576, 3, 1023, 700.0), (1100000, 6, 1022, 700.0),
                                          (262145, 4, 100, 700.0), (262145, 4, 101, 700.0), (262144, 4, 50, 700.0),
                                          (262145, 8, 31, 700.0), (262145, 9, 31, 700.0), (2097152, 6, 1500, 700.0),
                                          (1100000, 2, 200, 1e-3), (65536, 48, 100, 700.0), (65536, 49, 99, 700.0)])
def test_many_against_fp64(ctx, n, K, nb, width):
    rng = np.random.default_rng(n + K)
    X0 = rng.uniform(-2500.0, 2500.0, n).astype(np.float32)
    X = (rng.normal(0.0, width, n) + (X0 if width > 1.0 else 3.0)).astype(np.float32)
    col = rng.lognormal(0.0, 0.7, n).astype(np.float32)
    st = rng.choice([1, 1, 1, 2, 3], n).astype(np.uint8)
    tg = np.stack([rng.uniform(100, 800, K), rng.uniform(2000, 40000, K), np.full(K, 2500.0), rng.uniform(0, 2, K)], 1)
    got = ctx.reweight(X0, X, col, st, sample=SAMPLE, targets=tg, n_bins=nb, X_min=-2000.0, X_max=2000.0)
    f = (X - np.float32(-2000.0)) * np.float32(nb / 4000.0)
    b = np.where(f >= 0, np.where(f >= nb, nb + 1, np.minimum(f, 1e6).astype(np.int64)), nb)
    x0, c, ok = X0.astype(np.float64), col.astype(np.float64), st == 1
    for t in range(K):
        w = pdf(tg[t, :3], x0) / pdf(SAMPLE, x0) * np.exp(-tg[t, 3] * c)
        ref = np.bincount(b[ok], weights=w[ok], minlength=nb + 2) / n
        m = ref > 0
        assert np.array_equal(got[t] > 0, m)
        assert (np.abs(got[t][m] - ref[m]) / ref[m]).max(initial=0.0) < 1e-5


@pytest.mark.parametrize("nb", [40, 2000])
def test_a_column_that_is_not_a_number_stays_in_its_bin(ctx, nb):
    n = 600000
    X0 = np.linspace(-2400.0, 2400.0, n).astype(np.float32)
    col = np.ones(n, np.float32)
    col[n // 2] = np.nan
    got = ctx.reweight(X0, X0, col, np.ones(n, np.uint8), sample=SAMPLE, targets=[(300.0, 5000.0, 2500.0, 1.0)], n_bins=nb,
                       X_min=-2500.0, X_max=2500.0)[0]
    f = (X0[n // 2] - np.float32(-2500.0)) * np.float32(nb / 5000.0)
    assert np.flatnonzero(np.isnan(got)).tolist() == [int(f)]
