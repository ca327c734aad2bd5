"""The reweighting kernel's chunks, target groups and bins against FP64, element by element (1e-5
relative, as the other reweighting test): photon counts around the sorted chunks, target counts
around the 32 lanes, both sides of the line between the two kernels, one bin and the most bins, photons outside the range or not escaped."""
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


@pytest.mark.parametrize("n,K,nb", [(1, 1, 1), (255, 2, 7), (256, 33, 50), (257, 31, 4096), (2047, 3, 100),
                                    (2049, 64, 5), (70000, 5, 300), (70001, 300, 1), (400000, 40, 400),
                                    (257, 8300, 40), (2047, 1030, 100), (2049, 1025, 5), (65536, 32, 60),
                                    (65537, 33, 60)])
def test_chunks_against_fp64(ctx, n, K, nb):
    rng = np.random.default_rng(n + K)
    X0 = rng.uniform(-2500.0, 2500.0, n).astype(np.float32)
    X = (X0 + rng.normal(0.0, 700.0, n)).astype(np.float32)
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
