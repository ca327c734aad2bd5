"""Columns most of whose pairs are near (hot gas, or a box of few Doppler widths) are evaluated at
every bin: against the FP64 oracle (1e-5 relative, the bound of the other forest tests), and the
same bits in the whole box as where several CTAs and warps share a column.  Bin counts around one
to eight bins per thread, columns around the blocks of 32 cells and the staged chunk, and one
whose first chunk is cold and whose second is hot."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_11603_gb300 import thor
    c = thor.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n_bins,nz,dv,T0", [(129, 33, 3.0, 1e5), (256, 64, 2.0, 1e5), (257, 40, 2.0, 1e6), (513, 31, 4.0, 1e6),
                                             (769, 100, 1.0, 1e5), (1025, 128, 1.0, 1e6), (1537, 90, 1.0, 3e4),
                                             (2047, 1024, 1.0, 1e7), (2048, 1100, 1.0, 0.0)])
def test_hot_columns(ctx, orc, n_bins, nz, dv, T0):
    from paper_2507_11603_gb300 import synth
    ny, nx = 10, 32  # 320 sightlines: every column is one CTA's
    n, T, v = synth.forest_fields_numpy((nz, ny, nx), seed=n_bins, T0=T0 or 1e4)
    if T0 == 0.0:
        T[1024:] = 1e9
    kw = dict(ds_cm=synth.forest_scale(2.0, dv), dv_cell=dv, n_bins=n_bins, dv_bin=nz * dv / n_bins)
    whole = ctx.forest(n, T, v, **kw)
    sel = np.arange(0, 320, 53)
    ref = orc.forest(n, T, v, sel % nx, sel // nx, **kw)
    assert (np.abs(whole[sel].astype(np.float64) - ref) / ref).max() < 1e-5
    for first, count in ((0, 30), (200, 70), (319, 1)):
        part = ctx.forest(n, T, v, first=first, count=count, **kw)
        assert np.array_equal(part.view(np.uint32), whole[first:first + count].view(np.uint32)), (first, count)
