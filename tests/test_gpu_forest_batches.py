"""A sightline's optical depths are the same bits however it is batched: in the whole box, in
sub-ranges small enough that several CTAs (and warps) share a column, alone, and in rows staged
from host memory.  Column lengths around the staged chunk and the blocks of 32 cells, bin counts
on both sides of where the number of intervals changes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_11603_gb300 import thor
    c = thor.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n_bins,nz,dv", [(64, 64, 2.0), (129, 200, 1.0), (300, 1023, 1.0), (513, 300, 2.5), (1025, 1025, 2.0),
                                          (2048, 70, 20.0), (2048, 2100, 1.0)])
def test_batches_give_the_same_bits(ctx, n_bins, nz, dv):
    import torch
    from paper_2507_11603_gb300 import synth
    ny, nx = 20, 32  # 640 sightlines: every column is one CTA's
    f = [torch.as_tensor(a, device="cuda") for a in synth.forest_fields_numpy((nz, ny, nx), seed=n_bins + nz)]
    kw = dict(ds_cm=synth.forest_scale(2.0, dv), dv_cell=dv, n_bins=n_bins, dv_bin=nz * dv / n_bins)
    whole = ctx.forest(*f, **kw).cpu().numpy().view(np.uint32)
    for first, count in ((0, 320), (7, 150), (100, 70), (300, 30), (411, 15), (77, 7), (639, 1)):
        part = ctx.forest(*f, first=first, count=count, **kw).cpu().numpy().view(np.uint32)
        assert np.array_equal(part, whole[first:first + count]), (first, count)
    host = [a.cpu().numpy() for a in f]
    for rows in (1, 7):
        assert np.array_equal(ctx.forest(*host, stage_rows=rows, **kw).view(np.uint32), whole), rows
