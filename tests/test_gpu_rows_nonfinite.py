"""A value that is not finite at index 0 reaches only the rows that hold it (GPU).

The row kernels pad a row to its warp's longest with entries of weight 0 at index 0.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1607_01650_gb300 as dect  # noqa: E402


def _run(op, x, row, length, bad):
    """row, length: the rows that hold index 0, and their weights.  A row without it gives what it gives when the
    value is finite, up to the order of its sum: at most 150 positive terms, 150 x 2^-24 < 1e-5."""
    xt = torch.tensor(x, device="cuda")
    clean = op(xt).cpu().numpy()
    xt.view(x.shape[0], -1)[0, 0] = bad
    out = op(xt).cpu().numpy()
    np.testing.assert_array_equal(out[1:], clean[1:])
    out, clean = out[0].ravel(), clean[0].ravel()
    assert not np.isfinite(out[row[length > 1e-6]]).any()  # (a corner met within rounding may not count as met)
    rest = np.setdiff1d(np.arange(out.size), row)
    np.testing.assert_allclose(out[rest], clean[rest], rtol=1e-5)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("batch", [1, 2, 4, 8, 16, 17, 32, 64])
def test_fan_beam(batch, bad):
    g = synth.tiny_geometry(n=33, nv=11, nb=200, px=1.0, pitch=1.1, sod=80.0, sdd=160.0)  # rays miss the image
    plan = dect.Plan(g)
    ptr, pix, ln = plan.table()
    ray = np.repeat(np.arange(g.nv * g.nb), np.diff(ptr))
    assert (np.diff(ptr) == 0).any() and (pix == 0).any() and not (ray == 0).any()
    rng = np.random.default_rng(batch)
    x = rng.random((batch, g.n, g.n)).astype(np.float32)
    y = rng.random((batch, g.nv, g.nb)).astype(np.float32)
    _run(lambda v: dect.project(plan, v), x, ray[pix == 0], ln[pix == 0], bad)
    _run(lambda v: dect.backproject(plan, v), y, pix[ray == 0], ln[ray == 0], bad)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("batch", [1, 4, 16, 17])
def test_cone_beam(batch, bad):
    g = synth.ConeGeometry(n=17, nz=3, px=1.0, pz=1.3, nv=9, nr=9, nc=60, pu=1.3, pv=1.7, sod=60.0, sdd=130.0,
                           start=0.2, off_u=0.15)
    plan = dect.ConePlan(g)
    ptr, pix, ln = plan.table()
    ray = np.repeat(np.arange(g.nv * g.nr * g.nc), np.diff(ptr))
    assert (np.diff(ptr) == 0).any()
    rng = np.random.default_rng(batch)
    x = rng.random((batch, g.nz, g.n, g.n)).astype(np.float32)
    y = rng.random((batch, g.nv, g.nr, g.nc)).astype(np.float32)
    _run(lambda v: dect.project_cone(plan, v), x, ray[pix == 0], ln[pix == 0], bad)
    _run(lambda v: dect.backproject_cone(plan, v), y, pix[ray == 0], ln[ray == 0], bad)
