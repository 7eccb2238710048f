"""A and A^T on either side of the lines between their routes (GPU), against the oracle.

A^T of narrow passes takes a warp per pixel up to 9728 pixels (14592 where a pixel
meets 256 rays or more) and eight lanes beyond; A takes the line
table, above four images from 3.5 million elements on.  Cone-beam A takes a warp per ray up
to 24320 rays.  Tolerance 1e-5 relative L2, that of the projector tests.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1607_01650_gb300 as dect  # noqa: E402


def _geometry(n, nv, nb):
    return synth.tiny_geometry(n=n, nv=nv, nb=nb, px=1.0, pitch=1.2, sod=4.0 * n, sdd=8.0 * n)


SIZES = {
    "98": (98, 20, 150), "99": (99, 20, 150),          # 9604 and 9801 pixels of about 40 rays
    "120": (120, 150, 170), "121": (121, 150, 170),    # 14400 and 14641 pixels of about 270 rays
    "120 short rows": (120, 140, 170),                 # about 250 rays
    "below 3.5 million": (168, 90, 160), "above 3.5 million": (168, 100, 160),
}


def test_the_sizes_lie_where_they_are_meant_to():
    nnz = {k: dect.Plan(_geometry(*s)).nnz for k, s in SIZES.items()}
    assert nnz["98"] < 256 * 9604
    assert nnz["120"] >= 256 * 120 ** 2 and nnz["121"] >= 256 * 121 ** 2 and nnz["120 short rows"] < 256 * 120 ** 2
    assert nnz["below 3.5 million"] < 3.5e6 <= nnz["above 3.5 million"] < 4e6


@pytest.mark.parametrize("name", sorted(SIZES))
@pytest.mark.parametrize("batch", [1, 4, 5, 8, 13, 16])
def test_operators_match_oracle(name, batch):
    g = _geometry(*SIZES[name])
    plan, t = dect.Plan(g), oracle.table(g)
    rng = np.random.default_rng(batch)
    x = rng.standard_normal((batch, g.n, g.n)).astype(np.float32)
    y = rng.standard_normal((batch, g.nv, g.nb)).astype(np.float32)
    p = dect.project(plan, torch.tensor(x, device="cuda")).cpu().numpy()
    b = dect.backproject(plan, torch.tensor(y, device="cuda")).cpu().numpy()
    for k in (0, batch // 2, batch - 1):
        for got, want in ((p[k], oracle.project(t, x[k].astype(np.float64))),
                          (b[k], oracle.backproject(t, y[k].astype(np.float64)))):
            assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)


@pytest.mark.parametrize("n,nz,nr,nc", [(24, 16, 54, 50), (25, 17, 55, 50)])  # 9216 and 10625 voxels, 24300 and 24750 rays
@pytest.mark.parametrize("batch", [1, 2, 3, 8, 13, 16])
def test_cone_operators_match_oracle(n, nz, nr, nc, batch):
    g = synth.ConeGeometry(n=n, nz=nz, px=1.0, pz=1.1, nv=9, nr=nr, nc=nc, pu=1.7, pv=1.9, sod=80.0, sdd=170.0,
                           start=0.2, off_u=0.15)
    plan, t = dect.ConePlan(g), oracle.table3(g)
    rng = np.random.default_rng(batch)
    x = rng.standard_normal((batch, nz, n, n)).astype(np.float32)
    y = rng.standard_normal((batch, g.nv, nr, nc)).astype(np.float32)
    p = dect.project_cone(plan, torch.tensor(x, device="cuda")).cpu().numpy()
    b = dect.backproject_cone(plan, torch.tensor(y, device="cuda")).cpu().numpy()
    for k in (0, batch // 2, batch - 1):
        for got, want in ((p[k], oracle.project3(t, x[k].astype(np.float64))),
                          (b[k], oracle.backproject3(t, y[k].astype(np.float64)))):
            assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)


@pytest.mark.parametrize("n,nv,nb", [(64, 60, 92), (112, 180, 162)])
@pytest.mark.parametrize("batch", [2, 7, 14])
def test_a_warp_per_row_carries_its_rounding_too(n, nv, nb, batch):
    """Small images: sums of one sign, 5e-8 as for the eight lanes (test_gpu_lanes.py)."""
    g = _geometry(n, nv, nb)
    plan, t = dect.Plan(g), oracle.table(g)
    rng = np.random.default_rng(batch)
    x = rng.uniform(0.5, 1.5, (batch, g.n, g.n)).astype(np.float32)
    y = rng.uniform(0.5, 1.5, (batch, g.nv, g.nb)).astype(np.float32)
    p = dect.project(plan, torch.tensor(x, device="cuda")).cpu().numpy()
    b = dect.backproject(plan, torch.tensor(y, device="cuda")).cpu().numpy()
    for k in range(0, batch, 3):
        for got, want in ((p[k], oracle.project(t, x[k].astype(np.float64))),
                          (b[k], oracle.backproject(t, y[k].astype(np.float64)))):
            assert np.linalg.norm(got - want) <= 5e-8 * np.linalg.norm(want)
