"""The line table (narrow batches) against the oracle and the stored CSR table (GPU).

Geometries at the edges of the form: rays outside the image, rays that enter
through the sides, rays along grid lines, 45-degree views, sizes around the
32-line and 31-pixel blocks, fine and coarse detectors (where the form does not
hold and the plan keeps to the CSR kernels).  Tolerance 1e-5 relative L2, that
of the projector tests.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1607_01650_gb300 as dect  # noqa: E402

T = synth.tiny_geometry
GEOMS = {
    "4": T(n=4, nv=7, nb=9, px=1.0),
    "31": T(n=31, nv=9, nb=45, px=0.7, start=0.1, det_offset=0.37, sod=60.0, sdd=120.0),
    "32": T(n=32, nv=16, nb=64, px=1.0, sod=100.0, sdd=200.0),
    "33 wide": T(n=33, nv=11, nb=200, px=1.0, pitch=1.1, sod=80.0, sdd=160.0),
    "62 narrow": T(n=62, nv=10, nb=33, px=1.0, pitch=1.2, sod=200.0, sdd=400.0),
    "63": T(n=63, nv=13, nb=95, px=0.5, start=-0.3, det_offset=-2.0, sod=100.0, sdd=150.0),
    "aligned": T(n=64, nv=8, nb=65, px=1.0, pitch=2.0, sod=400.0, sdd=800.0),
    "45 degrees": T(n=40, nv=8, nb=61, px=1.0, start=np.pi / 4, sod=1e5, sdd=2e5, pitch=2.0),
    "fine": T(n=20, nv=6, nb=400, px=1.0, sod=60.0, sdd=120.0),
    "coarse": T(n=40, nv=6, nb=5, px=1.0, sod=120.0, sdd=240.0),
    "detector inside": T(n=24, nv=7, nb=30, px=1.0, sod=40.0, sdd=44.0, pitch=1.0),
    "short arc": T(n=45, nv=5, nb=70, px=1.0, sod=90.0, sdd=180.0, arc=0.7),
}


@pytest.mark.parametrize("name", sorted(GEOMS))
@pytest.mark.parametrize("batch", [1, 3, 4, 7, 16])
def test_operators_match_oracle(name, batch):
    g = GEOMS[name]
    plan, t = dect.Plan(g), oracle.table(g)
    rng = np.random.default_rng(batch)
    x = rng.standard_normal((batch, g.n, g.n)).astype(np.float32)
    y = rng.standard_normal((batch, g.nv, g.nb)).astype(np.float32)
    p = dect.project(plan, torch.tensor(x, device="cuda")).cpu().numpy()
    b = dect.backproject(plan, torch.tensor(y, device="cuda")).cpu().numpy()
    for k in range(batch):
        for got, want in ((p[k], oracle.project(t, x[k].astype(np.float64))),
                          (b[k], oracle.backproject(t, y[k].astype(np.float64)))):
            assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)


@pytest.mark.parametrize("batch", [17, 64, 65, 80])
def test_passes_of_both_forms(batch):
    """A wide pass on the CSR table and a narrow rest on the line table."""
    g = GEOMS["33 wide"]
    plan = dect.Plan(g)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(batch)
    x = torch.randn((batch, g.n, g.n), generator=gen, device="cuda")
    y = torch.randn((batch, g.nv, g.nb), generator=gen, device="cuda")
    p, b = dect.project(plan, x), dect.backproject(plan, y)
    for k in range(batch):
        for got, one in ((p[k], dect.project(plan, x[k])), (b[k], dect.backproject(plan, y[k]))):
            assert (got - one).norm() <= 1e-5 * one.norm()


@pytest.mark.parametrize("name", ["31", "33 wide", "aligned", "45 degrees"])
def test_values_that_are_not_finite_reach_only_their_rays_and_pixels(name):
    g = GEOMS[name]
    plan = dect.Plan(g)
    ptr, pix, ln = plan.table()
    ray = np.repeat(np.arange(g.nv * g.nb), np.diff(ptr))
    solid = ln > 1e-6 * g.px  # (a corner met within rounding may or may not count as touched)
    rng = np.random.default_rng(1)

    def check(out, touched, size):
        may, must = np.zeros(size, bool), np.zeros(size, bool)
        may[touched], must[touched[solid[sel]]] = True, True
        bad = ~np.isfinite(out.ravel())
        assert must.any() and not (bad & ~may).any() and not (must & ~bad).any()

    x = rng.random((2, g.n, g.n)).astype(np.float32)
    for value, at in ((np.nan, g.n * (g.n // 2) + g.n // 3), (np.inf, g.n * (g.n // 2) + 1)):
        x[1].flat[at] = value
        p = dect.project(plan, torch.tensor(x, device="cuda")).cpu().numpy()
        x[1].flat[at] = 0.5
        assert np.isfinite(p[0]).all()
        sel = pix == at
        check(p[1], ray[sel], g.nv * g.nb)
    y = rng.random((2, g.nv, g.nb)).astype(np.float32)
    r = int(ray[len(ray) // 3])
    y[0].flat[r] = np.nan
    b = dect.backproject(plan, torch.tensor(y, device="cuda")).cpu().numpy()
    sel = ray == r
    check(b[0], pix[sel], g.n * g.n)
    assert np.isfinite(b[1]).all()
