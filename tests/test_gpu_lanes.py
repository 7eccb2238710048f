"""Rows of eight lanes (cone-beam A and A^T of narrow batches) against the oracle (GPU).

Sizes around the 8 x 16 pixel tiles of A^T and the rows of one block, at every
batch width the kernels are built for.  Tolerance 1e-5 relative L2, that of the
projector tests.  The sums of A and A^T of narrow fan-beam batches carry their
rounding errors along: what remains is the rounding of the result (2^-23 / sqrt(12)
of its power of two, at most 3.5e-8) and of the 200 to 400 entries' lengths and
partial sums, less than as much again: 5e-8 together, rms.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1607_01650_gb300 as dect  # noqa: E402


@pytest.mark.parametrize("n,nz,nr,nc", [(7, 2, 3, 11), (16, 1, 1, 33), (17, 3, 4, 29)])
@pytest.mark.parametrize("batch", [1, 2, 4, 5, 8, 15, 16, 17])
def test_cone_operators_match_oracle(n, nz, nr, nc, batch):
    g = synth.ConeGeometry(n=n, nz=nz, px=1.0, pz=1.3, nv=9, nr=nr, nc=nc, pu=1.3, pv=1.7, sod=60.0,
                           sdd=130.0, start=0.2, off_u=0.15)
    plan, t = dect.ConePlan(g), oracle.table3(g)
    rng = np.random.default_rng(batch)
    x = rng.standard_normal((batch, nz, n, n)).astype(np.float32)
    y = rng.standard_normal((batch, g.nv, nr, nc)).astype(np.float32)
    p = dect.project_cone(plan, torch.tensor(x, device="cuda")).cpu().numpy()
    b = dect.backproject_cone(plan, torch.tensor(y, device="cuda")).cpu().numpy()
    for k in range(batch):
        for got, want in ((p[k], oracle.project3(t, x[k].astype(np.float64))),
                          (b[k], oracle.backproject3(t, y[k].astype(np.float64)))):
            assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)


@pytest.mark.parametrize("batch", [1, 7, 14])
def test_narrow_sums_carry_their_rounding(batch):
    g = synth.tiny_geometry(n=256, nv=120, nb=370, px=1.0, sod=700.0, sdd=1400.0)
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


def test_infinite_pixel_keeps_its_sign():
    g = synth.tiny_geometry(n=48, nv=20, nb=70, px=1.0, sod=100.0, sdd=200.0)
    plan = dect.Plan(g)
    x = torch.ones((1, 48, 48), device="cuda")
    clean = dect.project(plan, x)
    x[0, 20, 27] = float("-inf")
    y = dect.project(plan, x)
    hit = y != clean
    assert hit.any() and bool((y[hit] == float("-inf")).all())
    r = clean.clone()
    r[0, 3, 35] = float("inf")
    b = dect.backproject(plan, r)
    assert not torch.isnan(b).any() and bool((b == float("inf")).any())


@pytest.mark.parametrize("n,ns", [(33, 7), (52, 8)])
def test_eight_lane_backprojector_of_sixteen_channels(n, ns):
    g = synth.tiny_geometry(n=n, nv=24, nb=80, px=1.0, sod=130.0, sdd=260.0)
    m = np.stack([synth.make_slice(g, seed=400 + i, i0=1e5).m for i in range(ns)]).astype(np.float32)
    plan, t = dect.Plan(g), oracle.table(g)
    plan.set_tuning(16, 3)
    x, _ = dect.adm_tv(plan, torch.tensor(m, device="cuda"), dect.AdmParams(mu=4.0, rho=256.0, max_iter=12))
    for i in (0, ns - 1):
        op = oracle.AdmParams(mu=4.0, rho=256.0, max_iter=12, step_rule=oracle.CAUCHY)
        xo, _ = oracle.adm_dual(t, m[i].astype(np.float64), op)
        for e in range(2):  # the bound of the other variants' test
            assert np.linalg.norm(x[i, e].cpu().numpy() - xo[e]) <= 1e-4 * np.linalg.norm(xo[e])
