"""A G on the line table inside dect_adm_tv (GPU).

Up to 8 channels the table is used wherever the plan has it, by rule: the tests say
that it was, and compare every way into it with the FP64 oracle (1e-4 relative L2,
the bound of the other ADM tests): a cold and a warm start, the projected f-step, joint
TV, and a batch that narrows onto it.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1607_01650_gb300 as dect  # noqa: E402
from test_gpu_lines import GEOMS  # noqa: E402

LINES = 3
MU, RHO, B = 16.0, 256.0, (1.0, 0.6)


def _cuda(a):
    return torch.tensor(np.asarray(a), dtype=torch.float32, device="cuda")


@pytest.mark.parametrize("name", sorted(GEOMS) + ["three"])
def test_which_plans_have_the_table(name):
    """All whose rays end outside the image, from 4 x 4 pixels on."""
    g = GEOMS[name] if name != "three" else synth.tiny_geometry(n=3, nv=7, nb=9, px=1.0)
    want = 0 if name in ("detector inside", "three") else LINES
    for ns in (1, 2, 4):
        plans = [dect.Plan(g), dect.Plan(g)]
        rng = np.random.default_rng(ns)
        m = _cuda(rng.random((ns, 2, g.nv, g.nb)))
        for plan in plans:
            dect.adm_tv(plan, m, dect.AdmParams(mu=MU, rho=RHO, max_iter=2))
            choice, us = plan.fwd_tuning(2 * ns)
            assert choice == want and us[choice] > 0, (ns, choice)


@pytest.mark.parametrize("ns,variants", [(5, {0}), (8, {0}), (16, {0}), (32, {1, 2})])
def test_wide_batches_stay_on_the_stored_rows(ns, variants):
    """One variant at 16 and 32 channels, at 64 one of two that give the same bits: A's sums do not hang on a timing."""
    g = GEOMS["63"]
    m = _cuda(np.random.default_rng(0).random((ns, 2, g.nv, g.nb)))
    width = 1 << (2 * ns - 1).bit_length()
    plan, xs = dect.Plan(g), []
    prm = dect.AdmParams(mu=MU, rho=RHO, max_iter=12)
    dect.adm_tv(plan, m, prm)
    choice, us = plan.fwd_tuning(width)
    assert choice in variants and {v for v in range(4) if us[v] > 0} == variants
    for v in sorted(variants):
        plan.set_fwd_tuning(width, v)
        xs.append(dect.adm_tv(plan, m, prm)[0])
    assert all(torch.equal(x, xs[0]) for x in xs)


@pytest.mark.parametrize("ns", [1, 2, 4])
@pytest.mark.parametrize("opts", [{}, {"nonneg": True}, {"joint": True}])
@pytest.mark.parametrize("warm", [False, True])
def test_every_way_in_matches_oracle(ns, opts, warm):
    g = synth.tiny_geometry(n=48, nv=24, nb=72, px=1.0, sod=120.0, sdd=240.0)
    slices = [synth.make_slice(g, seed=40 + i, i0=2e2) for i in range(ns)]
    m = np.stack([s.m for s in slices]).astype(np.float32)
    x0 = (0.9 * np.stack([s.truth()[1] for s in slices])).astype(np.float32)
    plan, t = dect.Plan(g), oracle.table(g)
    prm = dect.AdmParams(mu=MU, rho=RHO, max_iter=25, warm_start=warm, **opts)
    x, reps = dect.adm_tv(plan, _cuda(m), prm, x=_cuda(x0) if warm else None)
    assert plan.fwd_tuning(2 * ns)[0] == LINES
    x = x.cpu().numpy()
    for i in range(ns):
        op = oracle.AdmParams(mu=MU, rho=RHO, max_iter=25, step_rule=oracle.CAUCHY, **opts)
        xo, _ = oracle.adm_dual(t, m[i].astype(np.float64), op, x0=x0[i].astype(np.float64) if warm else None)
        for e in range(2):
            assert np.linalg.norm(x[i, e] - xo[e]) <= 1e-4 * np.linalg.norm(xo[e])
            # the carried residual is A f - beta m of the result
            assert reps[2 * i + e].resid_drift <= 1e-5 * reps[2 * i + e].primal_res


@pytest.mark.parametrize("nonneg", [False, True])
def test_narrowing_onto_the_table(nonneg):
    """16 channels on the stored rows narrow to 8, 4 and 2 on the line table.  The projected run amplifies rounding
    (a change of 6e-8 in m moves the FP64 oracle's images by up to 4e-3 within 40 iterations), so its images are
    held to their own reports: residual and objective as the oracle forms them from the image."""
    g = synth.tiny_geometry(n=48, nv=24, nb=72, px=1.0, sod=120.0, sdd=240.0)
    doses = [3e2, 1e6, 1e3, 3e5, 1e4, 3e3, 1e5, 5e2]
    m = np.stack([synth.make_slice(g, seed=500 + i, i0=d).m for i, d in enumerate(doses)]).astype(np.float32)
    plan, t = dect.Plan(g), oracle.table(g)
    prm = dect.AdmParams(mu=MU, rho=RHO, max_iter=200, rel_obj_tol=1e-4, check_every=2, nonneg=nonneg)
    x, reps = dect.adm_tv(plan, _cuda(m), prm)
    # (of the projected runs three are still going at 200 iterations: 4 channels)
    assert all(plan.fwd_tuning(w)[0] == LINES for w in ((8, 4) if nonneg else (8, 4, 2)))
    assert plan.fwd_tuning(16)[0] == 0
    x = x.cpu().numpy()
    for i in range(len(doses)):
        for e in range(2):
            r, f = reps[2 * i + e], B[e] * x[i, e].astype(np.float64)
            g64 = B[e] * m[i, e].astype(np.float64)
            assert r.resid_drift <= 1e-5 * r.primal_res
            res = np.linalg.norm(oracle.project(t, f) - g64)
            phi = oracle.objective(t, g64, MU, f)
            assert abs(r.primal_res - res) <= 1e-5 * res and abs(r.objective - phi) <= 1e-5 * phi, (i, e)
            if not nonneg:
                op = oracle.AdmParams(mu=MU, rho=RHO, max_iter=r.iters, step_rule=oracle.CAUCHY)
                fo, _, _, _ = oracle.adm_channel(t, g64, op)
                assert np.linalg.norm(f - fo) <= 1e-4 * np.linalg.norm(fo), (i, e)
            else:
                assert f.min() >= 0.0
