"""dect_kernel_launches counts what dect_adm_tv launches, graph replays included (GPU)."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1607_01650_gb300 as dect  # noqa: E402

LINES = 3  # the A variant on the line table


@pytest.mark.parametrize("choice", [0, LINES])
@pytest.mark.parametrize("nonneg", [False, True])
def test_kernel_count_per_iteration(choice, nonneg):
    """TV step, A^T and A; a projected step forms A f anew, on the line table after a transpose of f."""
    g = synth.tiny_geometry(n=48, nv=24, nb=72, px=1.0, sod=120.0, sdd=240.0)
    plan = dect.Plan(g)
    m = torch.tensor(np.random.default_rng(0).random((1, 2, g.nv, g.nb)), dtype=torch.float32, device="cuda")
    plan.set_fwd_tuning(2, choice)

    def launches(iters):
        before = dect.kernel_launches()
        dect.adm_tv(plan, m, dect.AdmParams(mu=16.0, rho=256.0, max_iter=iters, nonneg=nonneg))
        return dect.kernel_launches() - before

    launches(20)
    per = 3 + (0 if not nonneg else 2 if choice == LINES else 1)
    assert launches(50) - launches(20) == 30 * per
    assert launches(23) - launches(20) == 3 * per
