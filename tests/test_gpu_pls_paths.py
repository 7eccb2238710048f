"""The decomposition's kernels at the edges of their paths (GPU).

The direct solve is formed in two FP32 words with an FP64 fallback near
rounding boundaries: its result is the FP64 value rounded once, so it must
equal numpy's bit for bit.  The CG takes four pixels of a row per thread where
n % 4 == 0 and u is 16-byte aligned, one otherwise; both against the oracle at
the parity tolerance (2e-4 relative L2).
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1607_01650_gb300 as dect  # noqa: E402


@pytest.mark.parametrize("n,batch", [(1, 1), (17, 2), (127, 1), (129, 3), (256, 2)])
@pytest.mark.parametrize("eta", [((0.0184, 0.0227), (0.0342, 0.0573)), ((-3.0, 1e3), (2e-9, 0.7)),
                                 ((1e30, 1.0), (1.0, 1e-28)), ((1.0, 0.0), (0.0, 1.0))])
def test_direct_solve_is_the_fp64_value_rounded_once(n, batch, eta):
    rng = np.random.default_rng(n + batch)
    x = (0.02 * rng.standard_normal((batch, 2, n, n))).astype(np.float32)
    x *= np.exp2(rng.integers(-30, 30, x.shape)).astype(np.float32) * (rng.random(x.shape) < 0.9)
    if n > 64:
        x[0, 0, 3, :6] = [np.inf, -np.inf, np.nan, 1e-42, -0.0, 3e38]
    u, _ = dect.pls_decompose(torch.tensor(x, device="cuda"), dect.PlsParams(eta=eta, gamma=0.0, max_iter=0))
    (a, c), (b, e) = eta
    with np.errstate(all="ignore"):
        h, lo, det = x[:, 0].astype(np.float64), x[:, 1].astype(np.float64), a * e - b * c
        want = np.stack([(e * h - b * lo) / det, (-c * h + a * lo) / det], 1).astype(np.float32)
    np.testing.assert_array_equal(u.cpu().numpy(), want)


def _mixture(n, seed):
    g = synth.tiny_geometry(n=n, px=1.0, sod=10.0 * n, sdd=20.0 * n)
    u = synth.rasterize(synth.random_ellipse_phantom(g, seed=seed, axis_range=(0.1 * n, 0.3 * n)), n, 1.0, 4)
    rng = np.random.default_rng(seed)
    return np.stack([synth.attenuation(u, k) + s * rng.standard_normal((n, n))
                     for k, s in ((0, 4e-4), (1, 6e-4))]).astype(np.float32)


@pytest.mark.parametrize("n", [2, 3, 5, 64, 66, 132])
@pytest.mark.parametrize("K,tol,gamma", [(7, 0.0, 0.1), (40, 1e-6, 3.0)])
def test_iterations_stops_and_an_empty_slice(n, K, tol, gamma):
    """Slices that stop at once (all zero) or late share the launches; more
    iterations than the first burst holds; u on a 4-byte boundary."""
    x = np.stack([_mixture(max(n, 8), 3)[:, :n, :n], np.zeros((2, n, n), np.float32), _mixture(max(n, 8), 9)[:, :n, :n]])
    prm = dect.PlsParams(gamma=gamma, max_iter=K, tol=tol)
    xd = torch.tensor(x, device="cuda")
    u, reps = dect.pls_decompose(xd, prm)
    buf = torch.zeros(x.size + 1, device="cuda")
    v, reps_v = dect.pls_decompose(xd, prm, u=buf[1:].view(x.shape))
    u, v = u.cpu().numpy(), v.cpu().numpy()
    assert not u[1].any() and reps[1][0] == (0, 0)
    op = oracle.PlsParams(gamma=gamma, max_iter=K if tol == 0 else 500, tol=0.0 if tol == 0 else 1e-10)
    for b in (0, 2):
        want = oracle.pls_decompose(x[b, 0].astype(np.float64), x[b, 1].astype(np.float64), op)[:2]
        for m in range(2):
            for got in (u, v):
                assert np.linalg.norm(got[b, m] - want[m]) <= 2e-4 * np.linalg.norm(want[m])
        assert reps[b][0] == reps_v[b][0]
        assert reps[b][0] == (K, K) if tol == 0 else max(reps[b][1]) < tol
