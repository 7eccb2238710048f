"""The FBP's kernels at the edges of their paths (GPU), against the FP64 oracle.

The ramp filter runs on the tensor cores with exact digits up to about 1170
bins and in FP64 beyond, and for rows whose values are not finite or leave the
digits' range; the back-projection runs at widths of 1, 2, 4, ... 64 images.
Tolerance: 1e-5 relative L2, the projection tolerance (FP32 interpolation and
sums), as in test_gpu_fbp.py.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1607_01650_gb300 as dect  # noqa: E402


def _sinograms(g, batch, seed=0):
    S, D = synth.ray_endpoints(g)
    rng = np.random.default_rng(seed)
    half = 0.5 * g.n * g.px
    out = []
    for b in range(batch):
        e = synth.Ellipse(0.1 * half * np.cos(b), 0.1 * half, 0.5 * half, 0.3 * half, 0.2 * b, 1.0, 0.0)
        out.append(synth.ellipse_chords([e], S, D, [0.02]) + 1e-3 * rng.standard_normal((g.nv, g.nb)))
    return np.stack(out).astype(np.float32)


def _check(g, m, plan=None):
    x = dect.fbp(plan or dect.Plan(g), torch.tensor(m, device="cuda")).cpu().numpy()
    for b in range(len(m)):
        want = oracle.fbp(g, m[b].astype(np.float64))
        assert np.linalg.norm(x[b] - want) <= 1e-5 * np.linalg.norm(want), b
    return x


@pytest.mark.parametrize("batch", [2, 3, 8, 9, 17, 33, 64, 67])
def test_every_width(batch):
    g = synth.tiny_geometry(n=21, nv=11, nb=35, px=1.0, start=0.3, det_offset=0.2)
    _check(g, _sinograms(g, batch))


@pytest.mark.parametrize("nb", [2, 3, 15, 16, 17, 31, 33, 46, 300, 737, 1170, 1300])
def test_every_filter_shape(nb):
    g = synth.tiny_geometry(n=24, nv=5, nb=nb, px=1.0)
    _check(g, _sinograms(g, 2))


def test_rows_outside_the_digits_range():
    g = synth.tiny_geometry(n=24, nv=9, nb=70, px=1.0)
    m = _sinograms(g, 5)
    m[1] *= np.float32(1e-25)
    m[2] *= np.float32(1e25)
    m[3, 4] = 0.0
    m[4, :, 1::2] *= np.float32(1e-6)
    _check(g, m)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_a_value_that_is_not_finite(bad):
    g = synth.tiny_geometry(n=24, nv=9, nb=70, px=1.0)
    m = _sinograms(g, 3)
    clean = _check(g, m)
    m[1, 4, 30] = bad
    x = dect.fbp(dect.Plan(g), torch.tensor(m, device="cuda")).cpu().numpy()
    want = oracle.fbp(g, m[1].astype(np.float64))
    np.testing.assert_array_equal(x[[0, 2]], clean[[0, 2]])
    np.testing.assert_array_equal(np.isfinite(x[1]), np.isfinite(want))
