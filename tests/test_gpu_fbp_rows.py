"""The FBP's ramp filter bin by bin, for rows of every range (GPU), against the FP64 oracle.

One view, a central column of pixels and numbers that FP32 holds exactly put every
bin on a pixel of its own, with the interpolation weight 1: a bin far below its
row's maximum has to be as accurate as any other.  Bins at the edges of the
filter's paths (1270 the last on the tensor cores).  Tolerance per bin: 8 u,
u = 2^-24; the filtered bin, the weight pi, the product and the sum round once each.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1607_01650_gb300 as dect  # noqa: E402


def _geometry(nb):
    # ds = pitch SOD / SDD = one pixel; n odd: the central column is the line through the isocentre
    return synth.tiny_geometry(n=nb + 1 - nb % 2, nv=1, nb=nb, px=1.0, pitch=2.0, sod=4096.0, sdd=8192.0,
                               det_offset=0.0 if nb % 2 else 1.0)


def _bins(g, x):
    first = 0 if g.nb % 2 else 1
    return x[first:first + g.nb, g.n // 2]


def _rows(nb):
    rng = np.random.default_rng(nb)
    b = np.arange(nb) - 0.5 * (nb - 1)
    c = lambda at, rad: 2 * np.sqrt(np.maximum((rad * nb) ** 2 - (b - at * nb) ** 2, 0))  # noqa: E731
    ct = 0.01 * (c(0, 0.42) - 0.5 * c(0, 0.4) + 0.3 * c(0.15, 0.04)) + 1e-3 * rng.standard_normal(nb)
    rows = [ct]
    for f in (10.0, 100.0, 1e4, 1e7):  # one bin far above the rest
        rows.append(ct.copy())
        rows[-1][nb // 2 + 3] = f * np.abs(ct).max()
    rows.append(ct * 10.0 ** np.linspace(0, -12, nb))
    rows.append(1e3 * (-1.0) ** np.arange(nb) * (1 + 1e-7 * np.arange(nb)))  # the largest digit sums
    rows.append(1e3 * np.sign(rng.standard_normal(nb)) * (2 - 2.0 ** -20))
    rows.append(np.where(np.arange(nb) == 1, 1.0, 0.0))
    rows.append(np.zeros(nb))
    return np.stack(rows).astype(np.float32)


@pytest.mark.parametrize("nb", [31, 736, 737, 1151, 1152, 1153, 1269, 1270, 1271])
def test_every_bin_of_rows_of_every_range(nb):
    g = _geometry(nb)
    m = _rows(nb)
    x = dect.fbp(dect.Plan(g), torch.tensor(m[:, None], device="cuda")).cpu().numpy()
    for k in range(len(m)):
        want = np.pi * oracle.fbp_filter(g, m[k][None].astype(np.float64))[0]
        err = np.abs(_bins(g, x[k]) - want)
        assert (err <= 8 * 2.0 ** -24 * np.abs(want)).all(), (k, int((err / np.abs(want)).argmax()))


@pytest.mark.parametrize("nb", [101, 150, 172, 199, 232])
def test_rows_with_few_bins_left_to_fp64(nb):
    """64 CT-like rows with air beside the object, in four blocks of 16: a bin in a hundred is summed again."""
    g = _geometry(nb)
    rng = np.random.default_rng(nb)
    b = np.arange(nb) - 0.5 * (nb - 1)
    m = np.empty((64, nb), np.float32)
    for k in range(64):
        rad = rng.uniform(0.2, 0.45) * nb
        p = 0.02 * 2 * np.sqrt(np.maximum(rad ** 2 - (b - rng.uniform(-0.05, 0.05) * nb) ** 2, 0)) * 100 / nb
        m[k] = -np.log(np.maximum(rng.poisson(2e5 * np.exp(-p)), 1) / 2e5)
    plan, mt = dect.Plan(g), torch.tensor(m[:, None], device="cuda")
    want = np.pi * np.stack([oracle.fbp_filter(g, r[None].astype(np.float64))[0] for r in m])
    for _ in range(5):
        x = dect.fbp(plan, mt).cpu().numpy()
        got = np.stack([_bins(g, r) for r in x])
        assert (np.abs(got - want) <= 8 * 2.0 ** -24 * np.abs(want)).all()


def test_rows_share_a_block_with_rows_of_other_ranges():
    """Rows that are left to FP64 in whole, in part and not at all beside one another give what they give alone."""
    g = _geometry(300)
    m = _rows(300)
    m[2, 17] = np.inf
    m[4] *= np.float32(1e-30)
    plan = dect.Plan(g)
    x = dect.fbp(plan, torch.tensor(m[:, None], device="cuda"))
    for k in range(len(m)):
        one = dect.fbp(plan, torch.tensor(m[k][None, None], device="cuda"))[0]
        assert torch.equal(torch.nan_to_num(x[k]), torch.nan_to_num(one)), k


@pytest.mark.parametrize("n,batch", [(33, 1), (301, 2), (64 * 4 + 1, 9)])
def test_pixel_weights_are_rounded_once(n, batch):
    """The row of pixels through the isocentre sees one bin, with interpolation weight 1, at every distance from
    the source.  That bin holds a power of two: the result is (SOD / L)^2 dtheta / 2 rounded to FP32, half a unit
    in the last place off (and 2^-20 of that for the two words)."""
    g = synth.tiny_geometry(n=n, nv=1, nb=17, px=0.7, pitch=2.0, sod=333.3, sdd=666.6)
    m = np.zeros((batch, 1, 17), np.float32)
    m[:, 0, 8] = 2.0 ** np.arange(batch)
    x = dect.fbp(dect.Plan(g), torch.tensor(m, device="cuda")).cpu().numpy().astype(np.float64)
    r = g.sod / (g.sod - (np.arange(n) + 0.5 - 0.5 * n) * g.px)
    for k in range(batch):
        want = np.pi * r * r * 2.0 ** k / 4
        assert (np.abs(x[k, n // 2] - want) <= 2.0 ** -24 * (1 + 2.0 ** -20) * want).all()


@pytest.mark.parametrize("nv", [19, 20])
def test_a_block_per_parity_and_one_for_both(nv):
    """64 images of 19 views make 76 blocks of 16 rows, the most that are split by parity; of 20 views 80."""
    g = synth.tiny_geometry(n=21, nv=nv, nb=35, px=1.0, start=0.3, det_offset=0.2)
    m = np.random.default_rng(nv).standard_normal((64, nv, 35)).astype(np.float32)
    x = dect.fbp(dect.Plan(g), torch.tensor(m, device="cuda")).cpu().numpy()
    for k in range(0, 64, 9):  # tolerance of test_gpu_fbp.py
        want = oracle.fbp(g, m[k].astype(np.float64))
        assert np.linalg.norm(x[k] - want) <= 1e-5 * np.linalg.norm(want)
