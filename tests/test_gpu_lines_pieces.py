"""The line table piece by piece (GPU): A of single pixels against the stored CSR table.

A ray's piece in a pixel has to be as accurate however short it is.  Both tables
come from the same walk in FP64; the CSR one rounds a length once (2^-24), the
line table rounds the fraction and its complement, the two words of the line's
length times it once more: 4 u, u = 2^-24, between them.  Pieces below 1e-9 of a
pixel are left to the walk's rounding.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1607_01650_gb300 as dect  # noqa: E402

T = synth.tiny_geometry
GEOMS = {
    "4": T(n=4, nv=301, nb=9, px=1.0),
    "33 wide": T(n=33, nv=211, nb=200, px=1.0, pitch=1.1, sod=80.0, sdd=160.0),
    "63": T(n=63, nv=113, nb=95, px=0.5, start=-0.3, det_offset=-2.0, sod=100.0, sdd=150.0),
    "96": T(n=96, nv=181, nb=140, px=1.0, start=0.01, sod=300.0, sdd=600.0),
}


@pytest.mark.parametrize("name", sorted(GEOMS))
@pytest.mark.parametrize("batch", [2, 4, 8, 16])
def test_pieces_of_every_size(name, batch):
    g = GEOMS[name]
    plan = dect.Plan(g)
    ptr, pix, ln = plan.table()
    ray = np.repeat(np.arange(g.nv * g.nb), np.diff(ptr))
    n, rng = g.n, np.random.default_rng(batch)
    # the corners, the middles of the sides, and pixels inside
    at = [0, n - 1, n * (n - 1), n * n - 1, n // 2, n * (n // 2), n * (n // 2) + n - 1, n * (n - 1) + n // 2]
    at = (at + rng.choice(n * n, 8).tolist())[:batch] if batch != 2 else [0, n * n - 1]
    x = np.zeros((batch, n * n), np.float32)
    x[np.arange(batch), at] = 1.0
    y = dect.project(plan, torch.tensor(x.reshape(batch, n, n), device="cuda")).cpu().numpy().reshape(batch, -1)
    short = 0
    for k in range(batch):
        sel = pix == at[k]
        want = np.zeros(g.nv * g.nb)
        np.add.at(want, ray[sel], ln[sel].astype(np.float64))
        err = np.abs(y[k] - want)
        assert (err <= 4 * 2.0 ** -24 * want + 1e-9 * g.px * (want <= 1e-9 * g.px)).all(), at[k]
        short += int(((want > 0) & (want < 1e-2 * g.px)).sum())
    assert short > 0 or name == "4"
