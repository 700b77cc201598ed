"""The window's screened decisions against the plain definition, node by node: cones and holes whose boundary
passes exactly through grid nodes, observers on and far from the grid, every radial law.

numpy's FP64 +, *, sqrt are the definition's operations one by one, so membership has to be the same; a value is
exp(x), whose argument carries a few roundings: |x| + 8 times 4 x 2^-53 bounds its relative difference.
"""
import math

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_0906_3978_gb300 as wf  # noqa: E402

DEV = "cuda:0"
DIAG = tuple(np.array([1.0, 1.0, 0.0]) / math.sqrt(2.0))


@pytest.fixture(scope="module")
def ctx():
    wf.build()
    c = wf.Context(0)
    yield c
    c.close()


def definition(sel, n, box):
    h = box / n
    d = [np.arange(n) * h - o for o in sel.observer]
    dx, dy, dz = d[0][:, None, None], d[1][None, :, None], d[2][None, None, :]
    r = np.sqrt((dx * dx + dy * dy) + dz * dz)
    dot = lambda v: (dx * v[0] + dy * v[1]) + dz * v[2]  # noqa: E731
    inside = (r > 0.0) & (dot(sel.axis) >= math.cos(sel.half_angle) * r)
    for hole in sel.holes:
        inside &= ~(dot(hole) > math.cos(hole[3]) * r)
    with np.errstate(divide="ignore", invalid="ignore"):
        t = r / sel.radial_params[0] if sel.radial_kind else r
        x = {0: 0.0 * r, 1: -(t * t), 2: sel.radial_params[1] * (np.log(t) + (1.0 - t))}[sel.radial_kind]
    return inside, np.where(inside, x, 0.0)


@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("n", [16, 108, 128])
@pytest.mark.parametrize("axis,half,observer", [
    ((1.0, 0.0, 0.0), math.pi / 4, (0.0, 8.0, 8.0)),          # faces of the cone through nodes
    (DIAG, math.pi / 4, (2.0, 2.0, 2.0)), ((0.0, 0.0, 1.0), math.pi / 2, (8.0, 8.0, 8.0)),
    ((0.0, 1.0, 0.0), math.pi, (5.0, 6.0, 7.0)), (DIAG, 0.0, (0.0, 0.0, 0.0)),
    ((1.0, 0.0, 0.0), 0.3, (-4.0e13, 8.0, 8.0)), (DIAG, 0.7, (8.0 + 1e-13, 8.0, 8.0))])
def test_membership_and_values(ctx, n, kind, axis, half, observer):
    box = 1.0 * n
    holes = np.array([[0.0, 1.0, 0.0, math.pi / 4], [1.0, 0.0, 0.0, 0.1], [DIAG[0], DIAG[1], 0.0, 0.0]])
    sel = synth.Selection(observer=observer, axis=axis, half_angle=half, holes=holes, radial_kind=kind,
                          radial_params=(0.3 * n, 2.5, 0.0, 0.0))
    n_obs = torch.ones((n, n, n), dtype=torch.float64, device=DEV)
    _, w, _, _, _ = ctx.build_noise(sel, n_obs, 1000, box, check=False)  # (an empty window is an error, w is made)
    w = w.cpu().numpy()
    inside, x = definition(sel, n, box)
    ref = np.where(inside, np.exp(x), 0.0)
    assert np.array_equal((w != 0.0)[ref > 1e-300], inside[ref > 1e-300]) and not w[~inside].any()
    ok = ref > 1e-300
    assert np.all(np.abs(w[ok] / ref[ok] - 1.0) <= (np.abs(x[ok]) + 8.0) * 4.0 * 2.0 ** -53)
