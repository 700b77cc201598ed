"""The mask projection's ray ranges and runs: observers inside, on the faces and outside of the box (rays that enter
late, leave early, graze or miss it), radial tables of any length, steps from a tenth of a cell to several cells.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_0906_3978_gb300 as wf  # noqa: E402
from test_gpu_evaluation import _fp32_face_margin  # noqa: E402

DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    wf.build()
    c = wf.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n", [16, 24, 72])
@pytest.mark.parametrize("observer", [(0.5, 0.5, 0.5), (0.0, 0.0, 0.0), (1.0, 0.5, 0.0), (-0.7, 0.4, 0.3), (1.5, 1.5, 1.5),
                                      (0.5, 0.5, 9.0)])
@pytest.mark.parametrize("n_r,step", [(1, 0.4), (31, 0.1), (33, 3.0), (257, 0.7)])
def test_ranges_and_runs(ctx, n, observer, n_r, step):
    rng = np.random.default_rng(n + n_r)
    box = 2.5 * n
    n_alpha, n_delta = 37, 19
    sky = rng.random((n_delta, n_alpha))
    wr = rng.random(n_r)
    obs = tuple(v * box for v in observer)
    geo = (0.0, 2 * np.pi / n_alpha, -np.pi / 2, np.pi / n_delta)
    dr = step * box / n
    w, cnt = ctx.project_mask(torch.from_numpy(sky).to(DEV), n, box, *geo, obs, dr, wr, want_counts=True)
    w_ref, c_ref, near = oracle.project_mask(sky, n, box, *geo, obs, dr, wr,
                                             face_margin=_fp32_face_margin(n, box, obs))
    w, cnt = w.cpu().numpy(), cnt.cpu().numpy()
    assert np.all(np.abs(cnt - c_ref) <= near)          # samples within the FP32 error of a face may move
    far = near == 0
    assert np.array_equal(cnt[far], c_ref[far])
    assert np.all(np.abs(w[far] - w_ref[far]) <= 1e-15 * np.abs(w_ref[far]))  # the finish's roundings
