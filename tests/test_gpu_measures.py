"""compare and density_stats where their fast paths can go wrong: values beside each other, at the ends of the
exponent range, on bin edges and shell radii, and fields of odd length.  Counts have to be the same; the divergence
is a sum of terms a log(a / b), each within 2^-48 of its size (the quotient's own rounding is 2^-53 of a).
"""
import numpy as np
import pytest

from oracle import evaluation as ev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_0906_3978_gb300 as wf  # noqa: E402

DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    wf.build()
    c = wf.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("cells", [1, 31, 257, 100003])
@pytest.mark.parametrize("kind", ["close", "wide", "signs", "extreme"])
def test_divergence(ctx, cells, kind):
    rng = np.random.default_rng(cells)
    a = np.exp(rng.normal(0.0, 1.0, cells))
    b = np.exp(rng.normal(0.0, 1.0, cells))
    if kind == "close":
        b = a * (1.0 + rng.normal(0.0, 1.0, cells) * 10.0 ** rng.uniform(-16.0, -1.0, cells))
    elif kind == "wide":
        b = np.exp(rng.uniform(-30.0, 30.0, cells))
    elif kind == "signs":
        a[::3] *= -1.0
        b[::2] = 0.0
    else:
        a[::2] = 10.0 ** rng.uniform(100.0, 200.0, a[::2].size)
    rec, tru = a - 1.0, b - 1.0
    got = ctx.compare(torch.from_numpy(rec).to(DEV), torch.from_numpy(tru).to(DEV))
    x, y = (1.0 + rec).astype(np.longdouble), (1.0 + tru).astype(np.longdouble)
    ok = (x > 0) & (y > 0)
    assert got["kl_excluded"] == cells - int(np.count_nonzero(ok))
    q = np.log(x[ok] / y[ok])
    size = float(np.sum(x[ok] * (1.0 + np.abs(q)))) / cells
    assert abs(got["d_kl"] - float(np.sum(x[ok] * q)) / cells) <= size * 2.0 ** -48


@pytest.mark.parametrize("n", [16, 72, 108])
@pytest.mark.parametrize("lo,width", [(0.0, 0.25), (-0.3, 0.1), (0.7, 1e-3), (0.0, 1e-12)])
def test_bins_and_shells(ctx, n, lo, width):
    rng = np.random.default_rng(n)
    nb, box = 20, 1.0 * n
    k = rng.integers(-3, nb + 4, (n, n, n))
    delta = (lo + k * width) - 1.0                                    # on the edges, as they round
    delta += np.where(rng.random((n, n, n)) < 0.5, 0.0, np.spacing(delta) * rng.integers(-2, 3, (n, n, n)))
    delta.ravel()[:4] = [np.inf, -np.inf, 1e300, -1e300]
    w = np.where(rng.random((n, n, n)) < 0.5, 0.0, 1.0)
    obs = (0.0, 3.0, 4.0)
    shells = [[0.0, 5.0], [5.0, 13.0], [3.0, 3.0], [0.0, np.inf], [-1.0, 0.0], [np.sqrt(2.0), np.sqrt(50.0)]]
    hist, _ = ctx.density_stats(torch.from_numpy(delta).to(DEV), torch.from_numpy(w).to(DEV), box, obs, shells, lo,
                                width, nb)
    ref, under, over = ev.density_hist(delta, w, box, obs, shells, lo, width, nb)
    assert np.array_equal(hist[:, :, :nb], ref)
    assert np.array_equal(hist[:, :, nb], under) and np.array_equal(hist[:, :, nb + 1], over)
