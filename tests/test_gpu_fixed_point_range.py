"""The fixed-point transforms at the ends of the FP64 range, and Fourier tables of many decades.

A power of two passes through a linear filter exactly, so a scaled field is held to the scaled result: 1e-13 of it (the
transforms leave 2e-16), two units of 2^-1074 where the values are subnormal (the last rounding is half of one).
"""
import numpy as np
import pytest

import oracle
import synth

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


def field(n, seed=1):
    return torch.from_numpy(np.random.default_rng(seed).standard_normal((n, n, n))).to(DEV)


def times(f, e):
    """f 2^e, the factor in two steps (either may not be a double's)."""
    return f * 2.0 ** (e // 2) * 2.0 ** (e - e // 2)


@pytest.mark.parametrize("e", [-1005, -960, -860, -700, 700, 960])
@pytest.mark.parametrize("n", [16, 108, 192])
def test_scaled_field(ctx, n, e):
    f = field(n)
    for g in (lambda x: ctx.smooth(x, 2.0 * n, 3.0), lambda x: ctx.deconvolve(x, 2.0 * n, 0.42, 5.0, 1.2)):
        ref, got = g(f), times(g(times(f, e)), -e)
        assert float(torch.linalg.norm(got - ref)) <= 1e-13 * float(torch.linalg.norm(ref))


def test_subnormal_field(ctx):
    n = 32
    f = times(field(n), -1060)
    ref = ctx.smooth(times(f, 1000), 2.0 * n, 3.0)
    assert float(times(times(ctx.smooth(f, 2.0 * n, 3.0), 1000) - ref, 0).abs().max()) <= 2.0 * 2.0 ** -74


def test_products_past_the_range(ctx):
    n = 24
    f = field(n)
    assert not ctx.deconvolve(times(f, -790), 2.0 * n, 0.42, 5.0, 1e120).any()
    assert not torch.isfinite(ctx.deconvolve(times(f, 600), 2.0 * n, 0.42, 5.0, 2.0 ** -600)).any()


def test_table_with_nan_gives_nan(ctx):
    f = field(16)
    assert torch.isnan(ctx.smooth(f, 1e-160, 1.0)).all()  # the exponent's k^2 is infinite, times 0 at k = 0
    assert torch.isnan(ctx.smooth(f, 1e-160, 0.0)).all()


@pytest.mark.parametrize("n", [16, 24, 32, 48, 64, 72, 96, 108, 128, 144, 192, 216, 256])
def test_deconvolve_every_size(ctx, n):
    """Against torch's FP64 transforms with the table of <K D>: 1e-13 (their own error is some 1e-16 log2 n^3)."""
    f, box, beta, sv, bias = field(n), 2.0 * n, 0.42, 5.0, 1.2
    k = 2.0 * np.pi / box * np.sqrt(np.arange(3 * (n // 2) ** 2 + 1))
    mu, wt = np.polynomial.legendre.leggauss(128)
    mu, wt = 0.5 * (mu + 1.0), 0.5 * wt
    kd = ((1 + beta * mu ** 2) ** 2 / (1 + 0.5 * (k[:, None] * sv * mu) ** 2) * wt).sum(axis=1)
    i = torch.arange(n, device=DEV)
    i = torch.where(i > n // 2, i - n, i)
    z = torch.arange(n // 2 + 1, device=DEV)
    n2 = (i * i)[:, None, None] + (i * i)[None, :, None] + (z * z)[None, None, :]
    t = torch.from_numpy(1.0 / (bias * np.sqrt(kd))).to(DEV)[n2]
    ref = torch.fft.irfftn(torch.fft.rfftn(f) * t, s=(n, n, n))
    got = ctx.deconvolve(f, box, beta, sv, bias)
    assert float(torch.linalg.norm(got - ref)) <= 1e-13 * float(torch.linalg.norm(ref))


@pytest.mark.parametrize("prec", [wf.FP64, wf.MIXED])
@pytest.mark.parametrize("n", [32, 96])
def test_prior_of_eight_decades(ctx, n, prec):
    """One exponent serves the prior's table: the solver's residual is the oracle's, to 1e-12 beside tol = 1e-9."""
    box = 4.0 * n
    sel = synth.selection_sdss_like(box, 5)
    w = oracle.window(sel, n, box)
    nbar = 0.05 * n ** 3 / w.sum()
    b = np.where(w > 0, np.random.default_rng(7).poisson(nbar * w) - nbar * w, 0.0)
    kf = 2.0 * np.pi / box
    pk = np.geomspace(0.5 * kf, 1.8 * kf * n, 64)
    pp = 1e4 * (pk / pk[0]) ** (-8.0 / np.log10(pk[-1] / pk[0]))
    s, _ = ctx.solve(torch.from_numpy(w).to(DEV), nbar, torch.from_numpy(b).to(DEV), box, pk, pp, tol=1e-9,
                     max_iter=20000, prec=prec)
    r = b - oracle.matvec(oracle.sinv_table(n, box, pk, pp), nbar, w, s.cpu().numpy())
    assert np.linalg.norm(r) <= (1e-9 + 1e-12) * np.linalg.norm(b)
