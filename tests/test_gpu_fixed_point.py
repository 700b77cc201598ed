"""The fixed-point transforms (64-bit integers in place of FP64 butterflies) against FP64 FFTs.

Tolerance: an FP64 transform of V points leaves about log2(V) rounding errors of 2^-53 on the rms of its
output, the fixed-point one less; the relative L2 difference is bounded by four times that.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_0906_3978_gb300 as wf  # noqa: E402

SIZES = [16, 24, 32, 48, 64, 72, 96, 108, 128, 144, 192, 216, 256, 288, 384, 512]
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    wf.build()
    c = wf.Context(0)
    yield c
    c.close()


def tol(points):
    return 4.0 * math.log2(points) * 2.0 ** -53


def rl2(a, r):
    return float(torch.linalg.norm(a - r) / torch.linalg.norm(r))


def lowpass(fine, n, unit):
    """The definition: every |k_i| < n/2 of the fine spectrum, sampled at n^3."""
    h, nf = n // 2, 2 * n
    spec = torch.fft.rfftn(fine.reshape(nf, nf, nf).to(torch.float64) * unit)
    out = torch.zeros((n, n, h + 1), dtype=torch.complex128, device=DEV)
    lo, hi = (slice(0, h), slice(0, h)), (slice(h + 1, n), slice(nf - h + 1, nf))
    for a, sa in (lo, hi):
        for b, sb in (lo, hi):
            out[a, b, :h] = spec[sa, sb, :h]
    return torch.fft.irfftn(out, s=(n, n, n))


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("kind", ["one", "crowd"])
def test_lowpass_every_size(ctx, n, kind):
    """One galaxy alone (most lines hold a single spike), and single galaxies beside 40000 in one cell
    (lines whose values differ by 4e4)."""
    rng = np.random.default_rng(n)
    box = 1.7 * n
    pos = rng.random((1 if kind == "one" else 200, 3)) * box
    if kind == "crowd":
        pos = np.concatenate([pos, np.full((40000, 3), 0.37 * box)])
    fine = torch.empty((2 * n) ** 3, dtype=torch.int64, device=DEV)
    got = ctx.grid_assign(torch.from_numpy(pos).to(DEV), n, box, wf.TSC, 2, fine_out=fine)
    assert rl2(got, lowpass(fine, n, 2.0 ** -48)) <= tol((2 * n) ** 3)


@pytest.mark.parametrize("n", [16, 72, 144])
def test_weighted_lowpass_over_the_mass_range(ctx, n):
    """Masses over nine decades up to 2^30 (Q32 units near 2^62)."""
    rng = np.random.default_rng(n + 1)
    box = 1.7 * n
    pos = rng.random((300, 3)) * box
    mass = 10.0 ** rng.uniform(0.0, 9.0, 300)
    fine = torch.empty((2 * n) ** 3, dtype=torch.int64, device=DEV)
    got = ctx.grid_assign_weighted(torch.from_numpy(pos).to(DEV), torch.from_numpy(mass).to(DEV), n, box, wf.TSC, 2,
                                   fine_out=fine)
    assert rl2(got, lowpass(fine, n, 2.0 ** -32)) <= tol((2 * n) ** 3)


def smoothed(f, n, box, r_s):
    m = torch.arange(n, device=DEV)
    m = torch.where(m > n // 2, m - n, m).to(torch.float64)
    z = torch.arange(n // 2 + 1, device=DEV, dtype=torch.float64)
    n2 = (m * m)[:, None, None] + (m * m)[None, :, None] + (z * z)[None, None, :]
    k2 = (2.0 * math.pi / box) ** 2 * n2
    return torch.fft.irfftn(torch.fft.rfftn(f) * torch.exp(-0.5 * k2 * r_s * r_s), s=(n, n, n))


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("kind", ["white", "spike", "tiny", "huge"])
def test_fourier_passes_every_size(ctx, n, kind):
    """The FP64 z, y and x passes (forward, multiplier, inverse): white noise, one value 1e9 above it, and
    fields near the ends of the exponent range."""
    g = torch.Generator(device=DEV)
    g.manual_seed(n)
    f = torch.randn((n, n, n), dtype=torch.float64, device=DEV, generator=g)
    if kind == "spike":
        f[n // 3, n // 2, 1] = 1e9
    scale = {"tiny": 1e-230, "huge": 1e290}.get(kind, 1.0)
    got = ctx.smooth(f * scale, 1.0 * n, 0.6) / scale
    assert rl2(got, smoothed(f, n, 1.0 * n, 0.6)) <= tol(n ** 3)


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_non_finite_fields_stay_non_finite(ctx, value):
    """Every value of the result depends on every value of the field."""
    f = torch.zeros((24, 24, 24), dtype=torch.float64, device=DEV)
    f[3, 4, 5] = value
    assert not bool(torch.isfinite(ctx.smooth(f, 24.0, 1.0)).any())
