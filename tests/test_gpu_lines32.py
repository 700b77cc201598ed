"""The FP32 CG passes on the line engine at every grid size: rows, tiles and radix plans differ for each.

The first iterates of the mixed solve are held to the FP64 path's (tests/test_gpu_parity.py derives the bound),
with the first and the second launch variant of every pass; the coarse-space passes by what they are for: a
deflated solve reaches the same residual in no more iterations.
"""
import math

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_0906_3978_gb300 as wf  # noqa: E402

SIZES = [16, 24, 32, 48, 64, 72, 96, 108, 128, 144, 192, 216, 256, 288, 384]
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    wf.build()
    c = wf.Context(0)
    yield c
    c.close()


def system(ctx, n):
    pr = synth.problem("c2", n_override=n, cache=False)
    nobs = ctx.grid_assign(torch.from_numpy(pr.pos).to(DEV), pr.n, pr.box, pr.scheme, 2)
    w, _, b, nbar = ctx.build_noise(pr.sel, nobs, pr.n_gal, pr.box)
    return pr, w, b, nbar


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("n", SIZES)
def test_first_iterates_every_size(ctx, n, variant):
    pr, w, b, nbar = system(ctx, n)
    before = ctx.tune_get()
    ctx.tune_set({f"{p}/f32/{n}": variant for p in ("xinv", "xupd", "ypass", "zturn")})
    try:
        for precond in (1, 0):
            out = [ctx.solve(w, nbar, b, pr.box, pr.pk_k, pr.pk_p, tol=1e-14, max_iter=3, precond=precond, prec=prec,
                             check=False)[0] for prec in (wf.FP64, wf.MIXED)]
            d = float(torch.linalg.norm(out[1] - out[0]) / torch.linalg.norm(out[0]))
            assert d <= 12.0 * math.log2(n) * 2.0 ** -24, (precond, d)
    finally:
        ctx.tune_set({f"{p}/f32/{n}": 0 for p in ("xinv", "xupd", "ypass", "zturn")})
        ctx.tune_set(before)


@pytest.mark.parametrize("n,k", [(16, 3), (24, 2), (48, 3), (72, 4), (108, 3), (144, 5), (216, 4), (256, 6)])
def test_coarse_space_passes(ctx, n, k):
    pr, w, b, nbar = system(ctx, n)
    args = dict(tol=1e-8, prec=wf.MIXED)
    _, plain = ctx.solve(w, nbar, b, pr.box, pr.pk_k, pr.pk_p, deflate=0, **args)
    _, info = ctx.solve(w, nbar, b, pr.box, pr.pk_k, pr.pk_p, deflate=k, **args)
    assert info.rel_residual <= 1e-8
    assert info.iters <= plain.iters + 2 * info.outer_iters
