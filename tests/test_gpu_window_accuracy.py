"""The window's radial law errs no more than the math library's logarithm and exponential would let it.

Both sides are held to the law in long double at the offsets' FP64 values: the library's side is the same formula in torch on
the device.  Over ~10^5 nodes the rms error of a side repeats to better than 1%; 2% are allowed.
"""
import math

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_0906_3978_gb300 as wf  # noqa: E402

DEV = "cuda:0"


@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 63, reason="long double is no wider than double here")
@pytest.mark.parametrize("n,kind,params", [(64, 1, (0.6, 0.0)), (64, 2, (0.3, 2.0)), (96, 2, (0.45, 3.5))])
def test_radial_law_rms(n, kind, params):
    wf.build()
    box = 1.953125 * n
    sel = synth.Selection(observer=(0.0, 0.5 * box, 0.04 * box), axis=(1.0, 0.0, 0.0), half_angle=math.radians(50.0),
                          holes=np.zeros((0, 4)), radial_kind=kind, radial_params=(params[0] * box, params[1], 0.0, 0.0))
    with wf.Context(0) as ctx:
        n_obs = torch.ones((n, n, n), dtype=torch.float64, device=DEV)
        w = ctx.build_noise(sel, n_obs, 1000, box)[0].cpu().numpy()
    at = np.nonzero(w > 0.0)
    d = [at[a] * np.float64(box / n) - np.float64(sel.observer[a]) for a in range(3)]
    p0, p1 = sel.radial_params[:2]
    r = np.sqrt(sum(x.astype(np.longdouble) ** 2 for x in d))
    t = r / np.longdouble(p0)
    law = np.exp(-t * t) if kind == 1 else np.exp(np.longdouble(p1) * (np.log(t) + (1 - t)))
    dx, dy, dz = (torch.from_numpy(x).to(DEV) for x in d)
    td = torch.sqrt((dx * dx + dy * dy) + dz * dz) / torch.full_like(dx, p0)  # (a scalar divisor is multiplied by 1 / p0)
    lib = torch.exp(-(td * td)) if kind == 1 else torch.exp(p1 * (torch.log(td) + (1.0 - td)))
    rms = [float(np.sqrt(np.mean(((v.astype(np.longdouble) - law) / law).astype(np.float64) ** 2)))
           for v in (w[at], lib.cpu().numpy())]
    assert rms[0] <= 1.02 * rms[1], rms
