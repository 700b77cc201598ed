"""The measured work of the library: the steps of a Wiener reconstruction through the public binding.

A reconstruction is gridding (`grid_assign`) -> window, data, noise (`build_noise`) -> Wiener solve
(`solve`), or many of them at once (`solve_batch`); around it stand the inverse-weighting estimator
(`grid_assign_weighted`), the sky-mask projection (`project_mask`), smoothing and deconvolution of a field
(`smooth`, `deconvolve`) and the evaluation of a result (`compare`, `density_stats`).  Sizes, boxes and
galaxy numbers are those of the benchmark workloads (64^3 over 200 Mpc/h, 256^3 and 512^3 over
500 Mpc/h), of the batched mocks (1.953 Mpc/h cells) and of the tests (ragged 2^a 3^b sizes).

The inputs are synthetic: log-normal galaxies thinned by a survey selection (a cone with holes and a
gamma radial law, or a corner observer with a Gaussian one), made on the GPU with torch.  `exact` restates
each step with torch in FP64.  The FP64 solutions of the mixed-precision solves are returned in single
precision, as an ensemble of maps is kept: a solution to a residual of 1e-6 holds no more digits.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_0906_3978_gb300 as wf

SIZES = (16, 24, 32, 48, 64, 72, 96, 108, 128, 144, 192, 216, 256, 288, 384, 512)
TWO_PI = 2.0 * math.pi
DEV = "cuda"


# ---- the cases ------------------------------------------------------------------------------
def listed():
    return [
        # the smallest survey workload: 2e4 galaxies, CIC, 128^3 fine grid (launches and latency)
        dict(name="grid_cic_64", kind="grid", n=64, cell=3.125, n_gal=20000, scheme=1, ss=2, survey="corner"),
        # the headline workload's gridding: 5e5 galaxies, TSC, 1024^3 fine grid
        dict(name="grid_tsc_512", kind="grid", n=512, cell=0.9765625, n_gal=500000, scheme=2, ss=2, survey="cone"),
        # inverse-weighting estimator on a ragged size: galaxies of mass 1 / w
        dict(name="grid_weighted_216", kind="weighted", n=216, cell=1.953125, n_gal=120000, scheme=2, ss=2,
             survey="cone"),
        # window, mean density, data and right-hand side of the 256^3 workload
        dict(name="noise_256", kind="noise", n=256, cell=1.953125, n_gal=150000, survey="cone"),
        # one small solve to 1e-8: launches and host steps count
        dict(name="solve_mixed_64", kind="solve", n=64, cell=3.125, n_gal=20000, survey="corner", prec="mixed",
             tol=1e-8, deflate=-1),
        # an ordinary mock on a ragged size
        dict(name="solve_mixed_144", kind="solve", n=144, cell=1.953125, n_gal=40000, survey="cone", prec="mixed",
             tol=1e-6, deflate=-1),
        # the headline: 512^3 to 1e-6, mixed precision, coarse space by size
        dict(name="solve_mixed_512", kind="solve", n=512, cell=0.9765625, n_gal=500000, survey="cone", prec="mixed",
             tol=1e-6, deflate=-1),
        # a reference solution in FP64 throughout, to 1e-12, on a ragged size
        dict(name="solve_fp64_108", kind="solve", n=108, cell=1.953125, n_gal=20000, survey="cone", prec="fp64",
             tol=1e-12, deflate=0),
        # an ensemble of 12 mocks of uneven size in one call
        dict(name="batch_mixed_12", kind="batch", sizes="64,96,128,192", count=12, cell=1.953125, density=0.02,
             tol=1e-6),
        # a reconstruction smoothed with r_S = 10 Mpc/h
        dict(name="smooth_256", kind="smooth", n=256, cell=1.953125, op="smooth", radius=10.0),
        # the 3D mask of a 1024 x 512 sky map, 2000 samples per ray, on the 512^3 grid
        dict(name="mask_512", kind="mask", n=512, cell=0.9765625, n_alpha=1024, n_delta=512, n_r=2000),
        # quality measures and density histograms of a smoothed 256^3 field
        dict(name="evaluate_256", kind="evaluate", n=256, cell=1.953125, n_bins=200, n_shells=4),
    ]


def _log_size(rng, lo, hi):
    """A compiled size in [lo, hi], spread over the logarithm."""
    t = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((s for s in SIZES if lo <= s <= hi), key=lambda s: abs(math.log(s / t)))


def draw(rng):
    kind = rng.choice(["grid", "grid", "weighted", "noise", "solve", "solve", "solve", "batch", "smooth", "mask",
                       "evaluate"])
    cell = round(math.exp(rng.uniform(math.log(0.95), math.log(4.0))), 6)
    dens = math.exp(rng.uniform(math.log(0.0035), math.log(0.1)))

    def gal(n):
        return max(50, min(int(dens * n ** 3), 2000000))

    survey = rng.choice(["cone", "cone", "corner"])
    if kind == "grid":
        n = _log_size(rng, 16, 512)
        return dict(kind=kind, n=n, cell=cell, n_gal=gal(n), scheme=rng.choice([1, 2, 2]), ss=rng.choice([1, 2, 2, 2]),
                    survey=survey)
    if kind == "weighted":
        n = _log_size(rng, 16, 384)
        return dict(kind=kind, n=n, cell=cell, n_gal=gal(n), scheme=rng.choice([1, 2, 2]), ss=2, survey=survey)
    if kind == "noise":
        n = _log_size(rng, 16, 512)
        return dict(kind=kind, n=n, cell=cell, n_gal=gal(n), survey=survey)
    if kind == "solve":
        prec = rng.choice(["mixed", "mixed", "mixed", "fp64"])
        if prec == "fp64":
            n = _log_size(rng, 16, 128)
            return dict(kind=kind, n=n, cell=cell, n_gal=gal(n), survey=survey, prec=prec, tol=1e-12, deflate=0)
        n = _log_size(rng, 24, 384)
        return dict(kind=kind, n=n, cell=cell, n_gal=gal(n), survey=survey, prec=prec,
                    tol=rng.choice([1e-6, 1e-6, 1e-8]), deflate=rng.choice([-1, -1, 0]))
    if kind == "batch":
        sizes = sorted(_log_size(rng, 32, 144) for _ in range(3))
        return dict(kind=kind, sizes=",".join(str(s) for s in sizes), count=rng.randint(3, 16), cell=cell,
                    density=round(max(dens, 0.01), 6), tol=1e-6)
    if kind == "smooth":
        n = _log_size(rng, 16, 512)
        return dict(kind=kind, n=n, cell=cell, op=rng.choice(["smooth", "deconvolve"]),
                    radius=round(cell * rng.uniform(1.0, 8.0), 6))
    if kind == "mask":
        n = _log_size(rng, 32, 384)
        na = 2 * rng.randint(n // 2 + 1, n + 40)
        return dict(kind=kind, n=n, cell=cell, n_alpha=na, n_delta=na // 2 + rng.randint(0, 5),
                    n_r=rng.randint(2 * n, 4 * n))
    n = _log_size(rng, 16, 512)
    return dict(kind=kind, n=n, cell=cell, n_bins=rng.randint(50, 400), n_shells=rng.randint(1, 4))


# ---- synthetic survey -----------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _power():
    """A smooth LCDM-shaped P(k) in (Mpc/h)^3 (BBKS transfer function, Gamma = 0.175, sigma_8 = 0.8)."""
    def shape(k):
        q = k / 0.175
        t = np.log(1 + 2.34 * q) / (2.34 * q)
        return k * (t * (1 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3 + (6.71 * q) ** 4) ** -0.25) ** 2

    kk = np.geomspace(1e-5, 1e2, 8192)
    x = 8.0 * kk
    win = 3.0 * (np.sin(x) - x * np.cos(x)) / x ** 3
    f = kk ** 3 * shape(kk) * win ** 2 / (2.0 * math.pi ** 2)
    lk = np.log(kk)
    amp = 0.64 / float(np.sum(0.5 * (f[1:] + f[:-1]) * np.diff(lk)))
    k = np.geomspace(1e-4, 1e2, 256)
    return k, amp * shape(k)


def _survey(case, box, seed):
    """The selection handed to the library: a 30-degree cone from the near face with 2-degree holes over
    5% of it and a gamma radial law, or a cone along the diagonal from the corner with a Gaussian law."""
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 17])
    if case.get("survey", "cone") == "corner":
        a = 1.0 / math.sqrt(3.0)
        return SimpleNamespace(observer=(0.0, 0.0, 0.0), axis=(a, a, a), half_angle=math.radians(30.0),
                               holes=np.zeros((0, 4)), radial_kind=1, radial_params=(0.6 * box, 0.0, 0.0, 0.0))
    half, rho = math.radians(30.0), math.radians(2.0)
    nh = int(round(0.05 * (1.0 - math.cos(half)) / (1.0 - math.cos(rho))))
    mu = 1.0 - rng.random(nh) * (1.0 - math.cos(half))
    phi = TWO_PI * rng.random(nh)
    s = np.sqrt(np.maximum(0.0, 1.0 - mu * mu))
    holes = np.stack([mu, s * np.cos(phi), s * np.sin(phi), np.full(nh, rho)], axis=1)
    holes[:, :3] /= np.linalg.norm(holes[:, :3], axis=1, keepdims=True)
    return SimpleNamespace(observer=(0.0, 0.5 * box, 0.04 * box), axis=(1.0, 0.0, 0.0), half_angle=half, holes=holes,
                           radial_kind=2, radial_params=(0.3 * box, 2.0, 0.0, 0.0))


def _selection(sel, dx, dy, dz):
    """The selection at offsets from the observer (FP64, the operations in the order of the definition)."""
    r = torch.sqrt((dx * dx + dy * dy) + dz * dz)
    ok = ((dx * sel.axis[0] + dy * sel.axis[1]) + dz * sel.axis[2]) >= r * math.cos(sel.half_angle)
    for h in np.asarray(sel.holes).reshape(-1, 4):
        ok &= ~(((dx * float(h[0]) + dy * float(h[1])) + dz * float(h[2])) > r * math.cos(float(h[3])))
    ok &= r > 0
    p = sel.radial_params
    if sel.radial_kind == 0:
        f = torch.ones_like(r)
    elif sel.radial_kind == 1:
        f = torch.exp(-((r / p[0]) ** 2))
    else:
        t = torch.where(r > 0, r, torch.ones_like(r)) / p[0]
        f = torch.exp(p[1] * (torch.log(t) + (1.0 - t)))
    return torch.where(ok, f, torch.zeros_like(f))


def _window(sel, n, box):
    """w at the nodes i H."""
    h = box / n
    i = torch.arange(n, dtype=torch.float64, device=DEV) * h
    o = sel.observer
    w = torch.empty((n, n, n), dtype=torch.float64, device=DEV)
    step = max(1, (1 << 24) // (n * n))
    for x0 in range(0, n, step):
        w[x0:x0 + step] = _selection(sel, (i[x0:x0 + step] - o[0])[:, None, None], (i - o[1])[None, :, None],
                                     (i - o[2])[None, None, :])
    return w


def _n2(n, half=True):
    """|m|^2 of the signed DFT indices (the last axis halved, as rfftn has it)."""
    f = torch.arange(n, device=DEV)
    f = torch.where(f > n // 2, f - n, f)
    z = torch.arange(n // 2 + 1, device=DEV) if half else f
    return (f * f)[:, None, None] + (f * f)[None, :, None] + (z * z)[None, None, :]


def _interp_power(k, pk):
    """log-log linear interpolation, the end segments extrapolated (numpy FP64)."""
    lk, lp = np.log(pk[0]), np.log(pk[1])
    x = np.log(k)
    j = np.clip(np.searchsorted(lk, x) - 1, 0, len(lk) - 2)
    t = (x - lk[j]) / (lk[j + 1] - lk[j])
    return np.exp(lp[j] + t * (lp[j + 1] - lp[j]))


def _field(n, box, gen, pk, smooth=0.0):
    """A Gaussian field with spectrum P(k) (FP32), optionally smoothed."""
    spec = torch.fft.rfftn(torch.randn((n, n, n), dtype=torch.float32, device=DEV, generator=gen))
    kf = TWO_PI / box
    m = np.arange(3 * (n // 2) ** 2 + 1, dtype=np.float64)
    tab = np.zeros_like(m)
    k = kf * np.sqrt(m[1:])
    tab[1:] = np.sqrt(_interp_power(k, pk) / (box / n) ** 3) * np.exp(-0.5 * (k * smooth) ** 2)
    spec *= torch.from_numpy(tab).to(DEV, torch.float32)[_n2(n)]
    return torch.fft.irfftn(spec, s=(n, n, n))


def _counts(case, n, box, sel, gen, pk, n_gal, w=None):
    """Poisson galaxy counts per cell of a log-normal field seen through the selection."""
    g = _field(n, box, gen, pk)
    lam = torch.exp(g - 0.5 * g.var())
    del g
    lam *= _window(sel, n, box).float() if w is None else w.float()
    lam *= n_gal / float(lam.sum(dtype=torch.float64))
    return torch.poisson(lam, generator=gen)


def _galaxies(case, seed):
    """(positions [N_gal, 3], selection) of a catalogue; positions uniform in their cells."""
    n, box = case["n"], case["n"] * case["cell"]
    gen, pk = _gen(seed), _power()
    sel = _survey(case, box, seed)
    c = _counts(case, n, box, sel, gen, pk, case["n_gal"]).to(torch.int64).reshape(-1)
    idx = torch.repeat_interleave(torch.arange(n ** 3, device=DEV), c)
    cellxyz = torch.stack([idx // (n * n), (idx // n) % n, idx % n], dim=1).to(torch.float64)
    u = torch.rand(cellxyz.shape, dtype=torch.float64, device=DEV, generator=gen)
    pos = (cellxyz + u) * (box / n)
    return pos[torch.randperm(pos.shape[0], device=DEV, generator=gen)].contiguous(), sel


def _observed(case, seed):
    """(n_obs [n, n, n], N_gal, selection): low-passed counts as the gridding gives them."""
    n, box = case["n"], case["n"] * case["cell"]
    gen, pk = _gen(seed), _power()
    sel = _survey(case, box, seed)
    c = _counts(case, n, box, sel, gen, pk, case["n_gal"]).to(torch.float64)
    spec = torch.fft.rfftn(c)
    f = torch.fft.fftfreq(n, device=DEV, dtype=torch.float64)
    s = torch.where(f.abs() < 0.5, torch.sinc(0.5 * f) ** 3, torch.zeros_like(f))
    fz = torch.fft.rfftfreq(n, device=DEV, dtype=torch.float64)
    sz = torch.where(fz < 0.5, torch.sinc(0.5 * fz) ** 3, torch.zeros_like(fz))
    spec *= s[:, None, None] * s[None, :, None] * sz[None, None, :]
    return torch.fft.irfftn(spec, s=(n, n, n)), int(round(float(c.sum()))), sel


def _data(n_obs, n_gal, w):
    """(nbar, d, b) of the data and noise model."""
    nbar = n_gal / float(w.sum())
    d = n_obs / nbar - w
    return nbar, d, torch.where(w > 0, nbar * d, torch.zeros_like(d))


def _system(case, seed):
    """One Wiener system: w, nbar, b, box, P(k)."""
    n_obs, n_gal, sel = _observed(case, seed)
    w = _window(sel, case["n"], case["n"] * case["cell"])
    nbar, _, b = _data(n_obs, n_gal, w)
    k, p = _power()
    return dict(w=w, nbar=nbar, b=b, box=case["n"] * case["cell"], pk_k=k, pk_p=p)


def _members(case):
    sizes = [int(s) for s in case["sizes"].split(",")]
    for i in range(case["count"]):
        n = sizes[(i * 5 + i // len(sizes)) % len(sizes)]
        yield i, dict(n=n, cell=case["cell"], n_gal=max(50, int(case["density"] * n ** 3)),
                      survey="corner" if i % 3 == 2 else "cone")


def _masses(case, pos, sel):
    """1 / w at each galaxy, capped as an estimator caps the weights of nearly unobserved regions."""
    o = sel.observer
    w = _selection(sel, pos[:, 0] - o[0], pos[:, 1] - o[1], pos[:, 2] - o[2])
    return torch.where(w > 1e-3, 1.0 / w.clamp_min(1e-3), torch.zeros_like(w))


def _sky(case, seed):
    """(sky map [n_delta, n_alpha], geometry, radial table) of a survey seen from inside the box."""
    n, box = case["n"], case["n"] * case["cell"]
    gen = _gen(seed)
    na, nd, nr = case["n_alpha"], case["n_delta"], case["n_r"]
    al = (torch.arange(na, dtype=torch.float64, device=DEV) + 0.5) * (TWO_PI / na)
    de = -0.5 * math.pi + (torch.arange(nd, dtype=torch.float64, device=DEV) + 0.5) * (math.pi / nd)
    inside = torch.cos(de)[:, None] * torch.cos(al)[None, :] >= math.cos(math.radians(30.0))
    comp = 0.8 + 0.2 * torch.rand((nd, na), dtype=torch.float64, device=DEV, generator=gen)
    sky = torch.where(inside, comp, torch.zeros_like(comp)).contiguous()
    dr = box / nr
    t = (np.arange(nr) + 0.5) * dr / (0.3 * box)
    wr = np.clip(t ** 2 * np.exp(2.0 * (1.0 - t)), 0.0, 1.0)
    geo = dict(alpha0=0.0, dalpha=TWO_PI / na, delta0=-0.5 * math.pi, ddelta=math.pi / nd,
               observer=(0.0, 0.5 * box, 0.04 * box), dr=dr)
    return sky, geo, wr


def _evaluated(case, seed):
    """A reference overdensity, a reconstruction of it and a window."""
    n, box = case["n"], case["n"] * case["cell"]
    gen, pk = _gen(seed), _power()
    g = _field(n, box, gen, pk, smooth=2.0 * case["cell"]).to(torch.float64)
    truth = torch.exp(g - 0.5 * g.var()) - 1.0
    rec = 0.8 * truth + 0.1 * torch.randn((n, n, n), dtype=torch.float64, device=DEV, generator=gen)
    w = _window(_survey(case, box, seed), n, box)
    obs = (0.0, 0.5 * box, 0.04 * box)
    s = case["n_shells"]
    shells = [[0.4 * box * i, 0.4 * box * (i + 1) if i + 1 < s else math.inf] for i in range(s)]
    return truth, rec, w, obs, shells


# ---- the library's side ---------------------------------------------------------------------
_CTX = []


def _ctx():
    """The program's one context: a reconstruction code keeps it for its lifetime."""
    if not _CTX:
        _CTX.append(wf.Context(torch.cuda.current_device()))
    return _CTX[0]


def prepare(case, seed):
    kind, n = case["kind"], case.get("n")
    st = SimpleNamespace(case=case, ctx=_ctx(), n=n, box=n * case["cell"] if n else None)
    if kind in ("grid", "weighted"):
        st.pos, sel = _galaxies(case, seed)
        st.mass = _masses(case, st.pos, sel) if kind == "weighted" else None
    elif kind == "noise":
        st.n_obs, st.n_gal, st.sel = _observed(case, seed)
    elif kind == "solve":
        st.sys = _system(case, seed)
    elif kind == "batch":
        st.probs = [dict(_system(c, seed * 1009 + i), tol=case["tol"], max_iter=20000, prec=wf.MIXED, deflate=-1)
                    for i, c in _members(case)]
    elif kind == "smooth":
        st.field = _field(n, st.box, _gen(seed), _power()).to(torch.float64).contiguous()
    elif kind == "mask":
        st.sky, st.geo, st.wr = _sky(case, seed)
    else:
        st.truth, st.rec, st.w, st.obs, st.shells = _evaluated(case, seed)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return st


def run(st):
    c, ctx, kind = st.case, st.ctx, st.case["kind"]
    if kind == "grid":
        return ctx.grid_assign(st.pos, st.n, st.box, c["scheme"], c["ss"])
    if kind == "weighted":
        return ctx.grid_assign_weighted(st.pos, st.mass, st.n, st.box, c["scheme"], c["ss"])
    if kind == "noise":
        w, d, b, nbar = ctx.build_noise(st.sel, st.n_obs, st.n_gal, st.box)
        return dict(w=w, d=d, b=b, nbar=nbar)
    if kind == "solve":
        s, _ = ctx.solve(st.sys["w"], st.sys["nbar"], st.sys["b"], st.box, st.sys["pk_k"], st.sys["pk_p"],
                         tol=c["tol"], max_iter=20000, prec=wf.FP64 if c["prec"] == "fp64" else wf.MIXED,
                         deflate=c["deflate"])
        return s if c["prec"] == "fp64" else s.float()
    if kind == "batch":
        status, maps, _ = ctx.solve_batch(st.probs)
        if status != wf.OK:
            raise RuntimeError(wf.status_string(status))
        return [m.float() for m in maps]
    if kind == "smooth":
        if c["op"] == "deconvolve":
            return ctx.deconvolve(st.field, st.box, 0.42, 5.0, 1.2)
        return ctx.smooth(st.field, st.box, c["radius"])
    if kind == "mask":
        g = st.geo
        return ctx.project_mask(st.sky, st.n, st.box, g["alpha0"], g["dalpha"], g["delta0"], g["ddelta"], g["observer"],
                                g["dr"], st.wr)
    hist, mom = ctx.density_stats(st.rec, st.w, st.box, st.obs, st.shells, -1.0, 6.0 / c["n_bins"], c["n_bins"])
    return dict(measures=ctx.compare(st.rec, st.truth), hist=hist, moments=_columns(mom))


def _columns(mom):
    """The moments by name: their magnitudes differ by many orders."""
    names = ("n_cells", "mean", "mu2", "mu3", "mu4", "skewness", "kurtosis", "pearson")
    return {k: np.ascontiguousarray(mom[..., j]) for j, k in enumerate(names)}


# ---- what a pass cannot do without ------------------------------------------------------------
def _fft(n):
    """Operations of one real 3D transform of n^3 points."""
    return 2.5 * n ** 3 * math.log2(n ** 3)


def _solve_work(n, prec):
    """w and b read, s written; a CG iteration reads and writes p, x and r, reads the data diagonal and
    takes two transforms; 100 iterations (mixed, coarse space) or 300 (FP64, to 1e-12) are counted."""
    word, its = (8, 300) if prec == "fp64" else (4, 100)
    return 24.0 * n ** 3 + its * 7.0 * word * n ** 3, its * (2 * _fft(n) + 14.0 * n ** 3)


def work(case):
    kind, n = case["kind"], case.get("n")
    v = float(n) ** 3 if n else 0.0
    if kind in ("grid", "weighted"):
        ng = case["n_gal"]
        fl = _fft(2 * n) + _fft(n) if case["ss"] == 2 else v
        return {"bytes": (24.0 if kind == "grid" else 32.0) * ng + 8 * v, "flops": fl + 200.0 * ng}
    if kind == "noise":
        return {"bytes": 32 * v, "flops": 30 * v}
    if kind == "solve":
        b, f = _solve_work(n, case["prec"])
        return {"bytes": b, "flops": f}
    if kind == "batch":
        bf = [_solve_work(c["n"], "mixed") for _, c in _members(case)]
        return {"bytes": sum(x[0] for x in bf), "flops": sum(x[1] for x in bf)}
    if kind == "smooth":
        return {"bytes": 16 * v, "flops": 2 * _fft(n) + v}
    if kind == "mask":
        pix = float(case["n_alpha"]) * case["n_delta"]
        return {"bytes": 8 * pix + 8 * v, "flops": 8.0 * pix * case["n_r"]}
    return {"bytes": 24 * v, "flops": 50 * v}


# ---- the same in FP64 with torch ---------------------------------------------------------------
def _axis(x, scale, nf, scheme):
    """Node indices and Q16 weights of one axis."""
    q = torch.floor(x * scale).to(torch.int64) % (nf * 65536)
    if scheme == wf.CIC:
        f = q & 0xFFFF
        return [(q >> 16) % nf, ((q >> 16) + 1) % nf], [65536 - f, f]
    qp = q + 32768
    j, d = qp >> 16, (qp & 0xFFFF) - 32768
    wm, wp = (32768 - d) ** 2 >> 17, (32768 + d) ** 2 >> 17
    return [(j - 1) % nf, j % nf, (j + 1) % nf], [wm, 65536 - wm - wp, wp]


def _gridded(pos, mass, n, box, scheme, ss):
    nf = ss * n
    scale = (nf * 65536.0) / box
    ax = [_axis(pos[:, a], scale, nf, scheme) for a in range(3)]
    fine = torch.zeros(nf ** 3, dtype=torch.int64, device=DEV)
    for i, wi in zip(*ax[0]):
        for j, wj in zip(*ax[1]):
            for k, wk in zip(*ax[2]):
                add = wi * wj * wk
                if mass is not None:
                    add = torch.round(add.to(torch.float64) * mass * (1.0 / 65536.0)).to(torch.int64)
                fine.index_add_(0, (i * nf + j) * nf + k, add)
    f = fine.to(torch.float64) * (2.0 ** -48 if mass is None else 2.0 ** -32)
    del fine
    f = f.reshape(nf, nf, nf)
    if ss == 1:
        return f
    spec = torch.fft.rfftn(f)
    del f
    h = n // 2
    out = torch.zeros((n, n, h + 1), dtype=torch.complex128, device=DEV)
    for a, sa in ((slice(0, h), slice(0, h)), (slice(h + 1, n), slice(nf - h + 1, nf))):
        for b, sb in ((slice(0, h), slice(0, h)), (slice(h + 1, n), slice(nf - h + 1, nf))):
            out[a, b, :h] = spec[sa, sb, :h]
    del spec
    return torch.fft.irfftn(out, s=(n, n, n))


def _solved(sy, target):
    """The Wiener mean, to a relative residual of `target` in FP64: preconditioned CG on half spectra in
    single precision inside an FP64 refinement."""
    w, nbar, b, box = sy["w"], sy["nbar"], sy["b"], sy["box"]
    n = b.shape[0]
    v, dv = float(n) ** 3, (box / n) ** 3
    m = np.arange(3 * (n // 2) ** 2 + 1, dtype=np.float64)
    sinv = np.zeros_like(m)
    sinv[1:] = dv / _interp_power((TWO_PI / box) * np.sqrt(m[1:]), (sy["pk_k"], sy["pk_p"]))
    c = np.ones_like(m)
    c[1:] = 1.0 / np.sqrt(sinv[1:])
    c[0] = 1.0 / math.sqrt(nbar * float(w.sum()) / v)
    n2 = _n2(n)
    si = torch.from_numpy(sinv).to(DEV)[n2]
    cs = torch.from_numpy(c).to(DEV, torch.float32)[n2]
    del n2
    d32 = (nbar * w).float()
    wgt = torch.full((n // 2 + 1,), 2.0, device=DEV)
    wgt[0] = wgt[-1] = 1.0
    wgt2 = wgt.repeat_interleave(2).reshape(1, 1, -1)

    def dot(x, y):
        x, y = torch.view_as_real(x).reshape(n, n, -1), torch.view_as_real(y).reshape(n, n, -1)
        return ((x * y).sum(dim=(0, 1), dtype=torch.float64) * wgt2.reshape(-1)).sum()

    def apply(p):
        t = torch.fft.irfftn(p * cs, s=(n, n, n))
        t *= d32
        q = torch.fft.rfftn(t)
        q *= cs
        q += p
        q[0, 0, 0] -= p[0, 0, 0]
        return q

    x = torch.zeros_like(b)
    res, bn = b.clone(), float(torch.linalg.norm(b))
    rel = 1.0
    for _ in range(14):
        if rel <= target:
            break
        r = torch.fft.rfftn((res / (rel * bn)).float()) * cs
        y, p, rr = torch.zeros_like(r), r.clone(), dot(r, r)
        rr0, it = float(rr), 0
        while it < 600:
            q = apply(p)
            a = rr / dot(p, q)
            y += a.float() * p
            r -= a.float() * q
            new = dot(r, r)
            p = r + (new / rr).float() * p
            rr = new
            it += 1
            if it % 10 == 0 and not float(rr) > 1e-9 * rr0:
                break
        x += (rel * bn) * torch.fft.irfftn(y * cs, s=(n, n, n)).double()
        del y, p, q, r
        res = b - (torch.fft.irfftn(si * torch.fft.rfftn(x), s=(n, n, n)) + nbar * w * x)
        rel = float(torch.linalg.norm(res)) / bn
    return x


def _rsd(k, beta, sigma_v):
    """<K D>_mu by 128-point Gauss-Legendre quadrature over mu."""
    mu, wt = np.polynomial.legendre.leggauss(128)
    mu, wt = 0.5 * (mu + 1.0), 0.5 * wt
    return ((1 + beta * mu ** 2) ** 2 / (1 + 0.5 * (k[:, None] * sigma_v * mu) ** 2) * wt).sum(axis=1)


def _masked(case, sky, geo, wr):
    """The projected mask: each sample's cell decided in FP32 as the definition has it, averages in FP64."""
    n, box = case["n"], case["n"] * case["cell"]
    na, nd, nr = case["n_alpha"], case["n_delta"], case["n_r"]
    h = box / n
    al = geo["alpha0"] + (np.arange(na) + 0.5) * geo["dalpha"]
    de = geo["delta0"] + (np.arange(nd) + 0.5) * geo["ddelta"]
    ca, sa, cd, sd = (torch.from_numpy(f(x)).to(DEV) for f, x in ((np.cos, al), (np.sin, al), (np.cos, de), (np.sin, de)))
    step = geo["dr"] / h
    g = [((cd[:, None] * ca[None, :]) * step).float(), ((cd[:, None] * sa[None, :]) * step).float(),
         (sd * step).float()[:, None].expand(nd, na)]
    o = [float(np.float32(v / h)) for v in geo["observer"]]
    tk = (torch.arange(nr, device=DEV).float() + 0.5)[None, None, :]
    rad = torch.from_numpy(np.asarray(wr)).to(DEV)
    sums = torch.zeros((3, n ** 3), dtype=torch.float64, device=DEV)
    rows = max(1, (1 << 25) // (na * nr))
    for j in range(0, nd, rows):
        cells = [torch.floor(tk * g[a][j:j + rows, :, None] + o[a]) for a in range(3)]
        ok = torch.ones_like(cells[0], dtype=torch.bool)
        for x in cells:
            ok &= (x >= 0) & (x < n)
        at = ((cells[0].long() * n + cells[1].long()) * n + cells[2].long())[ok]
        s = sky[j:j + rows, :, None].expand(ok.shape)[ok]
        sums[0].index_add_(0, at, s)
        sums[1].index_add_(0, at, rad[None, None, :].expand(ok.shape)[ok])
        sums[2].index_add_(0, at, torch.ones_like(s))
    cnt = sums[2].clamp_min(1.0)
    return ((sums[0] / cnt) * (sums[1] / cnt)).reshape(n, n, n)


def _moments(hist, lo, width):
    """N, mean, mu_2..mu_4, skewness, kurtosis and Pearson's skewness from the bin centres."""
    f = hist[..., :-2].astype(np.float64)
    c = (lo + (np.arange(f.shape[-1]) + 0.5) * width) - 1.0
    out = np.full(f.shape[:-1] + (8,), np.nan)
    for i in np.ndindex(*f.shape[:-1]):
        tot = f[i].sum()
        out[i][0] = tot
        if tot > 0:
            mean = (f[i] * c).sum() / tot
            mu = [(f[i] * (c - mean) ** p).sum() / tot for p in (2, 3, 4)]
            sig = math.sqrt(mu[0])
            with np.errstate(divide="ignore", invalid="ignore"):
                out[i][1:] = [mean, mu[0], mu[1], mu[2], np.float64(mu[1]) / sig ** 3, np.float64(mu[2]) / mu[0] ** 2 - 3.0,
                              np.float64(mean - c[int(np.argmax(f[i]))]) / sig]
    return out


def exact(case, seed):
    kind, n = case["kind"], case.get("n")
    box = n * case["cell"] if n else None
    if kind in ("grid", "weighted"):
        pos, sel = _galaxies(case, seed)
        return _gridded(pos, _masses(case, pos, sel) if kind == "weighted" else None, n, box, case["scheme"], case["ss"])
    if kind == "noise":
        n_obs, n_gal, sel = _observed(case, seed)
        w = _window(sel, n, box)
        nbar, d, b = _data(n_obs, n_gal, w)
        return dict(w=w, d=d, b=b, nbar=nbar)
    if kind == "solve":
        return _solved(_system(case, seed), 1e-13 if case["prec"] == "fp64" else 1e-10)
    if kind == "batch":
        return [_solved(_system(c, seed * 1009 + i), 1e-9) for i, c in _members(case)]
    if kind == "smooth":
        f = _field(n, box, _gen(seed), _power()).to(torch.float64)
        k = (TWO_PI / box) * np.sqrt(np.arange(3 * (n // 2) ** 2 + 1, dtype=np.float64))
        if case["op"] == "deconvolve":
            tab = 1.0 / (1.2 * np.sqrt(_rsd(k, 0.42, 5.0)))
        else:
            tab = np.exp(-0.5 * (k * case["radius"]) ** 2)
        return torch.fft.irfftn(torch.fft.rfftn(f) * torch.from_numpy(tab).to(DEV)[_n2(n)], s=(n, n, n))
    if kind == "mask":
        return _masked(case, *_sky(case, seed))
    truth, rec, w, obs, shells = _evaluated(case, seed)
    a, b = 1.0 + rec, 1.0 + truth
    ok = (a > 0) & (b > 0)
    kl = torch.where(ok, a * torch.log(torch.where(ok, a, b.abs() + 1) / torch.where(ok, b, b.abs() + 1)),
                     torch.zeros_like(a))
    measures = dict(r=float((rec * truth).sum() / (rec.norm() * truth.norm())),
                    d_euc=float(((rec - truth) ** 2).mean().sqrt()), d_kl=float(kl.mean()),
                    kl_excluded=int((~ok).sum()))
    nb, width = case["n_bins"], 6.0 / case["n_bins"]
    i = torch.arange(n, dtype=torch.float64, device=DEV) * (box / n)
    dx, dy, dz = (i - obs[0])[:, None, None], (i - obs[1])[None, :, None], (i - obs[2])[None, None, :]
    r = torch.sqrt((dx * dx + dy * dy) + dz * dz)
    q = torch.floor((a - -1.0) / width)
    slot = torch.where(q < 0, nb, torch.where(q >= nb, nb + 1, q)).to(torch.int64)
    hist = np.zeros((len(shells), 2, nb + 2), dtype=np.int64)
    for s, (lo, hi) in enumerate(shells):
        for g in (0, 1):
            at = slot[(r >= lo) & (r < hi) & ((w > 0) if g == 0 else (w <= 0))]
            hist[s, g] = torch.bincount(at, minlength=nb + 2).cpu().numpy()
    return dict(measures=measures, hist=hist, moments=_columns(_moments(hist, -1.0, width)))
