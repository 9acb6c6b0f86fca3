"""What a user of the framework has it do, as cases to measure.

The work of the library is the evaluation of parametric cluster-lens models:
maps of one model over a grid, and the chi2 of many parameter sets against
multiple-image constraints, alone, inside a sampler or with predicted images.
The sizes are those of this repository's benchmark, tests and request mix:
grids of 64 to 8192 nodes a side, 10 to 2000 potentials, 1 to 4096 parameter
sets, the 100-source constraint table of the 1000-potential model.

A case is a dict; "path" says which entry point it calls:

  hess, grad, pot   device maps (LENS_MIXED, or LENS_FP64 with "fp64")
  host              halo table -> upload -> deflection map in pinned memory
  source            source-plane chi2 of P sets, static sums cached
  mcmc              one Metropolis step of P chains over that chi2
  scaled            source-plane chi2 with the members' scaling factors free
                    ("nodes" > 0: with the scaling cache)
  image             image-plane chi2 of P sets with predicted images

The Hessian maps' magnification is handed on as its inverse det A = 1/mu, as a
program that traces critical curves takes it: mu itself has poles there.
"""
import json
import math
import os

import numpy as np
import torch

from paper_2004_06352_gb300 import api, inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GOLDEN = os.path.join(ROOT, "tests", "golden", "cfg2_constraints.json")
SIGMA = np.tile([0.1, 0.1, 0.01, 0.02, 0.01, 1.0, 0.05], 2)  # proposal widths of the 14 parameters
TEMPERATURE = 50.0
FT_RANGE = (0.5, 2.0)  # prior on the members' r_cut factor


def _map(name, path, nx, ny, n, half, rcut=8.0, dls=1.0, fp64=False, kinds="cluster"):
    return dict(name=name, path=path, nx=nx, ny=ny, n=n, half=half, rcut=rcut, dls=dls, fp64=fp64, kinds=kinds)


def _fit(name, path, P, n, nsrc, variant=0, grid=0, nodes=0):
    return dict(name=name, path=path, P=P, n=n, nsrc=nsrc, variant=variant, grid=grid, nodes=nodes)


def listed():
    return [
        # the benchmark: all six planes of a 1000-potential cluster at HST sampling
        _map("hess_2048_1000", "hess", 2048, 2048, 1000, 100.0),
        # the smallest request of the serving mix, where launches and latency count
        _map("hess_512_10", "hess", 512, 512, 10, 100.0, dls=0.8),
        # the largest request of the serving mix
        _map("hess_8192_2000", "hess", 8192, 8192, 2000, 100.0),
        # the published benchmark's map shape: 217 potentials on a 5000^2 grid over 150 arcsec
        _map("grad_5000_217", "grad", 5000, 5000, 217, 75.0),
        # end to end with an odd grid: table uploaded, map streamed to host memory, model released;
        # members with large cut radii (r_cut* = 45 arcsec)
        _map("host_1601_400", "host", 1601, 1203, 400, 80.0, rcut=45.0, dls=0.7),
        # potential and time-delay surface of a mid-size model of all potential kinds, ragged grid
        _map("pot_1537_500", "pot", 1537, 1021, 500, 60.0, dls=0.9, kinds="all"),
        # the plain double-precision deflection map of a 10-potential model
        _map("grad64_256_10", "grad", 256, 256, 10, 100.0, dls=0.7, fp64=True, kinds="galaxies"),
        # a step of the Bayesian fit: 4096 walkers over the two cluster potentials
        _fit("mcmc_4096", "mcmc", 4096, 1000, 100),
        # a handful of walkers against part of the images, plain source-plane residuals
        _fit("source_24", "source", 24, 1000, 37, variant=2),
        # a full-size batch of a fit, mu-weighted residuals
        _fit("source_4096_mu", "source", 4096, 300, 100, variant=1),
        # the members' scaling relations free as well, no prior interval given
        _fit("scaled_1000", "scaled", 1000, 1000, 100),
        # predicted images of 256 parameter sets on the 1024^2 search grid
        _fit("image_256", "image", 256, 1000, 100, grid=1024),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["hess", "hess", "grad", "host", "pot", "grad64", "hess64", "mcmc", "source", "scaled", "image"])
    if path in ("mcmc", "source", "scaled", "image"):
        P, n, nsrc = _log(rng, 1, 4096), _log(rng, 20, 1000), rng.randint(5, 100)
        variant = rng.choice([0, 0, 1, 2])
        if path == "image":
            return _fit_drawn(path, _log(rng, 1, 256), n, nsrc, 0, grid=_log(rng, 200, 1024))
        if path == "scaled":
            nodes = rng.choice([0, 32])
            return _fit_drawn(path, P if nodes else min(P, 1000), n, nsrc, variant, nodes=nodes)
        return _fit_drawn(path, P, n, nsrc, variant)
    n, half, rcut = _log(rng, 10, 2000), rng.choice([30.0, 60.0, 75.0, 100.0]), rng.choice([8.0, 8.0, 45.0])
    top = 8192.0 * 8192.0 * (2000.0 if rcut < 10.0 else 400.0) / n  # large members cost up to five times as much
    nx = _log(rng, 64, 8192)
    ny = max(64, min(8192, int(nx * rng.uniform(0.6, 1.4))))
    fp64 = path in ("grad64", "hess64")
    if fp64:  # the FP64 unit's rate bounds what is run in FP64
        top = 3e8 / n
    elif path == "host":
        top = min(top, 3e7)
    elif path == "pot":
        top = min(top, 4096.0 * 4096.0)
    shrink = min(1.0, math.sqrt(top / (float(nx) * ny)))
    nx, ny = max(33, int(nx * shrink)), max(31, int(ny * shrink))
    c = _map("", path.replace("64", "") if fp64 else path, nx, ny, n, half, rcut=rcut,
             dls=round(rng.uniform(0.3, 1.0), 3), fp64=fp64, kinds=rng.choice(["cluster", "cluster", "all", "galaxies"]))
    del c["name"]
    return c


def _fit_drawn(path, P, n, nsrc, variant, **kw):
    c = _fit("", path, P, n, nsrc, variant=variant, **kw)
    del c["name"]
    return c


# ------------------------------------------------------------------- inputs
def _table(case, seed):
    """Halo table of a map case: a cluster (two cluster-scale potentials and
    luminosity-scaled members), galaxies about one cluster potential, or the
    cluster with SIS and point-mass members among the dPIE ones."""
    n = case["n"]
    if case["kinds"] == "galaxies":
        g = [inputs.cfg1_model(seed=seed + k) for k in range((n + 8) // 9)]
        return np.concatenate([g[0][:1]] + [m[1:] for m in g])[:n]
    m = inputs.cfg2_model(seed=seed, n_members=n - 2, rcut_star=case["rcut"])
    m[2:, 1:3] *= case["half"] / 100.0  # members over the map's field
    if case["kinds"] == "all":
        m[5::7, 0] = api.LENS_SIS
        m[9::7, 0] = api.LENS_POINT
        m[5::7, 3:7] = m[9::7, 3:7] = 0.0
    return m


def _grid(case):
    h = case["half"]
    return inputs.grid(case["nx"], field=(-h, h, -h * case["ny"] / case["nx"], h * case["ny"] / case["nx"]), ny=case["ny"])


def _beta(seed):
    return np.random.default_rng([seed, 1]).uniform(-5.0, 5.0, 2)


def _fit_inputs(case, seed):
    """Model, constraints (the first nsrc sources of the fixed table, their
    positions measured anew) and parameter sets."""
    rng = np.random.default_rng([seed, 2])
    m = inputs.cfg2_model()[:case["n"]]
    with open(GOLDEN) as f:
        d = json.load(f)
    off = np.asarray(d["img_off"][:case["nsrc"] + 1], dtype=np.int32)
    k = int(off[-1])
    xy = np.stack([d["x"][:k], d["y"][:k]]) + rng.normal(0.0, 0.02, (2, k))
    cons = inputs.constraints_dict(off, xy[0], xy[1], np.full(k, d["sigma"]), d["dls_ds"][:case["nsrc"]])
    params = inputs.perturbed_params(m, (0, 1), case["P"], seed=seed)
    if case["path"] == "scaled":
        fb = np.clip(rng.normal(1.0, 0.1, case["P"]), 0.6, 1.5)
        ft = np.clip(np.exp(rng.normal(0.0, 0.25, case["P"])), 0.55, 1.9)
        params = np.concatenate([params, fb[:, None], ft[:, None]], axis=1)
    return m, cons, params


_context = None


def _ctx():
    """One context for the program, as a user's holds."""
    global _context
    if _context is None:
        _context = api.Context(0)
    return _context


class _State(dict):
    """Buffers and handles; releases the model (and its constraint sets)."""

    def __del__(self):
        if self.get("model"):
            try:
                self["ctx"].model_release(self["model"])
            except Exception:
                pass


def prepare(case, seed):
    ctx, dev, path = _ctx(), torch.device("cuda"), case["path"]
    s = _State(ctx=ctx, case=case)
    if path in ("hess", "grad", "pot", "host"):
        m = _table(case, seed)
        s["grid"] = _grid(case)
        shape = (6 if path == "hess" else 2, case["ny"], case["nx"])
        if path == "host":
            s["table"] = m
            s["out"] = torch.empty(shape, dtype=torch.float32, pin_memory=True)
            return s
        s["precision"] = api.LENS_FP64 if case["fp64"] else api.LENS_MIXED
        s["beta"] = _beta(seed)
        s["model"] = ctx.model_upload(m)
        s["out"] = torch.empty(shape, dtype=torch.float64 if case["fp64"] or path == "pot" else torch.float32, device=dev)
        return s
    m, cons, params = _fit_inputs(case, seed)
    P = case["P"]
    s["model"] = ctx.model_upload(m)
    s["cset"] = ctx.cset_create(s["model"], cons, (0, 1))
    s["params"] = torch.tensor(params, device=dev)
    s["chi2"] = torch.empty(P, dtype=torch.float64, device=dev)
    if path == "mcmc":
        s["sigma"] = torch.tensor(SIGMA, device=dev)
        s["step"] = torch.full((1,), 1 + seed % 1000, dtype=torch.int64, device=dev)
        s["scratch"] = torch.empty(16 * P, dtype=torch.float64, device=dev)
        s["accepted"] = torch.empty(P, dtype=torch.int32, device=dev)
        ctx.chi2_source(s["cset"], s["params"], P, case["variant"], s["chi2"])
        s["seed"] = seed
    elif path == "scaled" and case["nodes"]:
        ctx.cset_scaling_cache(s["cset"], *FT_RANGE, case["nodes"])
    elif path == "image":
        s["grid"] = inputs.grid(case["grid"])
        s["found"] = torch.empty((P, case["nsrc"]), dtype=torch.int32, device=dev)
    return s


def run(s):
    ctx, case = s["ctx"], s["case"]
    path = case["path"]
    if path == "hess":
        ctx.hessian_map(s["model"], s["grid"], case["dls"], s["precision"], s["out"])
        return {"alpha": s["out"][:2], "kappa_gamma": s["out"][2:5], "det": torch.reciprocal(s["out"][5])}
    if path == "grad":
        return ctx.grad_map(s["model"], s["grid"], case["dls"], s["precision"], s["out"])
    if path == "pot":
        return ctx.potential_map(s["model"], s["grid"], case["dls"], s["precision"], s["out"], beta=s["beta"])
    if path == "host":
        model = ctx.model_upload(s["table"])
        ctx.grad_map_host(model, s["grid"], case["dls"], api.LENS_MIXED, s["out"])
        ctx.wait()
        ctx.model_release(model)
        return s["out"]
    if path == "mcmc":
        ctx.mcmc_step_dev(s["cset"], s["params"], s["chi2"], case["P"], s["sigma"], TEMPERATURE, s["seed"], s["step"],
                          s["scratch"], s["accepted"], variant=case["variant"])
        return {"params": s["params"], "chi2": s["chi2"], "accepted": s["accepted"]}
    if path == "source":
        return ctx.chi2_source(s["cset"], s["params"], case["P"], case["variant"], s["chi2"])
    if path == "scaled":
        return ctx.chi2_source_scaled(s["cset"], s["params"], case["P"], case["variant"], s["chi2"])
    ctx.chi2_image(s["cset"], s["grid"], s["params"], case["P"], s["chi2"], s["found"])
    return {"chi2": s["chi2"], "found": s["found"]}


def _nimg(nsrc):
    with open(GOLDEN) as f:
        return json.load(f)["img_off"][nsrc]


def work(case):
    """Outputs and inputs once; operations as the sum over potentials is
    written: 65 a pair of node and potential with the Hessian, 45 without."""
    path, n = case["path"], case["n"]
    if path in ("hess", "grad", "pot", "host"):
        nodes = float(case["nx"]) * case["ny"]
        size = 8 if case["fp64"] or path == "pot" else 4
        return {"bytes": nodes * size * (6 if path == "hess" else 2) + 64.0 * n, "flops": nodes * n * (65 if path == "hess" else 45)}
    P, nimg = float(case["P"]), _nimg(case["nsrc"])
    hess = 45 if case["variant"] == 2 else 65
    if path == "image":  # the two varying potentials at the grid's nodes, the model at each image
        return {"bytes": P * (15 * 8 + 4 * case["nsrc"]) + 8.0 * case["grid"] ** 2,
                "flops": P * (45.0 * 2 * case["grid"] ** 2 + 45.0 * n * nimg)}
    each = 2 + (n - 2 if path == "scaled" and not case["nodes"] else 0)
    return {"bytes": P * 8 * (17 if path == "scaled" else 31 if path == "mcmc" else 15) + 72.0 * nimg, "flops": P * nimg * each * hess}


# ------------------------------------------------ the same results in 64 bits
def _potential(h, X, Y, hess, pot=False):
    """One potential's deflection (and kappa, gamma1, gamma2, or the
    potential) at X, Y, from the closed forms: dPIE as core minus cut."""
    type_, x0, y0, theta, eps, rc, rt, b0 = h
    dx, dy = X - x0, Y - y0
    if int(type_) != 0:
        r2 = dx * dx + dy * dy
        r2 = torch.where(r2 > 0, r2, torch.full_like(r2, math.inf))
        if int(type_) == 1:
            f = b0 / r2.sqrt()
            if pot:
                return b0 * (dx * dx + dy * dy).sqrt()
            k, g = 0.5 * f, 0.5 * f / r2
        else:
            f = b0 * b0 / r2
            if pot:
                return torch.where(torch.isfinite(r2), 0.5 * b0 * b0 * r2.log(), torch.zeros_like(r2))
            k, g = torch.zeros_like(f), f / r2
        out = [f * dx, f * dy]
        return out + [k, g * (dy * dy - dx * dx), -2.0 * g * dx * dy] if hess else out
    e1 = 1.0 + eps
    q, u = (1.0 - eps) / e1, 2.0 * math.sqrt(eps) / e1
    bq, sc, st = b0 * e1 * q, rc * e1, rt * e1
    c, s = math.cos(theta), math.sin(theta)
    x, y = c * dx + s * dy, c * dy - s * dx
    R = q * q * x * x + y * y
    pc, pt = (R + q * q * sc * sc).sqrt(), (R + q * q * st * st).sqrt()
    ux, uy = u * x, u * y
    ax = (bq / u) * (torch.atan(ux / (pc + sc)) - torch.atan(ux / (pt + st)))
    ay = (bq / u) * (torch.atanh(uy / (pc + q * q * sc)) - torch.atanh(uy / (pt + q * q * st)))
    if pot:
        lc, lt = ((pc + sc) ** 2 + ux * ux).log(), ((pt + st) ** 2 + ux * ux).log()
        return x * ax + y * ay - 0.5 * bq * (sc * lc - st * lt)
    out = [c * ax - s * ay, s * ax + c * ay]
    if hess:
        fc, ft = 1.0 / (pc * ((pc + sc) ** 2 + ux * ux)), 1.0 / (pt * ((pt + st) ** 2 + ux * ux))
        d = y * y - x * x
        g1 = 0.5 * bq * (fc * (d - u * u * sc * sc) - ft * (d - u * u * st * st))
        g2 = -bq * (fc - ft) * x * y
        c2, s2 = math.cos(2 * theta), math.sin(2 * theta)
        out += [0.5 * bq * (1.0 / pc - 1.0 / pt), c2 * g1 - s2 * g2, s2 * g1 + c2 * g2]
    return out


def _sums(table, X, Y, hess):
    total = None
    for h in table.tolist():
        v = _potential(h, X, Y, hess)
        total = v if total is None else [a + b for a, b in zip(total, v)]
    return total


def _exact_map(case, seed):
    m, g, path = _table(case, seed), _grid(case), case["path"]
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    i, j = (torch.arange(k, dtype=torch.float64, device=dev) for k in (case["nx"], case["ny"]))
    x = g["xmin"] + i * ((g["xmax"] - g["xmin"]) / (case["nx"] - 1))
    y = g["ymin"] + j * ((g["ymax"] - g["ymin"]) / (case["ny"] - 1))
    X, Y = x.expand(case["ny"], -1).contiguous(), y[:, None].expand(-1, case["nx"]).contiguous()
    r = case["dls"]
    if path == "pot":
        phi = torch.zeros_like(X)
        for h in m.tolist():
            phi += r * _potential(h, X, Y, False, pot=True)
        b = _beta(seed)
        return torch.stack([phi, 0.5 * ((X - b[0]) ** 2 + (Y - b[1]) ** 2) - phi])
    v = [r * t for t in _sums(m, X, Y, path == "hess")]
    if path != "hess":
        out = torch.stack(v)
        return out.cpu() if path == "host" else out
    return {"alpha": torch.stack(v[:2]), "kappa_gamma": torch.stack(v[2:]), "det": (1.0 - v[2]) ** 2 - v[3] ** 2 - v[4] ** 2}


def _chi2(m, cons, params, variant, dev):
    """Source-plane chi2 of every parameter set (14 or 16 parameters)."""
    x, y, sig = (torch.tensor(cons[k], device=dev) for k in ("x", "y", "sigma"))
    off = cons["img_off"]
    count = torch.tensor(np.diff(off), device=dev)
    src = torch.repeat_interleave(torch.arange(len(off) - 1, device=dev), count)
    ratio = torch.tensor(cons["dls_ds"], device=dev)[src]
    p = torch.tensor(params, device=dev)
    X, Y = x.expand(len(p), -1), y.expand(len(p), -1)
    if p.shape[1] == 16:
        total = [torch.zeros_like(X).contiguous() for _ in range(5)]
        fb, ft = p[:, 14:15], p[:, 15:16]
        for h in m[2:].tolist():
            v = _potential(h[:6] + [h[6] * ft, h[7] * fb], X, Y, True)
            for t, w in zip(total, v):
                t += w
    else:
        total = [t.expand(len(p), -1) for t in _sums(m[2:], x, y, True)]
    for k in range(2):
        x0, y0, eps, theta, rc, rt, b0 = (p[:, 7 * k + q][:, None] for q in range(7))
        total = [t + w for t, w in zip(total, _varying(x0, y0, eps, theta, rc, rt, b0, X, Y))]
    ax, ay, ka, g1, g2 = (ratio * t for t in total)
    bx, by = X - ax, Y - ay
    mean = lambda v: (torch.zeros(len(p), len(count), dtype=v.dtype, device=dev).index_add_(1, src, v) / count)[:, src]
    dx, dy = mean(bx) - bx, mean(by) - by
    if variant == 2:
        r2 = dx * dx + dy * dy
    else:
        a11, a22, a12 = 1.0 - ka - g1, 1.0 - ka + g1, -g2
        det = a11 * a22 - a12 * a12
        if variant == 1:
            r2 = (dx * dx + dy * dy) / det.abs()
        else:
            r2 = ((a22 * dx - a12 * dy) / det) ** 2 + ((a11 * dy - a12 * dx) / det) ** 2
    return (r2 / sig ** 2).sum(1)


def _varying(x0, y0, eps, theta, rc, rt, b0, X, Y):
    """_potential's dPIE with tensors for its parameters."""
    e1 = 1.0 + eps
    q, u = (1.0 - eps) / e1, 2.0 * eps.sqrt() / e1
    bq, sc, st = b0 * e1 * q, rc * e1, rt * e1
    c, s = theta.cos(), theta.sin()
    dx, dy = X - x0, Y - y0
    x, y = c * dx + s * dy, c * dy - s * dx
    R = q * q * x * x + y * y
    pc, pt = (R + q * q * sc * sc).sqrt(), (R + q * q * st * st).sqrt()
    ux, uy = u * x, u * y
    ax = (bq / u) * (torch.atan(ux / (pc + sc)) - torch.atan(ux / (pt + st)))
    ay = (bq / u) * (torch.atanh(uy / (pc + q * q * sc)) - torch.atanh(uy / (pt + q * q * st)))
    fc, ft = 1.0 / (pc * ((pc + sc) ** 2 + ux * ux)), 1.0 / (pt * ((pt + st) ** 2 + ux * ux))
    d = y * y - x * x
    g1 = 0.5 * bq * (fc * (d - u * u * sc * sc) - ft * (d - u * u * st * st))
    g2 = -bq * (fc - ft) * x * y
    c2, s2 = (2 * theta).cos(), (2 * theta).sin()
    return [c * ax - s * ay, s * ax + c * ay, 0.5 * bq * (1.0 / pc - 1.0 / pt), c2 * g1 - s2 * g2, s2 * g1 + c2 * g2]


def _philox(step, w, j, seed):
    """Words of Philox4x64-10 at counter (step, w, j, 0): numpy's generator
    advances its counter before it draws."""
    return np.random.Philox(counter=[step - 1, w, j, 0], key=[seed, 0]).random_raw(4)


def _exact_mcmc(case, seed):
    m, cons, p = _fit_inputs(case, seed)
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    step, P = 1 + seed % 1000, case["P"]
    unit = lambda v: ((v >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53
    raw = np.stack([np.concatenate([_philox(step, w, j, seed) for j in range(5)]) for w in range(P)])
    un = unit(raw)
    rad, ang = np.sqrt(-2.0 * np.log(un[:, 0:16:2])), 2.0 * np.pi * un[:, 1:16:2]
    z = np.stack([rad * np.cos(ang), rad * np.sin(ang)], axis=2).reshape(P, 16)[:, :14]
    prop = p + SIGMA * z
    c0, c1 = (_chi2(m, cons, v, case["variant"], dev).cpu().numpy() for v in (p, prop))
    for k in range(2):  # a proposal outside the dPIE domain is refused
        eps, rc, rt, b0 = (prop[:, 7 * k + q] for q in (2, 4, 5, 6))
        c1 = np.where((eps >= 0) & (eps < 1) & (rc > 0) & (rt > rc) & (b0 > 0), c1, np.nan)
    take = np.isfinite(c1) & (np.log(un[:, 16]) < -(c1 - c0) / (2.0 * TEMPERATURE))
    return {"params": np.where(take[:, None], prop, p), "chi2": np.where(take, c1, c0), "accepted": take.astype(np.int32)}


def exact(case, seed):
    path = case["path"]
    if path in ("hess", "grad", "pot", "host"):
        # over about 2e10 pairs it takes too long
        return _exact_map(case, seed) if float(case["nx"]) * case["ny"] * case["n"] < 2e10 else None
    if path == "image":  # a brute-force image search over 256 grids takes too long
        return None
    if path == "mcmc":
        return _exact_mcmc(case, seed)
    m, cons, params = _fit_inputs(case, seed)
    return _chi2(m, cons, params, case["variant"], torch.device("cuda" if torch.cuda.is_available() else "cpu"))
