"""What the speed of this framework is measured on: calls of its public entry points, as a
user's program makes them, over the sizes of its own configurations, tests and benchmark.

Every iteration runs a fixed number of times (tol = 0) unless the case says otherwise, so
that two builds do the same work.  Inputs come from paper_1607_05816_gb300.synth, made from
the seed alone.  `exact` restates each call in plain torch FP64 on the inputs as rounded to
the call's precision.
"""
import math

import numpy as np
import torch

from paper_1607_05816_gb300 import synth, uot, warmstart

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # one application of the log-domain Gibbs operator to a 1-D density, in the default
        # precision: the smallest call a program makes (its own loop around the operator)
        dict(name="operator_1d_f64", kind="operator", precision="f64", sizes="256", eps=1e-2, transpose=False),
        # the headline: a 256 x 256 image pair with the paper's eps-scaling, FP32, graph blocks
        dict(name="grid_256_f32", kind="grid", precision="f32", H=256, W=256, F1="kl:0.5", F2="kl:0.5", eps=1e-3,
             stages=10, stage_iters=20, iters=200, check_every=20, launch_mode=2),
        # the same problem in the default precision (the reference results of a study)
        dict(name="grid_256_f64", kind="grid", precision="f64", H=256, W=256, F1="kl:0.5", F2="kl:0.5", eps=1e-3,
             stages=10, stage_iters=1, iters=10, check_every=10, launch_mode=0),
        # time to a 1e-6 violation confirmed in FP64, with the translation step: a production solve
        dict(name="grid_256_to_tol", kind="grid_tol", H=256, W=256, lam=0.5, eps=1e-3, stages=10, stage_iters=100,
             check_every=20),
        # colour clouds of 20000 points each, FP32, the cost never stored
        dict(name="points_20000_f32", kind="points", precision="f32", n=20000, m=20000, d=3, F1="kl:0.1",
             F2="kl:0.1", eps=1e-3, stages=10, stage_iters=2, iters=20),
        # uneven 2-D clouds of a few thousand points in the default precision, with the primal,
        # the dual and the gap of the result
        dict(name="points_3001_f64", kind="points", precision="f64", n=3001, m=2477, d=2, F1="kl:0.5", F2="kl:0.5",
             eps=1e-2, stages=0, stage_iters=0, iters=20),
        # many small uneven problems in one call
        dict(name="batch_512", kind="batch", count=512, lo=64, hi=2048, eps=1e-2, iters=50),
        # the KL barycenter of 32 images
        dict(name="barycenter_32x128", kind="barycenter", K=32, H=128, W=128, bary="kl:1.0", eps=2e-3, iters=100),
        # two steps of the tumor growth flow on the paper's 3000 samples (a dense FP64 cost)
        dict(name="wf_flow_3000_f64", kind="wf", n=3000, species=1, eps=1e-8, tau=0.006, steps=2, iters=100),
        # colour transfer between two photographs of an odd size on the paper's bins (3-D grid)
        dict(name="color_427x640", kind="color", H=427, W=640, bins="64,32,32", lam=0.03, eps=2e-3, iters=300),
        # one training step of the warm-start network on a batch of 32 images
        dict(name="train_step_32", kind="train", N=32),
        # inference of that network and the batched solve from its potentials
        dict(name="warm_solve_32", kind="warm", N=32, lam=1.0, eps=1e-2, iters=60),
    ]


def draw(rng):
    def between(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def logu(lo, hi):
        return float("%.3g" % math.exp(rng.uniform(math.log(lo), math.log(hi))))

    def penalty():
        return rng.choice(["kl:%g" % logu(0.1, 2.0), "kl:%g" % logu(0.1, 2.0), "tv:%g" % logu(0.1, 1.0), "rg:0.7:1.3"])

    kind = rng.choice(["operator", "operator", "grid", "grid", "grid", "grid_tol", "points", "points", "batch",
                       "barycenter", "wf", "color", "train", "warm"])
    precision = rng.choice(["f32", "f64"])
    if kind == "operator":
        nd = rng.choice([1, 2, 3])
        hi = {1: 3000, 2: 256, 3: 64}[nd]
        sizes = ",".join(str(between(16, hi)) for _ in range(nd))
        return dict(kind=kind, precision=precision, sizes=sizes, eps=logu(1e-3, 1e-1), transpose=rng.random() < 0.5)
    if kind == "grid":
        big = precision == "f32"
        F1 = rng.choice([penalty(), penalty(), "eq"])
        return dict(kind=kind, precision=precision, H=between(24, 256), W=between(24, 256), F1=F1, F2=penalty(),
                    eps=logu(1e-3, 3e-2), stages=rng.choice([0, 10]), stage_iters=20 if big else 1,
                    iters=200 if big else 10, check_every=20 if big else 10, launch_mode=rng.choice([0, 2]))
    if kind == "grid_tol":
        return dict(kind=kind, H=between(48, 224), W=between(48, 224), lam=logu(0.3, 1.0), eps=logu(2e-3, 1e-2), stages=10,
                    stage_iters=40, check_every=20)
    if kind == "points":
        hi = 20000 if precision == "f32" else 3001
        return dict(kind=kind, precision=precision, n=between(400, hi), m=between(400, hi), d=rng.choice([2, 3]),
                    F1=penalty() if precision == "f32" else "kl:%g" % logu(0.1, 2.0), F2="kl:%g" % logu(0.1, 2.0),
                    eps=logu(1e-3, 2e-2), stages=rng.choice([0, 10]), stage_iters=1, iters=10)
    if kind == "batch":
        return dict(kind=kind, count=between(24, 512), lo=64, hi=between(256, 2048), eps=logu(5e-3, 5e-2), iters=50)
    if kind == "barycenter":
        return dict(kind=kind, K=between(3, 32), H=between(32, 128), W=between(32, 128),
                    bary=rng.choice(["kl:%g" % logu(0.3, 3.0), "eq"]), eps=logu(1e-3, 1e-2), iters=100)
    if kind == "wf":
        return dict(kind=kind, n=between(400, 3000), species=rng.choice([1, 2]), eps=logu(1e-8, 1e-5), tau=0.005,
                    steps=2, iters=40)
    if kind == "color":
        return dict(kind=kind, H=between(100, 640), W=between(100, 640),
                    bins=",".join(str(between(16, 64)) for _ in range(3)), lam=logu(0.01, 0.1), eps=logu(2e-3, 1e-2),
                    iters=100)
    if kind == "train":
        return dict(kind=kind, N=between(3, 32))
    return dict(kind=kind, N=between(3, 48), lam=logu(0.3, 3.0), eps=logu(3e-3, 5e-2), iters=60)


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------

def _dtype(case):
    return F64 if case.get("precision") == "f64" else torch.float32


def _precision(case):
    return uot.F64 if case.get("precision") == "f64" else uot.F32


def _ints(text):
    return [int(v) for v in text.split(",")]


def _div(text):
    f = text.split(":")
    return {"eq": lambda: uot.EQ(), "kl": lambda: uot.KL(float(f[1])), "tv": lambda: uot.TV(float(f[1])),
            "rg": lambda: uot.RG(float(f[1]), float(f[2]))}[f[0]]()


def _t(a, dtype=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device=DEV)


def _images(N, seed):
    """N pairs of 64 x 64 blob images with unit-order masses (the warm start's instances)."""
    inst = synth.warmstart_instances(N, seed=seed, group=N)
    return _t(inst["P"]), _t(inst["Q"]), inst


def prepare(case, seed):
    kind, dt = case["kind"], _dtype(case)
    s = {"case": case}
    if kind == "operator":
        sizes = _ints(case["sizes"])
        n = math.prod(sizes)
        axes = [_t(synth.grid_axis(k), dt) for k in sizes]
        g = torch.Generator(device=DEV).manual_seed(seed)
        # a potential of the size that a solve reaches, on cell weights
        s["W"] = 0.2 * torch.rand(n, generator=g, dtype=F64, device=DEV).to(dt) - 0.1
        s["w"] = torch.full((n,), 1.0 / n, dtype=dt, device=DEV)
        s["geo"] = uot.Geometry.grid(axes)
    elif kind in ("grid", "grid_tol"):
        d = synth.problem_grid2d(case["H"], case["W"], seed=seed)
        s["geo"] = uot.Geometry.grid([_t(a, dt) for a in d["xs"]], [_t(a, dt) for a in d["ys"]])
        s["p"], s["dx"], s["q"], s["dy"] = (_t(d[k], dt).ravel() for k in ("p", "dx", "q", "dy"))
    elif kind == "points":
        d = synth.problem_points(case["n"], case["m"], case["d"], seed=seed)
        s["geo"] = uot.Geometry.points(_t(d["x"], dt), _t(d["y"], dt))
        s["p"], s["dx"], s["q"], s["dy"] = (_t(d[k], dt) for k in ("p", "dx", "q", "dy"))
    elif kind == "batch":
        # the sizes belong to the case; the clouds, masses and penalties are the seed's
        g, gs = synth.rng(seed), synth.rng(case["count"])
        s["sizes"] = [tuple(int(v) for v in gs.integers(case["lo"], case["hi"] + 1, 2)) for _ in range(case["count"])]
        s["lams"] = [float(np.exp(g.uniform(np.log(0.05), np.log(5.0)))) for _ in s["sizes"]]
        s["divs"] = [(uot.KL(v), uot.KL(v)) for v in s["lams"]]
        for side, (pts, dens, wgt) in enumerate((("x", "p", "dx"), ("y", "q", "dy"))):
            ns = [nm[side] for nm in s["sizes"]]
            s[pts] = _t(np.concatenate([synth.mixture_points(g, n, 2, int(g.integers(1, 5))) for n in ns]))
            s[dens] = _t(np.concatenate([np.full(n, g.uniform(0.5, 2.0)) for n in ns]))
            s[wgt] = _t(np.concatenate([np.full(n, 1.0 / n) for n in ns]))
    elif kind == "barycenter":
        d = synth.barycenter_images(case["K"], case["H"], case["W"], seed=seed)
        s["geo"] = uot.Geometry.grid([_t(a) for a in d["xs"]])
        s["P"], s["dx"] = _t(d["P"].reshape(case["K"], -1)), _t(d["dx"]).ravel()
        s["alpha"] = [1.0 / case["K"]] * case["K"]
    elif kind == "wf":
        x, dx, P0 = synth.tumor_densities(case["n"], case["species"], seed=seed)
        s["geo"] = uot.Geometry.dense(uot.wf_cost(_t(x, F64), _t(x, F64), math.pi / 2))
        s["x"], s["dx"], s["P0"] = _t(x, F64), _t(dx, F64), _t(P0, F64)
    elif kind == "color":
        s["x"], s["y"] = (_t(synth.color_image(case["H"], case["W"], seed=2 * seed + k)) for k in (0, 1))
    elif kind in ("train", "warm"):
        N = case["N"]
        s["P"], s["Q"], inst = _images(N, seed)
        s["net"] = net = warmstart.WarmStartNetTC(seed=seed)
        if kind == "train":
            eps, lam = torch.as_tensor(inst["eps"], dtype=F64), torch.as_tensor(inst["lam"], dtype=F64)
            s["le"], s["ll"] = eps.log().float().to(DEV), lam.log().float().to(DEV)
            s["inv_lam"] = (1.0 / lam).float().to(DEV)
            s["feats"] = torch.empty(N * 4096, 64, dtype=torch.bfloat16, device=DEV)
            # potentials of the size that the solver's targets have: lambda times a smooth map
            s["U"] = (0.2 * lam.to(DEV).float()[:, None] * (s["P"] / (s["P"] + 1.0)).reshape(N, -1)).contiguous()
            s["V"] = (0.2 * lam.to(DEV).float()[:, None] * (s["Q"] / (s["Q"] + 1.0)).reshape(N, -1)).contiguous()
            # in the middle of training: moments from earlier batches
            g = torch.Generator(device=DEV).manual_seed(seed)
            net.t = 500
            for mo, ve in zip(net.m, net.v):
                for a, b in zip(mo, ve):
                    a.normal_(0.0, 1e-4, generator=g)
                    b.uniform_(0.5e-6, 2e-6, generator=g)
        else:
            axes = [_t(synth.grid_axis(64)) for _ in range(2)]
            s["geo"] = uot.Geometry.grid(axes)
            s["dx"] = torch.full((4096,), 1.0 / 4096, device=DEV)
    return s


# ---------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------

def _schedule(c):
    return dict(eps_start=0.1 if c["stages"] else None, eps_stages=c["stages"], iters_per_stage=c["stage_iters"])


def run(s):
    c = s["case"]
    kind, prec = c["kind"], _precision(c)
    if kind == "operator":
        return uot.gibbs_log(s["geo"], s["W"], s["w"], c["eps"], transpose=c["transpose"], precision=prec)
    if kind == "grid":
        U, V, _ = uot.solve(s["geo"], s["p"], s["dx"], s["q"], s["dy"], _div(c["F1"]), _div(c["F2"]), c["eps"],
                            precision=prec, max_iter=c["iters"], check_every=c["check_every"],
                            launch_mode=c["launch_mode"], **_schedule(c))
        return U, V
    if kind == "grid_tol":
        U, V, _ = uot.solve(s["geo"], s["p"], s["dx"], s["q"], s["dy"], uot.KL(c["lam"]), uot.KL(c["lam"]), c["eps"],
                            precision=prec, max_iter=20000, tol=1e-6, check_every=c["check_every"], launch_mode=2,
                            verify=True, translate=True, **_schedule(c))
        return U, V
    if kind == "points":
        F1, F2 = _div(c["F1"]), _div(c["F2"])
        U, V, _ = uot.solve(s["geo"], s["p"], s["dx"], s["q"], s["dy"], F1, F2, c["eps"], precision=prec,
                            max_iter=c["iters"], **_schedule(c))
        if c["precision"] == "f32":
            return {"U": U, "V": V}
        o = uot.objective(s["geo"], s["p"], s["dx"], s["q"], s["dy"], F1, F2, c["eps"], U, V, precision=prec)
        return {"U": U, "V": V, "primal": o["primal"], "dual": o["dual"]}
    if kind == "batch":
        U, V, _, _, _ = uot.solve_batch(s["sizes"], s["divs"], 2, s["x"], s["p"], s["dx"], s["y"], s["q"], s["dy"],
                                        c["eps"], max_iter=c["iters"])
        return U, V
    if kind == "barycenter":
        logh, U, V, _ = uot.barycenter_div(s["geo"], s["alpha"], s["P"], s["dx"], s["dx"], uot.EQ(), _div(c["bary"]),
                                           c["eps"], precision=prec, max_iter=c["iters"], check_every=50,
                                           launch_mode=2)
        return logh, U, V
    if kind == "wf":
        P, U, V, _ = uot.wf_flow(s["geo"], s["P0"], s["dx"], c["tau"], 1.0, 1.0, c["eps"], c["steps"],
                                 precision=uot.F64, iters=c["iters"])
        return P, U, V
    if kind == "color":
        img, T, _ = uot.color_transfer(s["x"], s["y"], uot.KL(c["lam"]), eps=c["eps"], iters=c["iters"],
                                       bins=tuple(_ints(c["bins"])))
        return img, T
    N, net = c["N"], s["net"]
    if kind == "train":
        uot.warmstart_features_nhwc(s["P"], s["Q"], s["le"], s["ll"], out=s["feats"])
        net.loss_dev.zero_()
        loss = net.train_step(s["feats"], s["U"], s["V"], s["inv_lam"], N, 64, 64, 3e-4)
        return {"loss": loss.float(), "params": net.params, "m": net.m}
    U0, V0 = net.predict(s["P"], s["Q"], [c["eps"]] * N, [c["lam"]] * N)
    lam = uot.KL(c["lam"])
    U, V, _ = uot.solve_many(s["geo"], s["P"].reshape(N, -1), s["dx"], s["Q"].reshape(N, -1), s["dx"], lam, lam,
                             c["eps"], precision=prec, max_iter=c["iters"], check_every=10, U0=U0, V0=V0,
                             launch_mode=2, translate=True)
    return U0, V0, U, V


# ---------------------------------------------------------------------------------------
# the work of one pass
# ---------------------------------------------------------------------------------------

def _grid_flops(sizes, batch=1):
    """One application of the separable operator: a multiply and an add per kernel entry."""
    n = math.prod(sizes)
    return 2.0 * batch * n * sum(sizes)


def _net_flops(pixels):
    """Forward pass of the network: 2 * 9 * Cin * Cout per pixel and layer."""
    return 18.0 * pixels * (4 * 128 + len(warmstart.TC_DILATIONS) * 128 * 128 + 128 * 2)


def work(case):
    c, kind = case, case["kind"]
    size = 8 if c.get("precision") == "f64" or kind == "wf" else 4
    if kind == "operator":
        sizes = _ints(c["sizes"])
        return {"bytes": 3.0 * size * math.prod(sizes), "flops": _grid_flops(sizes)}
    if kind in ("grid", "grid_tol"):
        n = c["H"] * c["W"]
        # to a tolerance: the iterations at the final eps depend on the data, some 200 of them
        its = c["stages"] * c["stage_iters"] + c.get("iters", 200)
        return {"bytes": 6.0 * size * n, "flops": 2 * its * _grid_flops([c["H"], c["W"]])}
    if kind == "points":
        its = c["stages"] * c["stage_iters"] + c["iters"]
        return {"bytes": size * (c["n"] + c["m"]) * (3.0 + c["d"]),
                "flops": 2.0 * its * c["n"] * c["m"] * (3 * c["d"] + 2)}
    if kind == "batch":
        mean = 0.5 * (c["lo"] + c["hi"])
        return {"bytes": 4.0 * 2 * c["count"] * mean * 5, "flops": 2.0 * c["count"] * c["iters"] * mean * mean * 8}
    if kind == "barycenter":
        n = c["H"] * c["W"]
        return {"bytes": 4.0 * n * (3 * c["K"] + 2), "flops": 2.0 * c["iters"] * _grid_flops([c["H"], c["W"]], c["K"])}
    if kind == "wf":
        its = c["steps"] * c["iters"] * c["species"]
        return {"bytes": 8.0 * c["n"] * c["n"], "flops": 2.0 * its * 2 * c["n"] * c["n"]}
    if kind == "color":
        bins = _ints(c["bins"])
        return {"bytes": 4.0 * (9 * c["H"] * c["W"] + 3 * math.prod(bins)),
                "flops": 2.0 * c["iters"] * _grid_flops(bins)}
    weights = 9.0 * (4 * 128 + len(warmstart.TC_DILATIONS) * 128 * 128 + 128 * 2)
    pixels = c["N"] * 4096
    if kind == "train":
        # the weights and both moments are read and written; the activations of every layer are
        # written by the forward pass and read by the backward pass (2 bytes, 128 channels)
        return {"bytes": 24.0 * weights + 2 * 2.0 * 128 * pixels * (1 + len(warmstart.TC_DILATIONS)),
                "flops": 3.0 * _net_flops(pixels)}
    return {"bytes": 2.0 * weights + 4.0 * 6 * pixels,
            "flops": _net_flops(pixels) + 2.0 * c["iters"] * _grid_flops([64, 64], c["N"])}


# ---------------------------------------------------------------------------------------
# the same calls in plain torch, 64 bits
# ---------------------------------------------------------------------------------------

def _lse(Z, dim):
    return torch.logsumexp(Z, dim)


def _sum_rows(L, M):
    """log sum_j e^{L[r, j] + M[i, j]} -> [r, i], in slices that fit the memory."""
    step = max(1, (1 << 27) // (M.shape[0] * M.shape[1]))
    return torch.cat([_lse(L[r:r + step, None, :] + M[None], 2) for r in range(0, L.shape[0], step)])


def _grid_op(L, xin, xout, eps):
    """log K e^L on a grid, one axis at a time; L [B, *shape of xin]."""
    for k, (a, b) in enumerate(zip(xin, xout)):
        M = -(b[:, None] - a[None, :]) ** 2 / eps
        L = L.movedim(k + 1, -1)
        shape = L.shape[:-1]
        L = _sum_rows(L.reshape(-1, len(a)), M).reshape(*shape, len(b)).movedim(-1, k + 1)
    return L


def _cloud_op(x, y, eps):
    """L -> log K e^L for point clouds (the cost formed in slices)."""
    step = max(1, (1 << 27) // len(y))

    def op(L):
        out = []
        for r in range(0, len(x), step):
            D = sum((x[r:r + step, None, k] - y[None, :, k]) ** 2 for k in range(x.shape[1]))
            out.append(_lse(L[None, :] - D / eps, 1))
        return torch.cat(out)
    return op


def _log(a):
    return torch.log(a.double())


def _prox(div, logp, S, eps):
    """Table 1 in log form."""
    f = div.split(":")
    u = torch.where(torch.isneginf(logp), logp, eps * logp - S)
    if f[0] == "kl":
        u = float(f[1]) / (float(f[1]) + eps) * u
    elif f[0] == "tv":
        u = u.clamp(-float(f[1]), float(f[1]))
    elif f[0] == "rg":
        u = torch.minimum(eps * math.log(float(f[2])) + u, (eps * math.log(float(f[1])) + u).clamp(min=0.0))
    return torch.where(torch.isneginf(S), S, u)


def _stages(c):
    if not c.get("stages") or 0.1 <= c["eps"]:
        return []
    rho = (0.1 / c["eps"]) ** (1.0 / c["stages"])
    return [(0.1 / rho ** k, c["stage_iters"]) for k in range(c["stages"])]


def _translate(U, V, lp, lq, lx, ly, lam):
    """The exact dual step along (U + c, V - c) for equal KL weights, per problem."""
    a = _lse(torch.where(torch.isneginf(lp), lp, lx + lp - U / lam), 1)
    b = _lse(torch.where(torch.isneginf(lq), lq, ly + lq - V / lam), 1)
    c = 0.5 * lam * (a - b)[:, None]
    return U + c, V - c


def _exact_grid(c, s):
    g = s["geo"]
    xs, ys = [a.double() for a in g.axes_x], [a.double() for a in g.axes_y]
    shx, shy = g.shape_x, g.shape_y
    lp, lq, lx, ly = (_log(s[k]).reshape(1, -1) for k in ("p", "q", "dx", "dy"))
    tol = c["kind"] == "grid_tol"
    d1, d2 = ("kl:%r" % c["lam"],) * 2 if tol else (c["F1"], c["F2"])
    U, V = torch.zeros_like(lp), torch.zeros_like(lq)
    for last, (eps, its) in [(False, st) for st in _stages(c)] + [(True, (c["eps"], c.get("iters", 20000)))]:
        for k in range(its):
            S = eps * _grid_op((V / eps + ly).reshape(1, *shy), ys, xs, eps).reshape(1, -1)
            Un = _prox(d1, lp, S, eps)
            check = (k + 1) % c["check_every"] == 0
            if tol and last and check:
                w, r, t = lx.exp(), ((U + S) / eps).nan_to_num(nan=-math.inf).exp(), ((Un + S) / eps).exp()
                done = float((w * (r - t).abs()).sum() / (w * t).sum()) <= 1e-6
            U = Un
            T = eps * _grid_op((U / eps + lx).reshape(1, *shx), xs, ys, eps).reshape(1, -1)
            V = _prox(d2, lq, T, eps)
            if tol and check:
                U, V = _translate(U, V, lp, lq, lx, ly, c["lam"])
                if last and done:
                    return U[0], V[0]
    return U[0], V[0]


def _exact_points(c, s):
    x, y = s["geo"].x.double(), s["geo"].y.double()
    lp, lq, lx, ly = (_log(s[k]) for k in ("p", "q", "dx", "dy"))
    U, V = torch.zeros_like(lp), torch.zeros_like(lq)
    for eps, its in _stages(c) + [(c["eps"], c["iters"])]:
        A, B = _cloud_op(x, y, eps), _cloud_op(y, x, eps)
        for _ in range(its):
            U = _prox(c["F1"], lp, eps * A(V / eps + ly), eps)
            V = _prox(c["F2"], lq, eps * B(U / eps + lx), eps)
    if c["precision"] == "f32":
        return {"U": U, "V": V}
    # KL penalties: the primal and the dual at (U, V)
    eps, wx, wy, p, q = c["eps"], s["dx"], s["dy"], s["p"], s["q"]
    r1, r2 = (U / eps + A(V / eps + ly)).exp(), (V / eps + B(U / eps + lx)).exp()
    mass, kmass = (wx * r1).sum(), (wx * A(ly).exp()).sum()
    lam1, lam2 = (float(c[k].split(":")[1]) for k in ("F1", "F2"))

    def kl(w, r, p):
        return (w * (r * torch.log(r / p) - r + p)).sum()
    ent = (wx * U * r1).sum() + (wy * V * r2).sum() - eps * mass + eps * kmass
    primal = lam1 * kl(wx, r1, p) + lam2 * kl(wy, r2, q) + ent
    dual = (-lam1 * (wx * p * torch.expm1(-U / lam1)).sum() - lam2 * (wy * q * torch.expm1(-V / lam2)).sum() -
            eps * (mass - kmass))
    return {"U": U, "V": V, "primal": float(primal), "dual": float(dual)}


def _exact_batch(c, s):
    eps, Us, Vs = c["eps"], [None] * len(s["sizes"]), [None] * len(s["sizes"])
    offs = np.cumsum([(0, 0)] + s["sizes"], axis=0)
    order = sorted(range(len(s["sizes"])), key=lambda k: s["sizes"][k])
    for at in range(0, len(order), 16):  # 16 problems of like sizes at a time, padded with empty points
        ks = order[at:at + 16]
        N, M = (max(s["sizes"][k][i] for k in ks) for i in (0, 1))

        def packed(name, side, width, fill):
            out = torch.full((len(ks), width) + s[name].shape[1:], fill, dtype=F64, device=DEV)
            for r, k in enumerate(ks):
                out[r, :s["sizes"][k][side]] = s[name][offs[k][side]:offs[k + 1][side]].double()
            return out
        x, y = packed("x", 0, N, 0.0), packed("y", 1, M, 0.0)
        lp, lq = (packed(*a).log() for a in (("p", 0, N, 0.0), ("q", 1, M, 0.0)))
        lx, ly = (packed(*a).log() for a in (("dx", 0, N, 0.0), ("dy", 1, M, 0.0)))
        lam = torch.tensor([s["lams"][k] for k in ks], dtype=F64, device=DEV)[:, None]
        f = lam / (lam + eps)
        C = -((x[:, :, None, :] - y[:, None, :, :]) ** 2).sum(3) / eps
        V = torch.zeros_like(lq)
        for _ in range(c["iters"]):
            U = f * (eps * lp - eps * _lse((V / eps + ly)[:, None, :] + C, 2))
            V = f * (eps * lq - eps * _lse((U / eps + lx)[:, :, None] + C, 1))
        for r, k in enumerate(ks):
            Us[k], Vs[k] = U[r, :s["sizes"][k][0]], V[r, :s["sizes"][k][1]]
    return torch.cat(Us), torch.cat(Vs)


def _exact_barycenter(c, s):
    axes = [a.double() for a in s["geo"].axes_x]
    K, eps, sh = c["K"], c["eps"], s["geo"].shape_x
    lp, lx = _log(s["P"]), _log(s["dx"])[None]
    alpha = torch.tensor(s["alpha"], dtype=F64, device=DEV)[:, None]
    V = torch.zeros_like(lp)
    for _ in range(c["iters"]):
        U = _prox("eq", lp, eps * _grid_op((V / eps + lx).reshape(K, *sh), axes, axes, eps).reshape(K, -1), eps)
        T = eps * _grid_op((U / eps + lx).reshape(K, *sh), axes, axes, eps).reshape(K, -1)
        if c["bary"] == "eq":
            h = (alpha * T).sum(0) / alpha.sum()
        else:
            e = eps + float(c["bary"].split(":")[1])
            h = e * (_lse(alpha.log() + T / e, 0) - alpha.sum().log())
        V = _prox(c["bary"], (h / eps)[None].expand_as(T), T, eps)
    return h, U, V


def _exact_wf(c, s):
    eps, cc = c["eps"], 1.0 - 2.0 * c["tau"]
    dist = (s["x"][:, None] - s["x"][None, :]).abs()
    M = torch.where(dist >= math.pi / 2, -math.inf, 2.0 * torch.log(torch.cos(dist))) / eps
    lx, logP, P = _log(s["dx"])[None], _log(s["P0"]), []
    for _ in range(c["steps"]):
        V = torch.zeros_like(logP)
        for _ in range(c["iters"]):
            U = _prox("kl:1.0", logP, eps * _sum_rows(V / eps + lx, M), eps)
            T = eps * _sum_rows(U / eps + lx, M.T.contiguous())
            tot = eps * _lse(T / eps, 0)
            V = torch.where(torch.isneginf(tot), -math.log(cc), (-tot / (1.0 + eps)).clamp(max=-math.log(cc)))
            V = V[None].expand_as(T)
        r2 = torch.where(torch.isneginf(T), T, (V + T) / eps)
        logP = r2 - r2.exp().sum(0).clamp(min=cc).log()
        P.append(logP.exp())
    return torch.stack(P), U, V.contiguous()


def _exact_color(c, s):
    bins, eps = _ints(c["bins"]), c["eps"]
    n = math.prod(bins)
    axes = [((torch.arange(k, dtype=F64, device=DEV) + 0.5) / k).float().double() for k in bins]

    def where(img):
        at = torch.zeros(img.numel() // 3, dtype=torch.int64, device=DEV)
        for a, k in enumerate(bins):  # the bin of a colour is decided in the image's own FP32
            at = at * k + (img.reshape(-1, 3)[:, a] * float(k)).floor().clamp(0, k - 1).long()
        return at
    bx, by = where(s["x"]), where(s["y"])
    lp, lq = (_log((torch.bincount(b, minlength=n).double() / len(b)).float())[None] for b in (bx, by))
    V = torch.zeros_like(lp)
    div = "kl:%r" % c["lam"]
    for _ in range(c["iters"]):
        U = _prox("eq", lp, eps * _grid_op((V / eps).reshape(1, *bins), axes, axes, eps).reshape(1, -1), eps)
        V = _prox(div, lq, eps * _grid_op((U / eps).reshape(1, *bins), axes, axes, eps).reshape(1, -1), eps)
    den = _grid_op((V / eps).reshape(1, *bins), axes, axes, eps).reshape(-1)
    own = torch.stack([a.reshape(-1) for a in torch.meshgrid(*axes, indexing="ij")], 1)
    T = []
    for k in range(3):
        num = _grid_op((V / eps + own[:, k].log()).reshape(1, *bins), axes, axes, eps).reshape(-1)
        T.append(torch.where(torch.isneginf(U[0]), own[:, k], (num - den).exp()))
    T = torch.stack(T, 1)
    return T[bx].reshape(s["x"].shape), T


def _shift(x, dy, dx):
    """x [N, H, W, C] moved so that entry (i, j) holds x at (i + dy, j + dx), zero outside."""
    H, W = x.shape[1:3]
    out = torch.zeros_like(x)
    i0, i1, j0, j1 = max(0, -dy), min(H, H - dy), max(0, -dx), min(W, W - dx)
    if i0 < i1 and j0 < j1:
        out[:, i0:i1, j0:j1] = x[:, i0 + dy:i1 + dy, j0 + dx:j1 + dx]
    return out


def _features(P, Q, le, ll):
    f = torch.stack([P.log().clamp(min=-30.0), Q.log().clamp(min=-30.0), le[:, None, None].expand_as(P),
                     ll[:, None, None].expand_as(P)], 3)
    return 0.25 * f


def _net_forward(net, params, x):
    acts = [x]
    for (w, b), (_, _, dil, leaky) in zip(params, net.layers):
        y = b + sum(_shift(x, (t // 3 - 1) * dil, (t % 3 - 1) * dil) @ w[:, :, t // 3, t % 3].T for t in range(9))
        x = torch.where(y < 0, 0.1 * y, y) if leaky else y
        acts.append(x)
    return acts


def _exact_train(c, s):
    net, N = s["net"], c["N"]
    params = [[t.double() for t in pr] for pr in net.params]
    acts = _net_forward(net, params, _features(s["P"].double(), s["Q"].double(), s["le"].double(), s["ll"].double()))
    target = (torch.stack([s["U"], s["V"]], 2).double() * s["inv_lam"].double()[:, None, None]).reshape(N, 64, 64, 2)
    diff = acts[-1] - target
    loss, g = (diff ** 2).mean(), 2.0 * diff / diff.numel()
    new_p, new_m = [None] * len(params), [None] * len(params)
    for li in range(len(params) - 1, -1, -1):
        w, _ = params[li]
        dil, x, gin = net.layers[li][2], acts[li], 0.0
        dw = torch.empty_like(w)
        for t in range(9):
            dy, dx = (t // 3 - 1) * dil, (t % 3 - 1) * dil
            dw[:, :, t // 3, t % 3] = g.reshape(-1, w.shape[0]).T @ _shift(x, dy, dx).reshape(-1, w.shape[1])
            gin = gin + _shift(g @ w[:, :, t // 3, t % 3], -dy, -dx)
        new_p[li], new_m[li] = [], []
        for p, d, m, v in zip(params[li], (dw, g.reshape(-1, w.shape[0]).sum(0)), net.m[li], net.v[li]):
            m, v = 0.9 * m.double() + 0.1 * d, 0.999 * v.double() + 0.001 * d * d
            new_m[li].append(m)
            new_p[li].append(p - 3e-4 * m / (1 - 0.9 ** 501) / ((v / (1 - 0.999 ** 501)).sqrt() + 1e-8))
        if li:
            g = gin * torch.where(x < 0, 0.1, 1.0)
    return {"loss": loss[None], "params": new_p, "m": new_m}


def _exact_warm(c, s):
    N, eps, lam = c["N"], c["eps"], c["lam"]
    full = torch.full((N,), 1.0, dtype=F64, device=DEV)
    x = _features(s["P"].double(), s["Q"].double(), full * math.log(eps), full * math.log(lam))
    out = lam * _net_forward(s["net"], [[t.double() for t in pr] for pr in s["net"].params], x)[-1]
    U0, V0 = (out[..., k].reshape(N, -1).contiguous() for k in (0, 1))
    axes = [a.double() for a in s["geo"].axes_x]
    lp, lq, lx = _log(s["P"]).reshape(N, -1), _log(s["Q"]).reshape(N, -1), _log(s["dx"])[None]
    V, div = V0, "kl:%r" % lam
    for k in range(c["iters"]):
        U = _prox(div, lp, eps * _grid_op((V / eps + lx).reshape(N, 64, 64), axes, axes, eps).reshape(N, -1), eps)
        V = _prox(div, lq, eps * _grid_op((U / eps + lx).reshape(N, 64, 64), axes, axes, eps).reshape(N, -1), eps)
        if (k + 1) % 10 == 0:
            U, V = _translate(U, V, lp, lq, lx, lx, lam)
    return U0, V0, U, V


def exact(case, seed):
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == "operator":
        axes, sizes = [a.double() for a in s["geo"].axes_x], _ints(case["sizes"])
        L = s["W"].double() / case["eps"] + _log(s["w"])
        return case["eps"] * _grid_op(L.reshape(1, *sizes), axes, axes, case["eps"]).reshape(-1)
    return {"grid": _exact_grid, "grid_tol": _exact_grid, "points": _exact_points, "batch": _exact_batch,
            "barycenter": _exact_barycenter, "wf": _exact_wf, "color": _exact_color, "train": _exact_train,
            "warm": _exact_warm}[kind](case, s)
