"""FP64 point clouds (on-the-fly rows, the solvers' stored kernel and its column pass) against the
oracle at the edges of the kernels: one point, rows that are no multiple of a CTA's 8, odd column
counts, dimensions 1 to 8, tiny and large eps, coordinates far apart, inputs without mass, and
solves whose potentials move by more than 300 eps (the kernel is stored anew) or that start from
-inf.

Bound of one application: an exponent (L - |x-y|^2/eps) is rounded to 2^-53 of its size a few
times, and the sum to nin 2^-53."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1607_05816_gb300 import uot as U

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("n,m,d,eps,scale,amp", [
    (1, 1, 1, 1e-2, 1.0, 0.1),
    (7, 33, 1, 1e-3, 1.0, 0.5),
    (257, 129, 2, 1e-2, 1.0, 0.3),
    (64, 300, 3, 1e-3, 1.0, 1.0),
    (40, 50, 5, 1e-1, 1.0, 0.3),
    (33, 21, 8, 1e-1, 2.0, 0.3),
    (50, 70, 2, 1e-6, 1.0, 1.0),       # exponents of millions
    (50, 70, 2, 1e-5, 1e4, 1.0),       # exponents of 1e13
    (30, 40, 3, 1e-8, 1e5, 1.0),       # ... and of 1e18
    (20, 30, 2, 1e-30, 1.0, 1.0),
])
@pytest.mark.parametrize("transpose", [False, True])
def test_points64_operator(n, m, d, eps, scale, amp, transpose):
    g = np.random.default_rng(n + m)
    x, y = scale * g.random((n, d)), scale * g.random((m, d))
    k = n if transpose else m
    W = amp * g.normal(size=k)
    w = g.uniform(0.5, 1.5, size=k) / k
    if k > 10:
        W[::7] = -np.inf
        w[3] = 0.0
    geo = U.Geometry.points(dev(x), dev(y))
    got = U.gibbs_log(geo, dev(W), dev(w), eps, transpose=transpose).cpu().numpy()
    with np.errstate(divide="ignore"):
        want = O.apply_K_log(O.Geometry("points", x=x, y=y), W, np.log(w), eps, transpose=transpose)
    f = np.isfinite(want)
    assert np.array_equal(np.isneginf(got), np.isneginf(want))
    size = np.abs(W[np.isfinite(W)]).max() + d * scale ** 2 + 20 * eps
    assert np.all(np.abs(got[f] - want[f]) <= 2.0 ** -49 * size + eps * k * 2.0 ** -52)


def test_points64_keeps_nan_and_empty_lines():
    g = np.random.default_rng(1)
    x, y = g.random((20, 2)), g.random((31, 2))
    geo = U.Geometry.points(dev(x), dev(y))
    w = np.full(31, 1 / 31)
    W = np.zeros(31)
    W[5] = np.nan
    assert torch.isnan(U.gibbs_log(geo, dev(W), dev(w), 1e-2)).all()
    assert torch.isneginf(U.gibbs_log(geo, dev(np.full(31, -np.inf)), dev(w), 1e-2)).all()


@pytest.mark.parametrize("F1,F2", [("kl", "kl"), ("tv", "kl"), ("eq", "kl"), ("rg", "tv")])
@pytest.mark.parametrize("n,m,d,eps,stages", [(61, 50, 2, 1e-2, 0), (130, 131, 3, 1e-3, 4), (40, 77, 1, 1e-4, 3),
                                              (25, 30, 6, 5e-2, 0)])
def test_points64_solve_matches_oracle(F1, F2, n, m, d, eps, stages):
    g = np.random.default_rng(n)
    x, y = g.random((n, d)), g.random((m, d)) + 0.3
    p, q = g.uniform(0.5, 1.5, n), g.uniform(0.5, 1.5, m)
    p[2] = 0.0
    q[::9] = 0.0  # columns without mass once V is updated
    dx, dy = np.full(n, 1 / n), np.full(m, 1 / m)
    mk = lambda M, k: {"kl": M.KL(0.4), "tv": M.TV(0.3), "eq": M.EQ(), "rg": M.RG(0.7, 1.3)}[k]
    V0 = 2.0 * g.normal(size=m)  # up to thousands of eps from where it ends
    V0[4] = -np.inf
    for launch_mode, check in ((0, 5), (2, 3)):
        kw = {} if stages else dict(V0=V0)
        ref = O.solve_log(O.Geometry("points", x=x, y=y), dx, dy, p, q, mk(O, F1), mk(O, F2), eps, max_iter=14,
                          eps_start=0.1 if stages else None, stages=stages or 10, iters_per_stage=3,
                          check_every=check, **kw)
        kw = {} if stages else dict(V0=dev(V0))
        Ug, Vg, info = U.solve(U.Geometry.points(dev(x), dev(y)), dev(p), dev(dx), dev(q), dev(dy), mk(U, F1),
                               mk(U, F2), eps, max_iter=14, eps_start=0.1 if stages else None, eps_stages=stages or 10,
                               iters_per_stage=3, check_every=check, launch_mode=launch_mode, **kw)
        for got, want in ((Ug, ref["U"]), (Vg, ref["V"])):
            got = got.cpu().numpy()
            f = np.isfinite(want)
            assert np.array_equal(np.isneginf(got), np.isneginf(want))
            assert np.max(np.abs(got[f] - want[f])) <= 1e-10 * max(1.0, np.max(np.abs(want[f])))
        assert abs(info["marg_err"] - ref["err"]) <= 1e-9 * max(1e-3, ref["err"])
