"""The FP64 grid pass (stored kernel times scaled inputs) at the edges of its tiles: one output
more or less than 64, inputs past a staged chunk of 256, axes and eps for which a tile needs 1, 2,
16 centres or none (plain log-sum-exp), unsorted and far-apart axes, empty lines, zero weights,
wide potentials, both directions, against the oracle's log-sum-exp.

Bound: an exponent is a sum of a few numbers, each rounded to 2^-53 of at most its own size, so
eps log K e^L is off by 2^-50 (max |L| + max cost / eps) eps, and the sum by nin 2^-53 more."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1607_05816_gb300 import uot as U

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def check(xs, ys, eps, amp, transpose, seed):
    g = np.random.default_rng(seed)
    shape_in = [len(a) for a in (xs if transpose else ys)]
    m = int(np.prod(shape_in))
    W = amp * g.normal(size=shape_in)
    W[g.random(shape_in) < 0.1] = -np.inf
    if len(shape_in) > 1 and shape_in[0] > 1:
        W[0] = -np.inf  # an empty line
    w = g.uniform(0.5, 1.5, size=shape_in) / m
    w[g.random(shape_in) < 0.05] = 0.0
    geo = U.Geometry.grid([dev(a) for a in xs], [dev(a) for a in ys])
    got = U.gibbs_log(geo, dev(W.ravel()), dev(w.ravel()), eps, transpose=transpose).cpu().numpy()
    with np.errstate(divide="ignore"):
        want = np.ravel(O.apply_K_log(O.Geometry("grid", xs=xs, ys=ys), W, np.log(w), eps, transpose=transpose))
    assert np.array_equal(np.isneginf(got), np.isneginf(want))
    f = np.isfinite(want)
    span = max(np.ptp(np.concatenate([a, b])) for a, b in zip(xs, ys)) ** 2
    fin = np.abs(W[np.isfinite(W)]).max()
    tol = 2.0 ** -49 * len(xs) * (fin + eps * 20 + span) + eps * sum(map(len, xs + ys)) * 2.0 ** -52
    assert np.all(np.abs(got[f] - want[f]) <= tol), (np.abs(got[f] - want[f]).max(), tol)


def axis(n, seed=None, scale=1.0):
    if seed is None:
        return scale * (np.arange(n) + 0.5) / n
    return scale * np.random.default_rng(seed).random(n)  # unsorted, uneven


@pytest.mark.parametrize("nx,ny,eps,scale", [
    ((9, 63), (8, 64), 1e-1, 1.0),
    ((8, 65), (9, 255), 1e-2, 1.0),
    ((10, 64), (9, 257), 3e-3, 1.0),    # two centres a tile
    ((8, 128), (8, 520), 1e-3, 1.0),
    ((40, 17), (30, 24), 1e-3, 1.0),    # many centres a tile
    ((30, 20), (20, 30), 1e-5, 1.0),    # out of reach: plain log-sum-exp
    ((20, 30), (20, 30), 1e-3, 30.0),   # costs far beyond the FP64 range
    ((12, 1), (1, 12), 1e-2, 1.0),
    ((5, 6, 70), (7, 4, 66), 2e-3, 1.0),
    ((300,), (3000,), 1e-2, 1.0),       # one line: no stored kernel
])
@pytest.mark.parametrize("uneven", [False, True])
@pytest.mark.parametrize("transpose", [False, True])
def test_f64_operator_at_tile_edges(nx, ny, eps, scale, uneven, transpose):
    xs = [axis(n, 7 + k if uneven else None, scale) for k, n in enumerate(nx)]
    ys = [axis(n, 70 + k if uneven else None, scale) for k, n in enumerate(ny)]
    check(xs, ys, eps, 0.3, transpose, 5)


def test_f64_operator_wide_potentials():
    """Potentials of 3000 eps: exponents far outside the FP64 range before the shift."""
    check([axis(20), axis(70)], [axis(20), axis(70)], 1e-3, 3.0, False, 9)


def test_f64_solve_through_eps_stages():
    """The stored kernels follow eps from stage to stage and from tiles with centres to tiles without."""
    g = np.random.default_rng(3)
    xs = [axis(12), axis(66)]
    n = 12 * 66
    dx = np.full((12, 66), 1.0 / n)
    p, q = g.uniform(0.5, 1.5, (12, 66)), g.uniform(0.5, 1.5, (12, 66))
    p[2:4] = 0.0
    ref = O.solve_log(O.Geometry("grid", xs=xs, ys=xs), dx, dx, p, q, O.KL(0.5), O.TV(0.3), 1e-4, max_iter=7,
                      eps_start=0.1, stages=5, iters_per_stage=3)
    geo = U.Geometry.grid([dev(a) for a in xs])
    for mode in (0, 2):
        Ug, Vg, _ = U.solve(geo, dev(p.ravel()), dev(dx.ravel()), dev(q.ravel()), dev(dx.ravel()), U.KL(0.5), U.TV(0.3),
                            1e-4, max_iter=7, eps_start=0.1, eps_stages=5, iters_per_stage=3, check_every=2,
                            launch_mode=mode)
        for got, want in ((Ug, ref["U"]), (Vg, ref["V"])):
            got, want = got.cpu().numpy(), np.ravel(want)
            f = np.isfinite(want)
            assert np.array_equal(np.isneginf(got), np.isneginf(want))
            assert np.max(np.abs(got[f] - want[f])) <= 1e-10 * max(1.0, np.max(np.abs(want[f])))
