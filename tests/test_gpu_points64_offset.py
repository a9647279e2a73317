"""FP64 point clouds whose coordinates have an offset large against their spread: FP32 copies move
the distances, and a solver's stored terms meet weights of e^150 and more.  Times near 1.7e9
(FP32 spacing 128) with X and Y on the two sides of a rounding boundary: true distances up to
20, FP32 distances 128.

Bar: an application rounds exponents of at most 400 a few times, 14 iterations (1e-10 relative,
as in the other FP64 point-cloud solves)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1607_05816_gb300 import uot as U

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def clouds(n, m, seed):
    g = np.random.default_rng(seed)
    base = 13281250 * 128.0  # 1.7e9, an FP32 number; base + 64 is the boundary
    return base + g.uniform(55.0, 63.9, (n, 1)), base + g.uniform(64.1, 75.0, (m, 1)), g


@pytest.mark.parametrize("swap", [False, True])
@pytest.mark.parametrize("n,m", [(200, 180), (33, 70)])
def test_offset_clouds_with_a_far_start(n, m, swap):
    x, y, g = clouds(n, m, n)
    if swap:
        x, y = y, x
        n, m = m, n
    eps, lam = 26.0, 13.0
    p, q = g.uniform(0.5, 1.5, n), g.uniform(0.5, 1.5, m)
    dx, dy = np.full(n, 1 / n), np.full(m, 1 / m)
    V0 = eps * g.uniform(-170.0, -130.0, m)  # the next V lies 120 eps above it
    ref = O.solve_log(O.Geometry("points", x=x, y=y), dx, dy, p, q, O.KL(lam), O.KL(lam), eps, max_iter=14,
                      check_every=5, V0=V0)
    Ug, Vg, _ = U.solve(U.Geometry.points(dev(x), dev(y)), dev(p), dev(dx), dev(q), dev(dy), U.KL(lam), U.KL(lam), eps,
                        max_iter=14, check_every=5, V0=dev(V0))
    for got, want in ((Ug, ref["U"]), (Vg, ref["V"])):
        got = got.cpu().numpy()
        assert np.isfinite(got).all()
        assert np.max(np.abs(got - want)) <= 1e-10 * max(1.0, np.max(np.abs(want)))
