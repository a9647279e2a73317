"""FP64 point-cloud solves at the limits of a launch grid's second dimension: more than 65535
blocks of 64 points on the X side (the rows of the stored kernel), and of 256 on the Y side.
Bar of the FP64 point-cloud solves."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1607_05816_gb300 import uot as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(64 * 65535 + 1, 3), (2, 256 * 65535 + 1)])
def test_more_blocks_than_a_second_dimension_holds(n, m):
    g = np.random.default_rng(5)
    x, y = g.random((n, 1)), g.random((m, 1))
    p, q = g.uniform(0.5, 1.5, n), g.uniform(0.5, 1.5, m)
    dx, dy = np.full(n, 1 / n), np.full(m, 1 / m)
    ref = O.solve_log(O.Geometry("points", x=x, y=y), dx, dy, p, q, O.KL(0.4), O.KL(0.4), 1e-2, max_iter=2,
                      check_every=2)
    dev = lambda a: torch.as_tensor(a, device="cuda")
    Ug, Vg, _ = U.solve(U.Geometry.points(dev(x), dev(y)), dev(p), dev(dx), dev(q), dev(dy), U.KL(0.4), U.KL(0.4), 1e-2,
                        max_iter=2, check_every=2)
    for got, want in ((Ug, ref["U"]), (Vg, ref["V"])):
        assert np.max(np.abs(got.cpu().numpy() - want)) <= 1e-10 * max(1.0, np.max(np.abs(want)))
