"""uot_set_stored_kernel_limit: with a limit below its kernel a FP64 point-cloud solve evaluates its
terms on the fly (fewer kernels a pass: no column merge) and returns the same to rounding; the
default stores it.  Bar of the FP64 point-cloud solves."""
import numpy as np
import pytest
import torch

from paper_1607_05816_gb300 import uot as U

pytestmark = pytest.mark.gpu


def test_limit_of_the_stored_kernel():
    g = np.random.default_rng(1)
    n, m, its = 300, 201, 12
    dev = lambda a: torch.as_tensor(a, device="cuda")
    geo = U.Geometry.points(dev(g.random((n, 2))), dev(g.random((m, 2))))
    p, q = dev(g.uniform(0.5, 1.5, n)), dev(g.uniform(0.5, 1.5, m))
    dx, dy = dev(np.full(n, 1 / n)), dev(np.full(m, 1 / m))

    def solve(limit):
        was = U.set_stored_kernel_limit(limit)
        try:
            before = U.launch_count()
            out = U.solve(geo, p, dx, q, dy, U.KL(0.5), U.KL(0.5), 1e-2, max_iter=its, check_every=its)[:2]
            return out, U.launch_count() - before
        finally:
            assert U.set_stored_kernel_limit(was) == limit
    need = 8 * n * (m + 1)  # rows of an even length
    assert U.set_stored_kernel_limit(-1) == 4 << 30
    stored, with_kernel = solve(need)
    fly, without = solve(need - 1)
    assert with_kernel - without == its  # a column pass is three kernels, a pass on the fly two
    assert solve(0)[1] == without
    for a, b in zip(stored, fly):
        assert float((a - b).abs().max()) <= 1e-10
