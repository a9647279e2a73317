"""FP32 point clouds with few outputs and many inputs: the chunks' partial sums are merged by a warp
per output from 64 chunks on and up to 32 outputs per SM, by a thread beyond.  Both sides of
both lines against the oracle, with sums that underflow the carried shift (recomputed by the
warp), empty inputs and a carried state.  Bar of the FP32 parity tests."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1607_05816_gb300 import uot as U

from test_gpu_parity import rel_err

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


def f32(a):
    return np.asarray(a, dtype=np.float32).astype(np.float64)


def dev(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float32), device="cuda")


@pytest.mark.parametrize("n,m,d", [(1, 62 * 1024, 2), (1, 70000, 2), (3, 70000, 1), (5, 70000, 3), (33, 66000, 2),
                                   (131, 200000, 2)])
@pytest.mark.parametrize("eps", [1e-1, 1e-3])
def test_operator_with_few_outputs(n, m, d, eps):
    g = np.random.default_rng(n + m)
    x, y = f32(g.random((n, d))), f32(g.random((m, d)))
    W = f32(0.1 * g.normal(size=m))
    W[::5] = -np.inf
    w = f32(np.full(m, 1 / m))
    got = U.gibbs_log(U.Geometry.points(dev(x), dev(y)), dev(W), dev(w), eps, precision=U.F32).double().cpu().numpy()
    want = O.apply_K_log(O.Geometry("points", x=x, y=y), W, np.log(w), eps)
    assert rel_err(got, want) <= 1e-5


@pytest.mark.parametrize("over", [0, 1])
def test_line_of_outputs(over):
    n, m = 32 * torch.cuda.get_device_properties(0).multi_processor_count + over, 70000
    g = np.random.default_rng(1)
    x, y = g.random((n, 2)), g.random((m, 2))
    W = 0.1 * g.normal(size=m)
    w = np.full(m, 1 / m)
    got = U.gibbs_log(U.Geometry.points(dev(x), dev(y)), dev(W), dev(w), 1e-2, precision=U.F32).double().cpu().numpy()
    at = np.r_[0:40, n - 40:n]
    want = O.apply_K_log(O.Geometry("points", x=f32(x)[at], y=f32(y)), f32(W), np.log(f32(w)), 1e-2)
    assert rel_err(got[at], want) <= 1e-5


@pytest.mark.parametrize("stages", [0, 4])
def test_solve_with_few_outputs(stages):
    g = np.random.default_rng(2)
    n, m = 40, 70000
    x, y = f32(g.random((n, 2))), f32(g.random((m, 2)))
    p, q = f32(g.uniform(0.5, 1.5, n)), f32(g.uniform(0.5, 1.5, m))
    q[::3] = 0.0
    dx, dy = f32(np.full(n, 1 / n)), f32(np.full(m, 1 / m))
    kw = dict(max_iter=6, check_every=3, eps_start=0.5 if stages else None, iters_per_stage=2)
    r = O.solve_log(O.Geometry("points", x=x, y=y), dx, dy, p, q, O.KL(0.4), O.KL(0.4), 2e-3, stages=stages or 10, **kw)
    Ug, Vg, _ = U.solve(U.Geometry.points(dev(x), dev(y)), dev(p), dev(dx), dev(q), dev(dy), U.KL(0.4), U.KL(0.4), 2e-3,
                        precision=U.F32, eps_stages=stages or 10, **kw)
    assert rel_err(Ug.double().cpu().numpy(), r["U"]) <= 1e-5
    assert rel_err(Vg.double().cpu().numpy(), r["V"]) <= 1e-5
