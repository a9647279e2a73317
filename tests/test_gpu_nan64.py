"""FP64 operators on dense costs and grids give NaN where an input is NaN (a log-sum-exp with a NaN
term is NaN), as point clouds do, instead of leaving the input out: one NaN on the line, a line of
NaN alone, a NaN cost (its row and column only), lines of every kernel: chunks of 32 columns,
more than one block of 256 inputs, stored and plain grid kernels, the operator on one line."""
import numpy as np
import pytest
import torch

from paper_1607_05816_gb300 import uot as U

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def apply(geo, W, eps, transpose=False):
    w = torch.full_like(W, 1.0 / W.numel())
    return U.gibbs_log(geo, W, w, eps, transpose=transpose, precision=U.F64)


@pytest.mark.parametrize("n,m", [(5, 7), (40, 33), (9, 4200), (1300, 700)])
@pytest.mark.parametrize("eps", [1e-2, 1e-8])
@pytest.mark.parametrize("transpose", [False, True])
def test_dense_nan(n, m, eps, transpose):
    g = np.random.default_rng(n)
    C = g.random((n, m))
    nin = n if transpose else m
    W = 0.1 * g.normal(size=nin)
    for at in (slice(nin // 2, nin // 2 + 1), slice(None)):
        Wn = W.copy()
        Wn[at] = np.nan
        assert torch.isnan(apply(U.Geometry.dense(dev(C)), dev(Wn), eps, transpose)).all()
    Cn = C.copy()
    Cn[n // 3, m - 1] = np.nan
    out = apply(U.Geometry.dense(dev(Cn)), dev(W), eps, transpose)
    nan = torch.isnan(out).cpu().numpy()
    assert np.array_equal(np.flatnonzero(nan), [m - 1 if transpose else n // 3])


@pytest.mark.parametrize("shape", [(30,), (700,), (3, 40), (20, 300), (64, 64), (9, 10, 12)])
@pytest.mark.parametrize("eps", [1e-2, 1e-9])
@pytest.mark.parametrize("whole", [False, True])
def test_grid_nan(shape, eps, whole):
    n = int(np.prod(shape))
    geo = U.Geometry.grid([dev(np.linspace(0.0, 1.0, k)) for k in shape])
    W = np.zeros(n)
    W[slice(None) if whole else slice(n // 2, n // 2 + 1)] = np.nan
    assert torch.isnan(apply(geo, dev(W), eps)).all()
    assert torch.isneginf(apply(geo, dev(np.full(n, -np.inf)), eps)).all()
    p = dev(np.ones(n))
    w = dev(np.full(n, 1.0 / n))
    with pytest.raises(Exception):
        U.solve(geo, p, w, p, w, U.KL(0.5), U.KL(0.5), eps, max_iter=3, V0=dev(W))
