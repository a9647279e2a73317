"""FP64 dense rows with 1, 2, 4 and 16 warps per row, and rows short enough for registers, on both
sides of every line of that rule (multiples of the SM count in rows, of 32 columns times 8 chunks
a warp in columns): plain, steep and empty inputs, few and all terms counting.  Bar of the FP64
parity tests."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1607_05816_gb300 import synth
from paper_1607_05816_gb300 import uot as U

from test_gpu_parity import TOL, T, rel_err, to_np

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


def check(C, W, eps, transpose=False):
    nin = len(W)
    w = np.full(nin, 1.0 / nin)
    want = O.apply_K_log(O.Geometry("dense", C=C), W, np.log(w), eps, transpose=transpose)
    got = to_np(U.gibbs_log(U.Geometry.dense(T(C, U.F64)), T(W, U.F64), T(w, U.F64), eps, transpose, U.F64))
    assert np.array_equal(np.isneginf(got), np.isneginf(want))
    f = np.isfinite(want)
    assert rel_err(got[f], want[f]) <= TOL[U.F64]


@pytest.mark.parametrize("rows,over", [(0, 1), (1, 0), (1, 1), (2, 0), (2, 1), (8, 0), (8, 1)])
@pytest.mark.parametrize("nin", [1, 256, 257, 512, 513, 1024, 1025])
@pytest.mark.parametrize("eps", [1.0, 1e-5])
def test_rows_at_the_lines_of_the_rule(rows, over, nin, eps):
    n = rows * torch.cuda.get_device_properties(0).multi_processor_count + over
    g = synth.rng(n + nin)
    x, y = np.sort(g.uniform(size=n)), np.sort(g.uniform(size=nin))
    W = 0.8 * y
    if nin > 8:
        W[g.integers(0, nin, size=nin // 8)] = -np.inf
    check(O.sqdist(x, y), W, eps)


@pytest.mark.parametrize("n", [1, 2, 17, 152])
@pytest.mark.parametrize("nin", [4064, 4065, 9001])
@pytest.mark.parametrize("eps", [10.0, 1e-2, 1e-6])
def test_few_long_rows(n, nin, eps):
    g = synth.rng(n)
    C = O.sqdist(g.uniform(size=(n, 2)), g.uniform(size=(nin, 2)))
    C[:, 100:300] = np.inf
    check(C, 0.1 * g.normal(size=nin), eps)
    check(C.T.copy(), 0.1 * g.normal(size=nin), eps, transpose=True)
