"""FP64 dense rows on 32-warp CTAs of eight rows: between four and eight rows per SM, up to 1280
columns in registers; both sides of those lines, with few and all terms counting, rows whose
exponents leave FP32's reach, and NaN.  Bar of the FP64 parity tests."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1607_05816_gb300 import synth
from paper_1607_05816_gb300 import uot as U

from test_gpu_parity import TOL, T, rel_err, to_np

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


def operator(C, W, eps):
    w = np.full(len(W), 1.0 / len(W))
    got = to_np(U.gibbs_log(U.Geometry.dense(T(C, U.F64)), T(W, U.F64), T(w, U.F64), eps, False, U.F64))
    return got, O.apply_K_log(O.Geometry("dense", C=C), W, np.log(w), eps)


@pytest.mark.parametrize("rows,over", [(4, 0), (4, 1), (5, 3), (8, 0), (8, 1)])
@pytest.mark.parametrize("nin", [1, 33, 1024, 1279, 1280, 1281])
@pytest.mark.parametrize("eps", [1.0, 1e-6, 1e-10])
def test_lines_of_the_rule(rows, over, nin, eps):
    n = rows * torch.cuda.get_device_properties(0).multi_processor_count + over
    g = synth.rng(n + nin)
    C = O.sqdist(np.sort(g.uniform(size=n)), np.sort(g.uniform(size=nin)))
    C[:, :nin // 7] = np.inf
    W = 0.3 * g.normal(size=nin)
    if nin > 8:
        W[g.integers(0, nin, size=nin // 8)] = -np.inf
    got, want = operator(C, W, eps)
    assert np.array_equal(np.isneginf(got), np.isneginf(want))
    f = np.isfinite(want)
    assert rel_err(got[f], want[f]) <= TOL[U.F64]


def test_nan_cost_and_input():
    n, nin = 5 * torch.cuda.get_device_properties(0).multi_processor_count, 900
    g = synth.rng(2)
    C, W = g.uniform(size=(n, nin)), np.zeros(nin)
    C[17, 400] = np.nan
    assert np.array_equal(np.flatnonzero(np.isnan(operator(C, W, 1e-2)[0])), [17])
    W[899] = np.nan
    assert np.isnan(operator(C, W, 1e-2)[0]).all()
