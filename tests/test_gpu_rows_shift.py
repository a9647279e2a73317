"""FP64 dense rows where the FP32 exponents that select a row's shift and terms are off by hundreds
to thousands (costs and potentials of 1e9 to 1e12 eps): the terms relative to the FP32 shift leave
the FP64 range, and the row's FP64 maximum has to take over.  Bar of the FP64 parity tests."""
import numpy as np
import pytest

import oracle as O
from paper_1607_05816_gb300 import synth
from paper_1607_05816_gb300 import uot as U

from test_gpu_parity import TOL, T, rel_err, to_np

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


@pytest.mark.parametrize("eps", [1e-9, 2e-10, 1e-10, 1e-12])
@pytest.mark.parametrize("n,m,kind", [(60, 900, "random"), (60, 900, "squared"), (9, 5000, "squared"),
                                      (1300, 64, "random"), (7, 33, "inf")])
@pytest.mark.parametrize("transpose", [False, True])
def test_rows_with_exponents_beyond_fp32(n, m, eps, kind, transpose):
    g = synth.rng(n + m)
    C = g.uniform(size=(n, m)) if kind != "squared" else O.sqdist(g.uniform(size=(n, 2)), g.uniform(size=(m, 2)))
    if kind == "inf":
        C[g.uniform(size=C.shape) < 0.5] = np.inf
        C[3] = np.inf
    nin = n if transpose else m
    W = 0.5 * g.normal(size=nin)
    w = np.full(nin, 1.0 / nin)
    want = O.apply_K_log(O.Geometry("dense", C=C), W, np.log(w), eps, transpose=transpose)
    got = to_np(U.gibbs_log(U.Geometry.dense(T(C, U.F64)), T(W, U.F64), T(w, U.F64), eps, transpose, U.F64))
    assert np.array_equal(np.isneginf(got), np.isneginf(want))
    f = np.isfinite(want)
    assert rel_err(got[f], want[f]) <= TOL[U.F64]


@pytest.mark.parametrize("eps", [1e-8, 1e-9, 1e-10])
@pytest.mark.parametrize("transpose", [False, True])
def test_rows_whose_exponents_cancel(eps, transpose):
    """Costs below zero whose part of the exponent cancels the potential's: the row's FP32 shift, from
    such a column, is off by its large parts, and must not hide columns with small ones."""
    n, m = 40, 640
    g = synth.rng(3)
    a = np.where(np.arange(m) < 320, g.uniform(0.5, 1.0, size=m), 0.0)
    C = -a[None, :] + eps * g.uniform(0.0, 30.0, size=(n, m)) + np.where(a > 0, 100.0 * eps, 0.0)[None, :]
    W = -a
    if transpose:
        C = C.T.copy()
    w = np.full(m, 1.0 / m)
    want = O.apply_K_log(O.Geometry("dense", C=C), W, np.log(w), eps, transpose=transpose)
    got = to_np(U.gibbs_log(U.Geometry.dense(T(C, U.F64)), T(W, U.F64), T(w, U.F64), eps, transpose, U.F64))
    # exponents of 1/eps are rounded to 2^-53 of their size, three times
    assert np.max(np.abs(got - want)) <= 4 * 2.0 ** -53 + 1e-10 * eps
