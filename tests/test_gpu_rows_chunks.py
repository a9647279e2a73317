"""GPU parity of the FP64 dense rows by chunks of 32 columns, at the sizes and
inputs where a chunk test could drop a term that counts: rows of 1 to 33 chunks
and a remainder, more than 128 chunks (bounds beyond the prefetched ones), 8 and
24 rows per CTA, unsorted points, a steep potential (every bound loose, the
maximum chunks away from the largest one), terms of one row filling its list
several times, costs of +inf and below zero, inputs of -inf.  Bar of the FP64
parity tests."""
import numpy as np
import pytest

import oracle as O
from paper_1607_05816_gb300 import synth
from paper_1607_05816_gb300 import uot as U

from test_gpu_parity import TOL, T, rel_err, to_np

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


@pytest.mark.parametrize("n,m,eps,kind", [
    (1, 1, 1e-2, "plain"), (3, 31, 1e-3, "plain"), (40, 33, 1e-6, "steep"), (1300, 500, 1e-8, "steep"),
    (1300, 500, 1e-4, "shuffled"), (7, 4200, 1e-7, "steep"), (7, 4200, 10.0, "plain"), (1217, 97, 1e-3, "inf"),
    (60, 900, 1e-2, "negative"), (60, 900, 1e-5, "shuffled")])
@pytest.mark.parametrize("transpose", [False, True])
def test_chunked_rows_parity(n, m, eps, kind, transpose):
    g = synth.rng(n + m)
    x, y = np.sort(g.uniform(0, 1, size=n)), np.sort(g.uniform(0, 1, size=m))
    if kind == "shuffled":
        x, y = g.permutation(x), g.permutation(y)
    C = O.sqdist(x, y)
    if kind == "inf":
        C[np.abs(x[:, None] - y[None, :]) > 0.05] = np.inf
    if kind == "negative":
        C = C - 0.3 * g.uniform(size=C.shape)
    nin, at = (n, x) if transpose else (m, y)
    W = {"steep": 0.8 * at, "plain": 0.01 * g.normal(size=nin)}.get(kind, 0.1 * np.sin(9 * at))
    if nin > 8:
        W[g.integers(0, nin, size=nin // 8)] = -np.inf
    w = np.full(nin, 1.0 / nin)
    want = O.apply_K_log(O.Geometry("dense", C=C), W, np.log(w), eps, transpose=transpose)
    got = to_np(U.gibbs_log(U.Geometry.dense(T(C, U.F64)), T(W, U.F64), T(w, U.F64), eps, transpose, U.F64))
    assert np.array_equal(np.isneginf(got), np.isneginf(want))
    f = np.isfinite(want)
    if f.any():
        assert rel_err(got[f], want[f]) <= TOL[U.F64]
