"""FP64 grid passes at every cut of a tile's 64 outputs into blocks (1 to 16, and none: the plain
log-sum-exp), on axes of ragged sizes, unsorted and uneven: the cut depends on eps, so eps runs
over the range on which each appears.  Bar of the FP64 parity tests."""
import numpy as np
import pytest

import oracle as O
from paper_1607_05816_gb300 import uot as U

from test_gpu_parity import TOL, T, rel_err, to_np

pytestmark = pytest.mark.gpu

REACH = 320.0


def cut(x, y, eps):
    """Blocks of the first tile of outputs x for inputs y (0: none fits), as the kernel documents them."""
    x = x[:64]
    for sub in (1, 2, 4, 8, 16):
        w = 64 // sub
        ok = True
        for s in range(0, len(x), w):
            b = x[s:s + w]
            c = 0.5 * (b.min() + b.max())
            d, D = max(b.max() - c, c - b.min()), np.abs(c - y).max()
            ok = ok and (d * d + 2 * d * D) / eps <= REACH
        if ok:
            return sub
    return 0


def axis(n, kind, g):
    x = np.linspace(0.0, 1.0, n) if kind == "even" else np.sort(g.uniform(size=n))
    return x[::-1].copy() if kind == "reversed" else x


@pytest.mark.parametrize("n,m,kind", [(64, 64, "even"), (61, 70, "uneven"), (130, 33, "reversed"), (5, 9, "even")])
def test_every_cut(n, m, kind):
    g = np.random.default_rng(n)
    x, y = axis(n, kind, g), axis(m, "even", g)
    z = np.linspace(0.0, 1.0, 8)  # eight lines: the stored kernel is used
    W = 0.05 * g.normal(size=8 * m)
    w = np.full(8 * m, 1 / (8 * m))
    seen = set()
    for eps in np.geomspace(1e-2, 1e-5, 19):
        seen.add(cut(x, y, eps))
        geo = U.Geometry.grid([T(z, U.F64), T(x, U.F64)], [T(z, U.F64), T(y, U.F64)])
        got = to_np(U.gibbs_log(geo, T(W, U.F64), T(w, U.F64), float(eps), precision=U.F64))
        cost = O.Geometry("dense", C=((z[:, None, None, None] - z[None, None, :, None]) ** 2
                                      + (x[None, :, None, None] - y[None, None, None, :]) ** 2).reshape(8 * n, 8 * m))
        assert rel_err(got, O.apply_K_log(cost, W, np.log(w), float(eps))) <= TOL[U.F64]
    if n >= 61 and kind != "uneven":
        assert seen >= {1, 2, 4, 8, 16, 0}
