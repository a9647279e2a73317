"""GPU parity of uot_solve_batch where clusters of CTAs share a problem: few or
uneven problems, with the schedule's own choice of the cluster size.

Sizes around the edges of the split: one block of 128 outputs (seven idle CTAs
in a cluster of 8), as many blocks as CTAs, one more, 16 warps' worth of blocks
per CTA, and the largest problem.  Bar of the batch parity tests: 1e-5."""
import numpy as np
import pytest

import oracle as O
from paper_1607_05816_gb300 import synth
from paper_1607_05816_gb300 import uot as U

from test_gpu_batch import make_divs, packed, rounded
from test_gpu_parity import rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,size,nprob,iters,translate", [
    (2, (1, 129), 5, 20, False), (2, (1020, 1030), 4, 8, False), (3, (250, 1300), 6, 6, False),
    (1, (300, 2100), 3, 6, False), (2, (3072, 3072), 1, 2, False), (2, (100, 900), 5, 20, True),
    (2, (60, 700), 330, 4, False)])
def test_batch_cluster_parity(d, size, nprob, iters, translate):
    probs = synth.batch_points(nprob=nprob, size=size, d=d, seed=140 + d + size[0])
    sizes = [(len(pr["x"]), len(pr["y"])) for pr in probs]
    udivs, odivs = make_divs(probs, ["kl"] if translate else ["kl", "tv"])
    args = packed(probs)
    eps = 0.02
    Ug, Vg, it, errs, _ = U.solve_batch(sizes, udivs, d, *args, eps, max_iter=iters, check_every=5,
                                        translate=translate)
    Ug, Vg = Ug.double().cpu().numpy(), Vg.double().cpu().numpy()
    xo = yo = 0
    for k, pr in enumerate(probs):
        n, m = sizes[k]
        assert it[k] == iters and np.isfinite(errs[k])
        if k % max(1, nprob // 6) == 0:
            og = O.Geometry("points", x=rounded(pr["x"]), y=rounded(pr["y"]))
            kw = dict(translate=True, check_every=5) if translate else {}
            r = O.solve_log(og, rounded(pr["dx"]), rounded(pr["dy"]), rounded(pr["p"]), rounded(pr["q"]), *odivs[k],
                            eps, max_iter=iters, **kw)
            assert rel_err(Ug[xo:xo + n], r["U"]) <= 1e-5, k
            assert rel_err(Vg[yo:yo + m], r["V"]) <= 1e-5, k
        xo += n
        yo += m


def test_batch_cluster_stops_at_tolerance():
    """Every CTA of a cluster takes the same stop decision; a side without mass is answered."""
    probs = synth.batch_points(nprob=3, size=(200, 1500), d=2, seed=9)
    sizes = [(len(pr["x"]), len(pr["y"])) for pr in probs]
    udivs, _ = make_divs(probs, ["kl"])
    x, p, dx, y, q, dy = packed(probs)
    Ug, Vg, it, errs, info = U.solve_batch(sizes, udivs, 2, x, p, dx, y, q, dy, 0.02, max_iter=20000, tol=1e-6,
                                           check_every=10)
    assert info["status"] == "UOT_OK" and max(errs) <= 1e-6 and max(it) < 20000
    q0 = q.clone()
    q0[:sizes[0][1]] = 0.0
    Ug, Vg, _, _, _ = U.solve_batch(sizes, udivs, 2, x, p, dx, y, q0, dy, 0.02, max_iter=5)
    assert bool((Vg[:sizes[0][1]] == -np.inf).all()) and bool(Ug[sizes[0][0]:].isfinite().all())
