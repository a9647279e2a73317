"""uot_solve_batch with every number of CTAs per problem, forced: parity with the oracle in each
dimension (idle CTAs, one block of 128 outputs per CTA, several, a ragged last one), the
translation step, the stop at a tolerance, and the schedule's own choice being one of them.
A forced size that cannot run is an error, so each case runs the size that it names.  Bar of
the batch parity tests: 1e-5."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1607_05816_gb300 import synth
from paper_1607_05816_gb300 import uot as U

from test_gpu_batch import make_divs, packed, rounded
from test_gpu_parity import rel_err

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


@pytest.fixture(params=[1, 2, 4, 8])
def ctas(request):
    U.force_batch_cluster(request.param)
    yield request.param
    U.force_batch_cluster(0)


@pytest.mark.parametrize("d", [1, 2, 3])
@pytest.mark.parametrize("size,translate", [((1, 140), False), ((120, 520), True), ((1020, 1100), False)])
def test_parity_at_every_cluster_size(ctas, d, size, translate):
    probs = synth.batch_points(nprob=4, size=size, d=d, seed=60 + d)
    sizes = [(len(pr["x"]), len(pr["y"])) for pr in probs]
    udivs, odivs = make_divs(probs, ["kl"] if translate else ["kl", "tv"])
    Ug, Vg, it, _, _ = U.solve_batch(sizes, udivs, d, *packed(probs), 0.02, max_iter=10, check_every=5,
                                     translate=translate)
    Ug, Vg = Ug.double().cpu().numpy(), Vg.double().cpu().numpy()
    assert it == [10] * 4
    xo = yo = 0
    for k, pr in enumerate(probs):
        og = O.Geometry("points", x=rounded(pr["x"]), y=rounded(pr["y"]))
        kw = dict(translate=True, check_every=5) if translate else {}
        r = O.solve_log(og, rounded(pr["dx"]), rounded(pr["dy"]), rounded(pr["p"]), rounded(pr["q"]), *odivs[k], 0.02,
                        max_iter=10, **kw)
        n, m = sizes[k]
        assert rel_err(Ug[xo:xo + n], r["U"]) <= 1e-5, k
        assert rel_err(Vg[yo:yo + m], r["V"]) <= 1e-5, k
        xo += n
        yo += m


def test_stop_at_tolerance_at_every_cluster_size(ctas):
    probs = synth.batch_points(nprob=3, size=(100, 900), d=2, seed=9)
    sizes = [(len(pr["x"]), len(pr["y"])) for pr in probs]
    udivs, _ = make_divs(probs, ["kl"])
    _, _, it, errs, info = U.solve_batch(sizes, udivs, 2, *packed(probs), 0.02, max_iter=20000, tol=1e-5, check_every=10)
    assert info["status"] == "UOT_OK" and max(errs) <= 1e-5 and max(it) < 20000
    assert all(i % 10 == 0 for i in it)


def test_few_large_problems_run_on_clusters():
    """The result is a cluster size's own, bit for bit, and not that of one CTA per problem."""
    probs = synth.batch_points(nprob=5, size=(1500, 2000), d=2, seed=3)
    sizes = [(len(pr["x"]), len(pr["y"])) for pr in probs]
    udivs, _ = make_divs(probs, ["kl"])
    args = packed(probs)

    def solve(ctas):
        U.force_batch_cluster(ctas)
        try:
            return U.solve_batch(sizes, udivs, 2, *args, 0.02, max_iter=10)[0]
        finally:
            U.force_batch_cluster(0)
    chosen = solve(0)
    assert not torch.equal(chosen, solve(1))
    assert any(torch.equal(chosen, solve(c)) for c in (2, 4, 8))


def test_invalid_sizes_are_refused():
    for c in (-1, 3, 16):
        with pytest.raises(Exception):
            U.force_batch_cluster(c)
