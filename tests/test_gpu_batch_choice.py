"""The schedule's choice of CTAs per problem where it is known which is faster: as many equal
problems as SMs fill the GPU with one CTA each (two would share every SM and wait for each other),
half as many are faster on two.  The choice is read from the result's bits: each number of CTAs
sums in an order of its own."""
import pytest
import torch

from paper_1607_05816_gb300 import synth
from paper_1607_05816_gb300 import uot as U

from test_gpu_batch import make_divs, packed

pytestmark = pytest.mark.gpu


def runs(nprob, size):
    probs = synth.batch_points(nprob=nprob, size=(size, size), d=2, seed=11)
    sizes = [(size, size)] * nprob
    udivs, _ = make_divs(probs, ["kl"])
    args = packed(probs)

    def solve(warps=0, ctas=0):
        U.force_batch_warps(warps)
        U.force_batch_cluster(ctas)
        try:
            return U.solve_batch(sizes, udivs, 2, *args, 0.02, max_iter=5)[0]
        finally:
            U.force_batch_warps(0)
            U.force_batch_cluster(0)
    return solve


@pytest.mark.parametrize("share,size", [(1.0, 300), (1.0, 512), (2.0, 512)])
def test_problems_that_fill_the_gpu_take_one_cta(share, size):
    solve = runs(int(share * torch.cuda.get_device_properties(0).multi_processor_count), size)
    chosen = solve()
    assert any(torch.equal(chosen, solve(warps=w)) for w in (8, 16))
    assert not torch.equal(chosen, solve(ctas=2))


def test_half_as_many_take_two():
    solve = runs(torch.cuda.get_device_properties(0).multi_processor_count // 2, 512)
    assert torch.equal(solve(), solve(ctas=2))
