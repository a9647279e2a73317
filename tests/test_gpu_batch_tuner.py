"""The batch tuner's sample: eight problems per SM (all of a smaller batch), so that both CTA sizes
work through a queue, and the 8-warp CTA kept unless the other is more than 3% faster."""
import re

import pytest
import torch

from paper_1607_05816_gb300 import synth
from paper_1607_05816_gb300 import uot as U

from test_gpu_batch import make_divs, packed

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nprob,size", [(2000, (20, 61)), (700, (20, 62))])
def test_sample_and_choice(nprob, size):
    probs = synth.batch_points(nprob=nprob, size=size, d=2, seed=4)
    sizes = [(len(pr["x"]), len(pr["y"])) for pr in probs]
    udivs, _ = make_divs(probs, ["kl"])
    U.solve_batch(sizes, udivs, 2, *packed(probs), 0.02, max_iter=2)
    row = next(m for m in map(re.compile(r"dev\d+ batch d=2 nmax=(\d+) mmax=(\d+) sample=(\d+) -> warps=(\d+); "
                                         r"8:([\d.]+)ms 16:([\d.]+)ms").match, U.autotune_table().splitlines())
               if m and int(m.group(1)) == size[1])
    sample, warps, t8, t16 = int(row.group(3)), int(row.group(4)), float(row.group(5)), float(row.group(6))
    assert sample == min(nprob, 8 * torch.cuda.get_device_properties(0).multi_processor_count)
    if abs(t8 / t16 - 1.03) > 0.05:  # (the table has three decimals)
        assert warps == (16 if t8 > 1.03 * t16 else 8)
