"""The tuner's choice among the FP32 grid tiles, read from its own table: a tile is chosen only if
none of the others was faster by more than the stated margins, and the warp-per-line kernel only
where it won by 5%."""
import re

import pytest
import torch

from paper_1607_05816_gb300 import uot as U

pytestmark = pytest.mark.gpu


def rows():
    for line in U.autotune_table().splitlines():
        m = re.match(r"dev\d+ lines=(\d+) nin=(\d+) nout=(\d+) batch=(\d+) -> ([^;]*);(.*)", line)
        if m:
            times = {k: float(v) for k, v in re.findall(r"(\S+?):(-?[\d.]+)us", m.group(6))}
            yield m.group(5), {k: v for k, v in times.items() if v > 0 and not k.startswith("blk")}


def test_choices_keep_their_margins():
    for shape, batch in (((93, 57), 20), ((57, 57), 20), ((48, 48), 32), ((40, 24), 16), ((64, 64), 17)):
        geo = U.Geometry.grid([torch.linspace(0, 1, k, device="cuda") for k in shape])
        n = shape[0] * shape[1]
        P = torch.ones(batch, n, device="cuda")
        w = torch.full((n,), 1.0 / n, device="cuda")
        U.solve_many(geo, P, w, P, w, U.KL(0.5), U.KL(0.5), 1e-2, precision=U.F32, max_iter=2)
    seen = 0
    for chosen, us in rows():
        if "line" not in us:
            continue
        others = min(v for k, v in us.items() if k != "line")
        seen += 1
        if chosen == "warp per line":
            assert 1.05 * us["line"] <= others + 0.02  # (the table has two decimals)
        else:
            assert 1.05 * us["line"] >= others - 0.02 or us["8x4"] <= 1.05 * us["line"] + 0.02
    assert seen >= 5
