"""FP32 grid passes that take four lines per CTA (131072 inputs and more over the
batch) against the oracle: line counts that leave a ragged last CTA, lines
shorter than a warp and longer than the registers hold, outputs beyond one tile,
empty lines, every tile shape with such a form.  Bar of the FP32 parity tests."""
import numpy as np
import pytest

import oracle as O
from paper_1607_05816_gb300 import synth
from paper_1607_05816_gb300 import uot as U

from test_gpu_parity import TOL, T, rel_err, round_geom, rounded, to_np

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


@pytest.mark.parametrize("tile", [0, 1, 4, 5])  # 8 and 4 warps, 4 and 2 outputs per lane
@pytest.mark.parametrize("sx,sy", [((3, 70), (1030, 300)), ((40, 30, 20), (72, 70, 28)), ((2, 600), (1025, 140))])
def test_four_line_tiles(tile, sx, sy):
    g = synth.rng(sum(sx))
    xs, ys = [synth.grid_axis(n) for n in sx], [synth.grid_axis(n) for n in sy]
    og = O.Geometry("grid", xs=xs, ys=ys)
    W = 0.1 * g.normal(size=sy)
    W.reshape(-1, sy[-1])[::11] = -np.inf  # empty lines of the first pass
    W, w = rounded(U.F32, W, np.full(sy, 1.0 / np.prod(sy)))
    geo = U.Geometry.grid([T(a, U.F32) for a in xs], [T(a, U.F32) for a in ys])
    U.force_grid_tile(tile)
    try:
        got = U.gibbs_log(geo, T(W, U.F32).ravel(), T(w, U.F32).ravel(), 0.02, False, U.F32)
    finally:
        U.force_grid_tile(-1)
    assert rel_err(to_np(got), O.apply_K_log(round_geom(og, U.F32), W, np.log(w), 0.02)) <= TOL[U.F32]


@pytest.mark.parametrize("tile", [1, 5])
def test_four_line_tiles_in_a_batched_solve(tile):
    """150 problems of 31 x 29: lines of one batch entry end inside a CTA; checked iterations."""
    g = synth.rng(3)
    B, sh = 150, (31, 29)
    xs = [synth.grid_axis(n) for n in sh]
    og = O.Geometry("grid", xs=xs, ys=xs)
    dx = np.full(sh, 1.0 / np.prod(sh))
    P, Q = g.uniform(0.5, 1.5, size=(B,) + sh), g.uniform(0.5, 1.5, size=(B,) + sh)
    P, Q, dx = rounded(U.F32, P, Q, dx)
    geo = U.Geometry.grid([T(a, U.F32) for a in xs], [T(a, U.F32) for a in xs])
    U.force_grid_tile(tile)
    try:
        Ug, Vg, info = U.solve_many(geo, T(P.reshape(B, -1), U.F32), T(dx, U.F32).ravel(), T(Q.reshape(B, -1), U.F32),
                                    T(dx, U.F32).ravel(), U.KL(0.5), U.KL(0.5), 0.02, precision=U.F32, max_iter=20,
                                    check_every=10)
    finally:
        U.force_grid_tile(-1)
    assert np.isfinite(info["marg_err"])
    for k in (0, 70, 149):
        r = O.solve_log(round_geom(og, U.F32), dx, dx, P[k], Q[k], O.KL(0.5), O.KL(0.5), 0.02, max_iter=20)
        assert rel_err(to_np(Ug[k]), r["U"]) <= TOL[U.F32]
        assert rel_err(to_np(Vg[k]), r["V"]) <= TOL[U.F32]
