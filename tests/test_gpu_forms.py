"""J of every compiled form of the solve at the bin and line counts where its
tiling changes (bins per lane, tiles that end inside a line, bins of two lines
in one warp), against the FP64 oracle at the forms' accuracy."""
import numpy as np
import pytest

import synth
from helpers import j_rel_err

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (1, 32), (1, 33), (1, 64), (1, 65), (1, 100), (1, 128), (1, 129), (1, 200), (2, 16), (2, 33), (2, 64),
         (3, 21), (3, 43), (4, 40), (5, 13), (8, 9)]


@pytest.mark.parametrize("precision,order,tol", [("FP32", 2, 1e-4), ("FP32", 4, 1e-4), ("FP64", 2, 1e-10),
                                                 ("FP32_DT64", 2, 1e-4)])
@pytest.mark.parametrize("lines,bins", SIZES)
def test_forms_at_tile_edges(orc, lines, bins, precision, order, tol):
    import paper_2011_14998_gb300 as mgx

    m = synth.random_cloud(70, seed=lines * 1000 + bins, n_lines=lines, n_freq=bins, x_span=4.0, l_min=1, l_max=1)
    ctx = mgx.Context(0)
    try:
        mid = ctx.load(m)
        J = ctx.solve_J(mid, precision=getattr(mgx, "MGX_" + precision), I_bdy=0.05, order=order)
        rays = ctx.rays(mid)
    finally:
        ctx.close()
    Jo = orc.OracleModel(m, rays=rays).solve_J(orc.params(I_bdy=0.05, order=order))
    assert j_rel_err(J, Jo)[0] < tol
