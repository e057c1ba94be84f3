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


@pytest.mark.parametrize("n,l_min,l_max", [(8, 0, 0), (27, 1, 1), (60, 0, 2), (300, 2, 2)])
@pytest.mark.parametrize("precision", ["FP32", "FP64"])
def test_pairs_dealt_to_several_warps(orc, n, l_min, l_max, precision):
    """Few origins: the pairs of an origin are solved by several warps.  J of the per-model and
    the batched call (alone and next to a larger model, which changes the share) is the same
    bit for bit, and the sum of solve_u over the pairs."""
    import paper_2011_14998_gb300 as mgx

    prec = getattr(mgx, "MGX_" + precision)
    m = synth.random_cloud(n, seed=n, n_lines=2, n_freq=20, l_min=l_min, l_max=l_max)
    # as many lines and bins as m: another bin count would take another compiled form in the batch
    big = synth.with_lines(synth.wind_model(3000, seed=1, n_freq=20, level=1), 2, 20)
    ctx = mgx.Context(0)
    try:
        mid, bid = ctx.load(m), ctx.load(big)
        J = ctx.solve_J(mid, precision=prec)
        alone = ctx.solve_J_batch([mid], precision=prec)[0].cpu().numpy()
        both = ctx.solve_J_batch([bid, mid], precision=prec)
        u = ctx.solve_u(mid, 0, n, precision=prec)
        w = 2.0 / (12.0 * 4.0 ** (ctx.rays(mid) >> 28))
        rays = ctx.rays(mid)
        Jb = ctx.solve_J(bid, precision=prec)
    finally:
        ctx.close()
    np.testing.assert_array_equal(J, alone)
    np.testing.assert_array_equal(J, both[1].cpu().numpy())
    np.testing.assert_array_equal(Jb, both[0].cpu().numpy())
    np.testing.assert_allclose((w[:, :, None] * u).sum(1), J, rtol=1e-12)
    assert j_rel_err(J, orc.OracleModel(m, rays=rays).solve_J(orc.params()))[0] < (1e-4 if precision == "FP32" else 1e-10)


@pytest.mark.parametrize("dtau_max", [1.0, 2.0, 3.5, 10.0, 1e3, 1e6])
@pytest.mark.parametrize("lines,bins", [(1, 20), (2, 33)])
def test_double_pivots_over_thick_and_thin_cells(orc, lines, bins, dtau_max):
    """MGX_FP32_DT64 where thick cells (increments to some hundreds, which a large dtau_max leaves
    whole) stand next to thin ones: J and the sum of u against the oracle, within twice the
    form's stated error of 4.8e-6."""
    import paper_2011_14998_gb300 as mgx

    m = synth.random_cloud(90, seed=5 + lines, n_lines=lines, n_freq=bins, x_span=4.0, l_min=1, l_max=1)
    f = 10.0 ** np.random.default_rng(5 + lines).uniform(-3, 2.5, 90)
    m = dict(m, chi0=m["chi0"] * f[:, None], eta0=m["eta0"] * f[:, None], chi_c=m["chi_c"] * f, eta_c=m["eta_c"] * f)
    ctx = mgx.Context(0)
    try:
        mid = ctx.load(m)
        rays = ctx.rays(mid)
        kw = dict(precision=mgx.MGX_FP32_DT64, I_bdy=0.05, dtau_max=dtau_max)
        J = ctx.solve_J(mid, **kw)
        batch = ctx.solve_J_batch([mid], **kw)[0].cpu().numpy()
        u = ctx.solve_u(mid, 0, 90, **kw)
    finally:
        ctx.close()
    Jo = orc.OracleModel(m, rays=rays).solve_J(orc.params(I_bdy=0.05, dtau_max=dtau_max))
    w = 2.0 / (12.0 * 4.0 ** (rays >> 28))
    for got in (J, batch, (w[:, :, None] * u).sum(1)):
        assert j_rel_err(got, Jo)[0] < 9.6e-6


def emissivity_units(mgx, lines, bins, exponent, floor):
    """J in FP64 of a patchy cloud with emissivities (and I_bdy) in units 2^-exponent of the
    plain ones, in plain units; `floor`: the continuum's emissivity, of its plain one."""
    m = synth.random_cloud(90, seed=5 + lines, n_lines=lines, n_freq=bins, x_span=4.0, l_min=1, l_max=1)
    f = 10.0 ** np.random.default_rng(5 + lines).uniform(1, 3, 90)
    s = 2.0 ** exponent
    m = dict(m, chi0=m["chi0"] * f[:, None] * (1e-6 if floor == 0.0 else 1.0), eta0=m["eta0"] * f[:, None] * s,
             chi_c=m["chi_c"] * f, eta_c=m["eta_c"] * f * s * floor)
    ctx = mgx.Context(0)
    try:
        return ctx.solve_J(ctx.load(m), precision=mgx.MGX_FP64, I_bdy=0.05 * s * floor) / s
    finally:
        ctx.close()


@pytest.mark.parametrize("lines,bins", [(1, 20), (2, 33)])
@pytest.mark.parametrize("exponent", [-155, -300])
def test_small_emissivities(lines, bins, exponent):
    """Line emissivities that single precision does not hold, over no continuum emissivity: powers of
    two in the units change nothing but the exponents (1e-14: some roundings all the same)."""
    import paper_2011_14998_gb300 as mgx

    np.testing.assert_allclose(emissivity_units(mgx, lines, bins, exponent, 0.0), emissivity_units(mgx, lines, bins, 0, 0.0),
                               rtol=1e-14)


@pytest.mark.parametrize("lines,bins", [(1, 20), (2, 33)])
@pytest.mark.parametrize("exponent", [280, 300, 600, 800, 900])
def test_large_emissivities(lines, bins, exponent):
    """Source functions to 2^900 over optical depths of hundreds, which the homogeneous rows would
    carry past the range: J in plain units within 64 rows of four roundings each."""
    import paper_2011_14998_gb300 as mgx

    np.testing.assert_allclose(emissivity_units(mgx, lines, bins, exponent, 1.0), emissivity_units(mgx, lines, bins, 0, 1.0),
                               rtol=256 * 2.0 ** -53)
