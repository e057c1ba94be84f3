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


def fp64_error(orc, m, **kw):
    import paper_2011_14998_gb300 as mgx

    ctx = mgx.Context(0)
    try:
        mid = ctx.load(m)
        rays = ctx.rays(mid)
        J = ctx.solve_J(mid, precision=mgx.MGX_FP64, I_bdy=0.05, **kw)
    finally:
        ctx.close()
    return j_rel_err(J, orc.OracleModel(m, rays=rays).solve_J(orc.params(I_bdy=0.05, **kw)))[0]


@pytest.mark.parametrize("bins", [1, 20, 64, 100])
@pytest.mark.parametrize("x_span,ratio", [(4.0, 20.0), (16.0, 10.0), (16.0, 1.0), (13.0, 1.0), (64.0, 3.0)])
def test_fp64_wide_arguments(orc, bins, x_span, ratio):
    """One line whose profile arguments span 31 widths and more on some samples and fewer on others
    (the argument's two forms).  The argument carries five roundings, so an opacity 72 times that
    in its wings (|a| to 6) and J some ten times more: 1e-12 covers both sides."""
    m = synth.random_cloud(120, seed=bins, n_lines=1, n_freq=bins, x_span=x_span, l_min=1, l_max=1)
    m = dict(m, dvw=m["dvw"] * ratio ** np.random.default_rng(bins).uniform(-1, 1, 120))
    assert fp64_error(orc, m) < 1e-12


def test_fp64_plain_samples_between_others(orc):
    """Continua below 1e-150 at a third of the points: samples the fixed-point form leaves to the plain
    step, single and in a row, at any place of a round of records."""
    rng = np.random.default_rng(3)
    m = synth.random_cloud(200, seed=3, n_lines=1, n_freq=40, x_span=4.0, l_min=1, l_max=1)
    tiny = np.where(rng.random(200) < 0.3, 1e-160, 1.0)
    assert fp64_error(orc, dict(m, chi_c=m["chi_c"] * tiny, eta_c=m["eta_c"] * tiny)) < 1e-12


@pytest.mark.parametrize("lines", [1, 2, 5])
def test_fp64_composed_rows(orc, lines):
    """A long static bar, most of it without line opacity, so that its rows are composed by eight, with
    thick cells (split, or too thick to compose) and cells with lines between them.  Some 200 rows of six
    roundings each, on both sides: 3e-13."""
    rng = np.random.default_rng(lines)
    g = np.stack(np.meshgrid(np.arange(60.0), np.arange(3.0), np.arange(3.0), indexing="ij"), -1).reshape(-1, 3)
    pos = g + rng.uniform(-0.2, 0.2, g.shape)
    off, nbr = synth.delaunay_csr(pos)
    n = len(pos)
    m = synth.random_cloud(n, seed=lines, n_lines=lines, n_freq=40, l_min=1, l_max=1)
    on = (rng.random(n) < 0.04)[:, None]
    thick = np.where(rng.random(n) < 0.03, 10.0 ** rng.uniform(1, 4, n), 1.0)
    chi_c = 10.0 ** rng.uniform(-2, -0.5, n) * thick
    m = dict(m, pos=pos, vel=np.zeros((n, 3)), nbr_off=off, nbr_idx=nbr, chi0=m["chi0"] * on, eta0=m["eta0"] * on,
             chi_c=chi_c, eta_c=chi_c * rng.uniform(0.2, 1.5, n))
    for dtau_max in (0.5, 1e5):
        assert fp64_error(orc, m, dtau_max=dtau_max) < 3e-13


def test_fp64_rows_of_equal_increments(orc):
    """Intervals of some hundred velocity samples, most without a line: their rows repeat one map, whose
    rounding must not add up.  Over the origins of a thin cloud the roundings of J (some 1e-15 each, for
    lines of some thousand rows) average out: the mean relative difference from the oracle stays below 2e-15."""
    import paper_2011_14998_gb300 as mgx

    m = synth.random_cloud(60, seed=8, n_lines=1, n_freq=20, x_span=4.0, l_min=1, l_max=1, v_rms=2.0)
    for dvw, chi in ((0.02, 1.0), (0.02, 1e-2), (0.01, 10.0)):
        q = dict(m, dvw=dvw * m["dvw"], chi0=chi * m["chi0"], eta0=chi * m["eta0"], chi_c=chi * m["chi_c"],
                 eta_c=chi * m["eta_c"])
        ctx = mgx.Context(0)
        try:
            mid = ctx.load(q)
            rays = ctx.rays(mid)
            J = ctx.solve_J(mid, precision=mgx.MGX_FP64, I_bdy=0.05)
        finally:
            ctx.close()
        o = np.arange(0, 60, 4)
        Jo = orc.OracleModel(q, rays=rays).solve_J(orc.params(I_bdy=0.05), origins=o)
        d = J[o] / Jo - 1.0
        print(dvw, chi, d.mean(), d.std(), np.abs(d).max())
        assert abs(d.mean()) < 2e-15
