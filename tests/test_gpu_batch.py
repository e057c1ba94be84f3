"""Batched, length-binned persistent solve (mgx_solve_J_batch) and its CUDA-graph
replay: same J as the per-model solve and as the oracle, for models of different
sizes, line counts, bin counts and ray sets in one launch."""
import numpy as np
import pytest

from helpers import j_rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    import synth

    import paper_2011_14998_gb300 as mgx

    mgx.build()
    ctx = mgx.Context(0)
    models = [
        synth.wind_model(900, seed=31, n_freq=50, level=2),
        synth.random_cloud(150, seed=5, n_lines=3, n_freq=13, x_span=3.5, l_min=0, l_max=2, v_rms=1.5),
        synth.grid_model(6, n_freq=9),
        synth.wind_model(600, seed=32, n_freq=20, level=1, l_min=0),
    ]
    mids = [ctx.load(m) for m in models]
    yield ctx, models, mids
    ctx.close()


@pytest.mark.parametrize("prec,tol", [(1, 1e-5), (0, 1e-13)])
def test_batch_matches_single_model_solves(setup, prec, tol):
    ctx, models, mids = setup
    singles = [ctx.solve_J(m, precision=prec) for m in mids]
    outs = ctx.solve_J_batch(mids, precision=prec)
    for J1, Jb in zip(singles, outs):
        assert Jb.shape == J1.shape
        assert j_rel_err(Jb.cpu().numpy(), J1)[0] <= tol


def test_batch_against_oracle(setup, orc):
    ctx, models, mids = setup
    outs = ctx.solve_J_batch(mids, precision=0, dtau_max=0.4, I_bdy=0.05)
    for m, mid, Jb in zip(models, mids, outs):
        om = orc.OracleModel(m, rays=ctx.rays(mid))
        origins = np.arange(0, len(m["pos"]), 7)
        Jo = om.solve_J(orc.params(dtau_max=0.4, I_bdy=0.05), origins=origins)
        assert j_rel_err(Jb.cpu().numpy()[origins], Jo)[0] < 1e-10


def test_graph_replay_with_ray_rebuild(setup):
    import paper_2011_14998_gb300 as mgx

    ctx, models, mids = setup
    ref = ctx.solve_J_batch(mids, precision=1)
    outs = ctx.solve_J_batch(mids, precision=1, flags=mgx.MGX_BATCH_GRAPH | mgx.MGX_BATCH_RAYS)
    first = [o.clone() for o in outs]
    for o in outs:
        o.fill_(float("nan"))
    ctx.solve_J_batch(mids, precision=1, outs=outs, flags=mgx.MGX_BATCH_GRAPH | mgx.MGX_BATCH_RAYS)  # replay
    for a, b, r in zip(first, outs, ref):
        assert np.array_equal(a.cpu().numpy(), b.cpu().numpy())
        assert np.array_equal(a.cpu().numpy(), r.cpu().numpy())


def test_batch_rejects_bad_arguments(setup):
    import torch

    import paper_2011_14998_gb300 as mgx

    ctx, models, mids = setup
    out = torch.empty((900, 50), dtype=torch.float64, device="cuda")
    with pytest.raises(mgx.MgxError):  # a model twice
        mgx.mgx_solve_J_batch(ctx.ptr, [mids[0], mids[0]], mgx.solve_params(), [out, out])


def test_batch_host_outputs(setup):
    """Outputs in host memory (pageable and pinned, mixed with device memory)
    receive the same J as device outputs, in the eager step and in graph replays."""
    import torch

    import paper_2011_14998_gb300 as mgx

    ctx, models, mids = setup
    ref = [o.cpu().numpy() for o in ctx.solve_J_batch(mids, precision=1)]
    outs = []
    for k, o in enumerate(ref):
        if k % 3 == 0:
            outs.append(torch.full(o.shape, -1.0, dtype=torch.float64))
        elif k % 3 == 1:
            outs.append(torch.full(o.shape, -1.0, dtype=torch.float64).pin_memory())
        else:
            outs.append(torch.full(o.shape, -1.0, dtype=torch.float64, device="cuda"))
    params = mgx.solve_params(precision=mgx.MGX_FP32)
    for flags in (0, mgx.MGX_BATCH_GRAPH, mgx.MGX_BATCH_GRAPH):  # eager, plan + capture, replay
        for o in outs:
            o.fill_(-1.0)
        mgx.mgx_solve_J_batch(ctx.ptr, mids, params, outs, flags)
        for o, r in zip(outs, ref):
            assert np.array_equal(o.cpu().numpy(), r)


def test_tuning_changes_speed_not_results(setup):
    """The tracer grid, the row width and the work-list order never change J; the bins per lane
    select a differently compiled kernel, so single-precision J may differ in
    its rounding (fused multiply-adds), far inside the FP32 tolerance."""
    import paper_2011_14998_gb300 as mgx

    ctx, models, mids = setup
    flags = mgx.MGX_BATCH_GRAPH | mgx.MGX_BATCH_RAYS
    ctx.set_tuning(None)
    ref = [o.cpu().numpy() for o in ctx.solve_J_batch(mids, precision=1, flags=flags)]
    for t in ({"bins_per_lane": 2, "trace_ctas_per_sm": 4, "tail_permille": 5, "schedule": 0},
              {"bins_per_lane": 2, "trace_ctas_per_sm": 16, "tail_permille": 1000, "schedule": 1},
              {"bins_per_lane": 1, "trace_ctas_per_sm": 8, "tail_permille": 80, "schedule": 0}):
        ctx.set_tuning(t)
        assert ctx.tuning() == t
        outs = ctx.solve_J_batch(mids, precision=1, flags=flags)
        for o, r in zip(outs, ref):
            if t["bins_per_lane"] == 2:  # the automatic choice for this batch (up to 50 bins)
                assert np.array_equal(o.cpu().numpy(), r)
            else:
                assert j_rel_err(o.cpu().numpy(), r)[0] < 1e-5
    ctx.set_tuning(None)
    assert ctx.tuning() == {"bins_per_lane": 0, "trace_ctas_per_sm": 0, "tail_permille": 0, "schedule": 0}
    with pytest.raises(mgx.MgxError):
        ctx.set_tuning({"bins_per_lane": 3})
    with pytest.raises(mgx.MgxError):
        ctx.set_tuning({"trace_ctas_per_sm": 33})


def test_autotune_keeps_fastest_candidate(setup):
    import paper_2011_14998_gb300 as mgx

    ctx, models, mids = setup
    flags = mgx.MGX_BATCH_GRAPH | mgx.MGX_BATCH_RAYS
    ctx.set_tuning(None)
    ref = [o.cpu().numpy() for o in ctx.solve_J_batch(mids, precision=1, flags=flags)]
    trials, outs = ctx.autotune(mids, precision=1, flags=flags, reps=2)
    assert 5 <= len(trials) <= 10
    assert all(t["step_ms"] > 0 for t in trials)
    best = min(trials, key=lambda t: t["step_ms"])
    chosen = ctx.tuning()
    assert chosen == {k: best[k] for k in chosen}
    for o, r in zip(outs, ref):
        assert j_rel_err(o.cpu().numpy(), r)[0] < 1e-5
    ctx.set_tuning(None)


class LimitedPool:
    """The device's current memory pool replaced by one of at most `limit` bytes (0: no limit).  What is
    allocated inside is freed inside; the pool itself, empty, is left to the process."""

    def __init__(self, limit):
        import ctypes as C

        class Props(C.Structure):
            _fields_ = [("alloc_type", C.c_int), ("handle_types", C.c_int), ("location_type", C.c_int),
                        ("location_id", C.c_int), ("security", C.c_void_p), ("max_size", C.c_size_t),
                        ("usage", C.c_ushort), ("reserved", C.c_ubyte * 54)]

        self.C, self.cu = C, C.CDLL("libcuda.so.1")
        self.props = Props(alloc_type=1, location_type=1, max_size=limit)  # pinned, on device 0
        self.pool, self.before = C.c_void_p(), C.c_void_p()

    def __enter__(self):
        assert self.cu.cuDeviceGetMemPool(self.C.byref(self.before), 0) == 0
        assert self.cu.cuMemPoolCreate(self.C.byref(self.pool), self.C.byref(self.props)) == 0
        assert self.cu.cuDeviceSetMemPool(0, self.pool) == 0
        return self

    def used_high(self):
        v = self.C.c_uint64()
        assert self.cu.cuMemPoolGetAttribute(self.pool, 8, self.C.byref(v)) == 0  # CU_MEMPOOL_ATTR_USED_MEM_HIGH
        return v.value

    def __exit__(self, *_):
        assert self.cu.cuDeviceSetMemPool(0, self.before) == 0
        assert self.cu.cuMemPoolTrimTo(self.pool, self.C.c_size_t(0)) == 0


@pytest.mark.parametrize("batch", [True, False])
def test_without_room_for_u(batch):
    """Few items: u of every pair takes half of the call's memory.  Where there is room for it or for the
    rest, but not for both, the call goes on with one warp per item, and J is the same bit for bit."""
    import torch

    import synth

    import paper_2011_14998_gb300 as mgx

    torch.zeros(1, device="cuda")
    m = synth.random_cloud(400, seed=2, n_lines=1, n_freq=20, l_min=4, l_max=4)
    u_bytes = 400 * 1536 * 20 * 8

    def call(limit):
        with LimitedPool(limit) as pool:
            ctx = mgx.Context(0)
            try:
                mid = ctx.load(m)
                J = (ctx.solve_J_batch([mid], precision=mgx.MGX_FP32)[0].cpu().numpy() if batch
                     else ctx.solve_J(mid, precision=mgx.MGX_FP32))
                return J, pool.used_high()
            finally:
                ctx.close()
                torch.cuda.synchronize()

    J, high = call(0)
    assert high > u_bytes  # u was held
    rest = high - u_bytes
    np.testing.assert_array_equal(call(high - min(u_bytes, rest) // 2)[0], J)


def test_failed_set_rays_leaves_no_ray_set():
    """A ray set for which there is no memory (200 000 points of 393 216 pairs: 315 GB): the model has
    none then, instead of the old one's flag over freed arrays, and can be given one again."""
    import paper_2011_14998_gb300 as mgx

    n = 200_000
    rng = np.random.default_rng(2)
    one = np.ones((n, 1))
    m = dict(pos=rng.random((n, 3)), vel=np.zeros((n, 3)), nbr_off=np.zeros(n + 1, np.int64), nbr_idx=np.zeros(0, np.int32),
             nu0=np.array([1e11]), chi0=one, eta0=one, dvw=one[:, 0], chi_c=one[:, 0], eta_c=one[:, 0], n_freq=2,
             x_span=1.0, l_min=0, l_max=0)
    ctx = mgx.Context(0)
    try:
        mid = ctx.load(m)
        J = ctx.solve_J(mid, I_bdy=0.5)
        with pytest.raises(mgx.MgxError) as e:
            ctx.set_rays(mid, 8, 8)
        assert e.value.status == mgx.MGX_ENOMEM
        for call in (ctx.solve_J, lambda i: ctx.solve_J_batch([i])):
            with pytest.raises(mgx.MgxError) as e:
                call(mid)
            assert e.value.status == mgx.MGX_ESTATE
        ctx.set_rays(mid, 0, 0)
        np.testing.assert_array_equal(ctx.solve_J(mid, I_bdy=0.5), J)
    finally:
        ctx.close()


@pytest.mark.parametrize("what", ["lines", "more bins", "span", "rays", "sample", "deeper tables"])
def test_step_of_a_changed_model(what):
    """A captured step whose model is given other lines (in the same arrays; of another span; with more
    bins) or another ray set (of as many sample points; of fewer), or whose direction tables are replaced for
    another model's finer rays, another model having taken what was freed: the next calls give what a
    new context gives."""
    import synth

    import paper_2011_14998_gb300 as mgx

    a = synth.random_cloud(300, seed=4, n_lines=1, n_freq=20, l_min=0, l_max=1)
    b = synth.random_cloud(300, seed=5, n_lines=1, n_freq=20, l_min=0, l_max=1)
    flags = mgx.MGX_BATCH_GRAPH | mgx.MGX_BATCH_RAYS

    def set_lines(ctx, mid, m):
        mgx.mgx_set_lines(ctx.ptr, mid, m["nu0"], m["chi0"], m["eta0"], m["dvw"], m["chi_c"], m["eta_c"], m["n_freq"],
                          m["x_span"])

    bins = 40 if what == "more bins" else 20
    lines = dict(a, chi0=0.1 * a["chi0"], eta0=0.2 * a["eta0"], n_freq=bins, x_span=2.0 if what == "span" else a["x_span"])
    sample = np.random.default_rng(1).integers(0, 300, 150 if what == "rays" else 300).astype(np.int32)
    changed = dict(a) if what in ("rays", "sample", "deeper tables") else lines
    if what in ("rays", "sample"):
        changed["sample"] = sample
    import torch

    outs = [torch.empty((300, bins), dtype=torch.float64, device="cuda")]
    ctx = mgx.Context(0)
    try:
        mid = ctx.load(dict(a, n_freq=bins) if what != "more bins" else a)
        ctx.solve_J_batch([mid], outs=outs, flags=flags)
        if what in ("rays", "sample"):
            ctx.set_rays(mid, 0, 1, sample)
        elif what != "deeper tables":
            set_lines(ctx, mid, changed)
        ctx.load(b, l_min=0 if what != "deeper tables" else 2, l_max=1 if what != "deeper tables" else 2)
        J = ctx.solve_J_batch([mid], outs=outs, flags=flags)[0].cpu().numpy()
        again = ctx.solve_J_batch([mid], outs=outs, flags=flags)[0].cpu().numpy()
    finally:
        ctx.close()
    ctx = mgx.Context(0)
    try:
        ref = ctx.solve_J_batch([ctx.load(changed)], flags=flags)[0].cpu().numpy()
    finally:
        ctx.close()
    np.testing.assert_array_equal(J, ref)
    np.testing.assert_array_equal(again, ref)


@pytest.mark.parametrize("bad", ["id", "negative id", "offset", "negative offset", "falling offsets"])
def test_graphs_out_of_range_are_refused(bad):
    """Neighbour ids and offsets far outside the arrays: MGX_EINVAL, and the context works on."""
    import synth

    import paper_2011_14998_gb300 as mgx

    m = synth.random_cloud(60, seed=1, l_min=0, l_max=0)
    off, nbr = m["nbr_off"].astype(np.int64).copy(), m["nbr_idx"].copy()
    if bad == "id":
        nbr[7] = 2 ** 31 - 1
    elif bad == "negative id":
        nbr[7] = -2 ** 31
    elif bad == "offset":
        off[9] = 2 ** 40
    elif bad == "negative offset":
        off[9] = -2 ** 40
    else:
        off[9] = off[8] - 1
    ctx = mgx.Context(0)
    try:
        with pytest.raises(mgx.MgxError) as e:
            ctx.load(dict(m, nbr_off=off, nbr_idx=nbr))
        assert e.value.status == mgx.MGX_EINVAL
        assert np.isfinite(ctx.solve_J(ctx.load(m))).all()
    finally:
        ctx.close()
