"""What may change between, and around, the calls that run level sweeps: kernel
variants, masks, streams of other contexts, memory."""
import numpy as np
import pytest
import torch

import workloads
from _helpers import tiny_workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import __graft_entry__ as g
    g.build()


@pytest.fixture
def level_context(monkeypatch):
    """make(precision, ckpt_k, cluster, env, **workload): a context whose boxes
    are advanced by level sweeps whatever their number of points."""
    made = []

    def make(precision=0, ckpt_k=0, cluster=0, env=None, **kw):
        import paper_2205_06649_gb300 as dd
        wl = tiny_workload(**{**dict(obs_count=400, obs_every=2, corr_len=1.5), **kw})
        inp = workloads.generate(wl)
        for k, v in {"DD4DV_LEVEL_MIN_POINTS": 1, **(env or {})}.items():
            monkeypatch.setenv(k, str(v))
        ctx = dd.Context(wl.nlon, wl.nlat, inp["dt"], wl.nsteps, precision=precision)
        made.append(ctx)
        ctx.set_background(inp["x_b0"])
        ctx.set_background_error(wl.sigma_b, wl.corr_len, wl.rf_passes)
        so = np.asarray(wl.sigma_o)[inp["obs_var"]]
        y = np.where(inp["obs_var"] == 0, workloads.H_REF, 0.0) + so * inp["obs_noise"]
        ctx.set_observations(inp["obs_level"], inp["obs_var"], inp["obs_fi"], inp["obs_fj"], y, so)
        ctx.set_decomposition(wl.P1, wl.P2, wl.Q, wl.o_lon, wl.o_lat, wl.o_t, inp["lon_cuts"], inp["lat_cuts"],
                              inp["t_cuts"], cluster=cluster, ckpt_k=ckpt_k)
        return ctx

    yield make
    for ctx in made:
        ctx.destroy()


def controls(ctx, seed=17):
    return 0.3 * np.random.default_rng(seed).standard_normal(ctx.ctrl_total)


RAGGED = dict(nlon=70, nlat=38, nsteps=30, P1=3, P2=2, Q=2, o_lon=3, o_lat=3, o_t=3, uneven=True)


@pytest.mark.parametrize("precision", [0, 1])
def test_backward_after_a_variant_change_reads_what_was_stored(level_context, precision):
    """Under checkpoints the cluster forward stores every fourth level only; a
    backward pass that follows a return to the level sweeps must recompute the
    others, not read them as if they were there."""
    ctx = level_context(precision, ckpt_k=4, **RAGGED)
    assert ctx.sweep_kernels() == {"forward": 5, "adjoint": 5}
    w = controls(ctx)
    _, ref = ctx.eval(w)
    ctx.eval(0.0 * w)   # other levels in the trajectory buffer
    ctx.set_sweep_variant(1, 1)
    ctx.eval_forward(w)
    ctx.set_sweep_variant(0, 0)
    assert np.array_equal(ctx.eval_backward(), ref)
    ctx.eval_forward(w)   # and the other way: a level forward, a cluster adjoint
    ctx.set_sweep_variant(1, 1)
    assert np.array_equal(ctx.eval_backward(), ref)


RING = {
    "ragged": RAGGED,
    "many rows": dict(nlon=384, nlat=160, nsteps=12, P1=4, P2=2, Q=4, o_lon=4, o_lat=4),
    "wide": dict(nlon=560, nlat=90, nsteps=6, P1=2, P2=2, Q=2, o_lon=4, o_lat=3),     # boxes 288 wide, rows in threes
    "walls": dict(nlon=52, nlat=64, nsteps=9, P1=2, P2=1, Q=3, o_lon=3, o_t=1),
    "one box": dict(nlon=33, nlat=100, nsteps=9, P1=1, P2=1, Q=1),                    # periodic
}


@pytest.mark.parametrize("name", list(RING))
@pytest.mark.parametrize("ctas", [1, 3, 8])
def test_pipelined_adjoint_in_its_steady_state(level_context, name, ctas):
    """The pipelined adjoint with so few CTAs that each takes many tiles: slots
    and descriptors come round again, masked boxes are passed over (the last
    ones too), gradients stay bit for bit those of the plain phases."""
    out, kernels = [], []
    for env in (dict(DD4DV_RING_MIN_TILES=0, DD4DV_RING_MAX_CTAS=ctas), dict(DD4DV_RING_MIN_TILES=1 << 40)):
        ctx = level_context(1, env=env, **RING[name])
        w, rng = controls(ctx), np.random.default_rng(3)
        p, force = rng.standard_normal(ctx.ctrl_total), rng.standard_normal(ctx.traj_total)
        ctx.exchange(0.5 * w)
        k0 = ctx.launch_count()
        r = [ctx.eval(w)[1], ctx.gn_hessvec(w, p), ctx.adjoint(w, force)]
        kernels.append(ctx.launch_count() - k0)
        for m in ((np.arange(ctx.n_sub) % 3 == 0), np.arange(ctx.n_sub) < (ctx.n_sub + 1) // 2):
            ctx.set_owned(m.astype(np.int32))
            r.append(ctx.eval(w)[1])
        out.append(r)
    assert kernels[0] != kernels[1]   # (the pipelined form adds the observations in a kernel of their own)
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_lost_copy_is_reported_and_never_returned_as_a_gradient(level_context, monkeypatch):
    """A wait of the pipelined adjoint that runs out (here: at once, no polls)
    gives DD4DV_ETIMEOUT; a call with device pointers does not synchronise, so
    its gradient is NaN and the next call reports it.  The context stays usable."""
    import paper_2205_06649_gb300 as dd
    many = RING["many rows"]
    ref = level_context(1, env=dict(DD4DV_RING_MIN_TILES=1 << 40), **many)
    w = controls(ref)
    J, g = ref.eval(w)
    ctx = level_context(1, env=dict(DD4DV_RING_MIN_TILES=0, DD4DV_RING_MAX_CTAS=8, DD4DV_RING_EXPIRE=1), **many)
    monkeypatch.delenv("DD4DV_RING_EXPIRE")
    with pytest.raises(dd.DD4DVError, match="ETIMEOUT.*did not reach"):
        ctx.eval(w)
    wd = torch.as_tensor(w, device="cuda")
    Jd, gd = ctx.eval(wd)
    torch.cuda.synchronize()
    assert np.array_equal(Jd.cpu().numpy(), J) and torch.isnan(gd).any()
    with pytest.raises(dd.DD4DVError, match="ETIMEOUT"):
        ctx.eval(wd)
    ctx.set_sweep_variant(1, 1)
    assert np.array_equal(ctx.eval(w)[1], g)


def test_pipelined_adjoints_of_two_contexts_on_two_threads(level_context):
    """Two contexts whose pipelined launches ask for different amounts of shared
    memory, each on its own thread: neither may lower the limit that the other is
    about to launch with."""
    import threading
    env = dict(DD4DV_RING_MIN_TILES=0)
    pair = [level_context(1, env=env, nlon=33, nlat=14, nsteps=40, P1=1, P2=1, Q=1),
            level_context(1, env=env, nlon=384, nlat=160, nsteps=40, P1=4, P2=2, Q=1, o_lon=4, o_lat=4)]
    w = [controls(c) for c in pair]
    ref = [c.eval(v)[1] for c, v in zip(pair, w)]
    wrong = []

    def work(k):
        try:
            for _ in range(60):
                if not np.array_equal(pair[k].eval(w[k])[1], ref[k]):
                    wrong.append((k, "gradient"))
        except Exception as e:   # noqa: BLE001 (shown below)
            wrong.append((k, str(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


@pytest.mark.parametrize("precision,ckpt_k", [(0, 0), (0, -1), (1, 0)])
def test_tiles_of_several_rounds(level_context, precision, ckpt_k):
    """Tiles in which a thread takes several points (decompositions of more than
    2 million points): states and gradients to the last bit as with one round, J
    up to the order of its sums (1e-13 of FP64 terms, as between sweep kinds)."""
    out = []
    for rounds in (1, 2, 4):
        ctx = level_context(precision, ckpt_k, env=dict(DD4DV_LEVEL_ROUNDS=rounds, DD4DV_RING_MIN_TILES=1 << 40), **RAGGED)
        w = controls(ctx)
        ctx.exchange(0.5 * w)
        J, g = ctx.eval(w)
        out.append((J, g, ctx.trajectories(w), ctx.gn_hessvec(w, 0.1 * w)))
    for J, *rest in out[1:]:
        assert np.max(np.abs(J - out[0][0])) <= 1e-13 * np.max(np.abs(J))
        for a, b in zip(rest, out[0][1:]):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("precision,ring,rounds", [(0, 0, 1), (0, 0, 2), (1, 0, 1), (1, 0, 4), (1, 1, 4)])
def test_owned_boxes_alone_give_what_all_of_them_give(level_context, precision, ring, rounds):
    """Evaluations and local solves of a share of the boxes launch those boxes
    alone: J, gradients and solved controls to the last bit as with all boxes
    owned, whatever the share (windows of one length only, one box, none)."""
    import paper_2205_06649_gb300 as dd
    env = dict(DD4DV_RING_MIN_TILES=0 if ring else 1 << 40, DD4DV_LEVEL_ROUNDS=rounds)
    kw = dict(env=env, nlon=96, nlat=60, nsteps=31, P1=3, P2=2, Q=3, o_lon=3, o_lat=3, o_t=3, uneven=True)
    ctx = level_context(precision, **kw)
    w = controls(ctx)
    b, off = np.asarray(ctx.boxes), np.asarray(ctx.offsets)
    n = ctx.n_sub
    J, g = ctx.eval(w)
    masks = [np.arange(n) % 2 == 1, b[:, 5] - b[:, 4] == (b[:, 5] - b[:, 4]).min(), np.arange(n) == n - 1,
             np.arange(n) < n // 3, np.zeros(n, dtype=bool)]
    for m in masks:
        ctx.set_owned(m.astype(np.int32))
        Jm, gm = ctx.eval(w)
        Jf = ctx.eval_forward(w)
        gb = ctx.eval_backward()
        for s in np.nonzero(m)[0]:
            c = slice(off[s], off[s + 1])
            assert Jm[s] == J[s] and Jf[s] == J[s], s
            assert np.array_equal(gm[c], g[c]) and np.array_equal(gb[c], g[c]), s
    ctx.set_owned(None)
    J2, g2 = ctx.eval(w)
    assert np.array_equal(J2, J) and np.array_equal(g2, g)
    # an outer iteration in three shares against one of all boxes
    solver = dd.solver_defaults(max_local_iters=6, max_outer=1, eps_outer=0.0)
    whole = level_context(precision, **kw)
    whole.outer_step(solver)
    got = np.zeros(ctx.ctrl_total)
    for k in range(3):
        ctx.set_owned((np.arange(n) % 3 == k).astype(np.int32))
        ctx.set_controls(0.0 * got)
        ctx.local_solve(solver)
        x = ctx.get_controls()
        for s in range(k, n, 3):
            got[off[s]:off[s + 1]] = x[off[s]:off[s + 1]]
    assert np.array_equal(got, whole.get_controls()) and got.any()


# ---- memory ----

GRID = dict(nlon=512, nlat=256, nsteps=10, P1=6, P2=4, Q=1, o_lon=4, o_lat=4, corr_len=0.0)   # 190,000 points a level


class Hog:
    """Holds all device memory but `leave` bytes."""

    def __init__(self, leave):
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        self.t = torch.empty(max(0, free - int(leave)), dtype=torch.uint8, device="cuda")

    def __enter__(self):
        return self

    def __exit__(self, *_):
        del self.t
        torch.cuda.empty_cache()


def test_level_scratch_leaves_the_reserve(level_context):
    """With less free memory than the reserve of the optional buffers (4 GB + 5 %
    of the device) the level sweeps' scratch is left out: what the context
    allocates later has to find its memory."""
    ref = level_context(0, **GRID)
    assert ref.sweep_kernels() == {"forward": 5, "adjoint": 5}
    w = controls(ref)
    g = ref.eval(w)[1]
    with Hog(4 * 2**30 + 0.05 * torch.cuda.mem_get_info()[1] - 256 * 2**20):
        ctx = level_context(0, ckpt_k=-1, **GRID)
        assert 5 not in ctx.sweep_kernels().values()
        assert np.array_equal(ctx.eval(w)[1], g)


def test_lazily_made_buffers_find_the_memory_of_the_level_scratch(level_context):
    """A Gauss-Newton product needs a trajectory more.  Where only the level
    sweeps' scratch (here five levels of ten) stands in its way, that goes and the
    cluster sweeps run."""
    kw = {**GRID, "nsteps": 3}
    ref = level_context(0, **kw)
    w, p = controls(ref), controls(ref, 5)
    h = ref.gn_hessvec(w, p)
    ctx = level_context(0, **kw)
    b = np.asarray(ctx.boxes)
    level = 3 * 8 * int(np.sum(b[:, 3] * ((b[:, 1] + 3) // 4 * 4)))
    need = 4 * level + 4 * 8 * ctx.ctrl_total   # four levels of dx and four control vectors
    assert 5 * level > 16 * 2**20
    with Hog(need - 2.5 * level):
        assert ctx.sweep_kernels() == {"forward": 5, "adjoint": 5}
        got = ctx.gn_hessvec(w, p)
        assert 5 not in ctx.sweep_kernels().values()
    assert np.max(np.abs(got - h)) <= 1e-12 * np.max(np.abs(h))
    _, g = ref.eval(w)
    assert np.array_equal(ctx.eval(w)[1], g)


def test_launch_shapes_give_the_level_scratch_back(level_context):
    ctx = level_context(0, **GRID)
    cfg = ctx.sweep_config()
    free = torch.cuda.mem_get_info()[0]
    ctx.set_sweep_config(cfg["forward"], cfg["adjoint"], cfg["stored_stages"])
    assert torch.cuda.mem_get_info()[0] - free >= 16 * 2**20


def test_kept_turkel_zwas_block_is_given_back(level_context):
    """The block that Turkel-Zwas calls keep (here 75 MB) goes when another
    allocation needs it, and comes back with the next such call."""
    import paper_2205_06649_gb300 as dd
    kw = dict(nlon=256, nlat=128, nsteps=90, P1=4, P2=4, Q=1, o_lon=4, o_lat=4, o_t=0, corr_len=0.0, obs_count=100)
    wl = tiny_workload(**kw)
    inp = workloads.generate(wl)
    ctx = dd.Context(wl.nlon, wl.nlat, inp["dt"], wl.nsteps)
    try:
        ctx.set_background(inp["x_b0"])
        ctx.set_background_error(wl.sigma_b, 0.0, 4)
        so = np.asarray(wl.sigma_o)[inp["obs_var"]]
        ctx.set_observations(inp["obs_level"], inp["obs_var"], inp["obs_fi"], inp["obs_fj"], 0.0 * so, so)
        v = 0.1 * np.random.default_rng(1).standard_normal(3 * wl.nlon * wl.nlat)
        J, g = ctx.tz_eval(2, 1, 0.5, v)
        dec = (wl.P1, wl.P2, wl.Q, wl.o_lon, wl.o_lat, wl.o_t, inp["lon_cuts"], inp["lat_cuts"], inp["t_cuts"])
        ctx.set_decomposition(*dec, ckpt_k=-1, cluster=4)   # (loads its kernels)
        b = np.asarray(ctx.boxes)
        copies = 8 * 3 * (wl.nsteps + 1) * (int(np.sum(b[:, 3] * ((b[:, 1] + 3) // 4 * 4))) + wl.nlon * wl.nlat)
        ctx.set_background(inp["x_b0"])                     # frees the decomposition
        free = torch.cuda.mem_get_info()[0]
        ctx.set_decomposition(*dec, ckpt_k=-1, cluster=4)
        used = free - torch.cuda.mem_get_info()[0] - copies   # without the copies for a reset, which are optional
        ctx.set_background(inp["x_b0"])
        with Hog(used - 40 * 2**20):
            ctx.set_decomposition(*dec, ckpt_k=-1, cluster=4)
        J2, g2 = ctx.tz_eval(2, 1, 0.5, v)
        assert J2 == J and np.max(np.abs(g2 - g)) <= 1e-12 * np.max(np.abs(g))
    finally:
        ctx.destroy()
