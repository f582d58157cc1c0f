"""The level sweeps (all subdomains advanced together, one launch per RK3
stage) against the cluster sweeps on the same context: trajectories, gradients
and adjoint runs bit for bit, J up to the order of its partial sums (FP64: a
few roundings of at most 1e5 terms, 1e-13; FP32 state: the cluster sweeps add a
thread's FP32 terms in FP32, 1e-6 as between launch shapes), with boxes that
are periodic, at walls, one tile or several, of widths that are and are not
multiples of a thread's columns, and windows of different lengths; the FP32
adjoint also by the pipelined kernels (one and several tiles per CTA)."""
import numpy as np
import pytest
import torch

import workloads
from _helpers import tiny_workload

pytestmark = pytest.mark.gpu

CASES = {
    "ragged": dict(),                                                                # uneven boxes and windows
    "periodic": dict(nlon=61, nlat=38, nsteps=23, P1=1, P2=2, Q=2, o_lat=2, o_t=2),   # odd width, wrap in lon
    "one box": dict(nlon=33, nlat=14, nsteps=9, P1=1, P2=1, Q=1),
    "walls": dict(nlon=24, nlat=12, nsteps=9, P1=3, P2=1, Q=2, o_lon=2, o_t=1),       # both walls in every box
    "many rows": dict(nlon=384, nlat=160, nsteps=12, P1=4, P2=2, Q=4, o_lon=4, o_lat=4),   # several tiles per CTA
    "wide": dict(nlon=300, nlat=48, nsteps=6, P1=2, P2=2, Q=1, o_lon=3, o_lat=3),     # several tiles per box
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("precision,ckpt_k,pipelined",
                         [(0, 0, 0), (0, -1, 0), (0, -3, 0), (1, 0, 0), (1, 4, 0), (1, 0, 1), (1, 4, 1)])
def test_level_sweeps_equal_cluster_sweeps(monkeypatch, name, precision, ckpt_k, pipelined):
    import paper_2205_06649_gb300 as dd
    over = dict(obs_count=400, obs_every=2, corr_len=1.5)
    wl = (workloads.preset("ragged") if name == "ragged" else tiny_workload(**{**over, **CASES[name]}))
    inp = workloads.generate(wl)
    monkeypatch.setenv("DD4DV_LEVEL_MIN_POINTS", "1")
    monkeypatch.setenv("DD4DV_RING_MIN_TILES", "0" if pipelined else str(1 << 40))
    ctx = dd.Context(wl.nlon, wl.nlat, inp["dt"], wl.nsteps, precision=precision)
    ctx.set_background(inp["x_b0"])
    ctx.set_background_error(wl.sigma_b, wl.corr_len, wl.rf_passes)
    so = np.asarray(wl.sigma_o)[inp["obs_var"]]
    y = np.where(inp["obs_var"] == 0, workloads.H_REF, 0.0) + so * inp["obs_noise"]
    ctx.set_observations(inp["obs_level"], inp["obs_var"], inp["obs_fi"], inp["obs_fj"], y, so)
    ctx.set_decomposition(wl.P1, wl.P2, wl.Q, wl.o_lon, wl.o_lat, wl.o_t, inp["lon_cuts"], inp["lat_cuts"],
                          inp["t_cuts"], ckpt_k=ckpt_k)
    assert ctx.sweep_kernels() == {"forward": 5, "adjoint": 5}
    cfg = ctx.sweep_config()
    rng = np.random.default_rng(17)
    w = 0.3 * rng.standard_normal(ctx.ctrl_total)
    p = rng.standard_normal(ctx.ctrl_total)
    force = rng.standard_normal(ctx.traj_total)
    odd = (np.arange(ctx.n_sub) % 2 == 0).astype(np.int32)
    out = []
    for level in (True, False):
        if not level:
            ctx.set_sweep_config(cfg["forward"], cfg["adjoint"], cfg["stored_stages"])
            assert 5 not in ctx.sweep_kernels().values()
        J, g = ctx.eval(w)
        J2 = ctx.eval_forward(w)
        g2 = ctx.eval_backward(scale=np.linspace(0.5, 2.0, ctx.n_sub))
        x, a, h = ctx.trajectories(w), ctx.adjoint(w, force), ctx.gn_hessvec(w, p)
        ctx.exchange(w)
        Je, ge = ctx.eval(0.5 * w)
        ctx.reset_exchange()
        ctx.set_owned(odd)
        Jm, gm = ctx.eval(w)
        ctx.set_owned(None)
        out.append(dict(J=J, J2=J2, Je=Je, Jm=Jm, g=g, g2=g2, x=x, a=a, h=h, ge=ge, gm=gm))
    ctx.destroy()
    lev, clu = out
    for k in ("g", "g2", "x", "a", "ge", "gm") + (("h",) if precision else ()):
        assert np.array_equal(lev[k], clu[k]), (name, k)
    # FP64 products: the level tangent-linear sweep's contractions are the compiler's, some 1e3 roundings deep
    assert np.max(np.abs(lev["h"] - clu["h"])) <= 1e-12 * np.max(np.abs(clu["h"])), name
    bar = 1e-13 if precision == 0 else 1e-6
    for k in ("J", "J2", "Je", "Jm"):
        assert np.max(np.abs(lev[k] - clu[k])) <= bar * np.max(np.abs(clu[k])), (name, k)


@pytest.mark.parametrize("nlon,nlat", [(3, 2), (5, 3), (24, 12), (129, 40), (1100, 600)])
def test_global_step_kernel_matches_oracle(nlon, nlat):
    """The global model by the step kernel (tiles with halos; grids smaller than
    a tile and its halo) and, on the largest grid, by the stage kernels, against
    the oracle's model: two steps within 1e-13 relative (FP64 roundings)."""
    import oracle
    import paper_2205_06649_gb300 as dd
    rng = np.random.default_rng(nlon)
    x0 = np.stack([4000 + 10 * rng.standard_normal((nlat, nlon)), rng.standard_normal((nlat, nlon)),
                   rng.standard_normal((nlat, nlon))])
    grid = oracle.Grid(nlon, nlat, workloads.RADIUS, workloads.GRAVITY, workloads.OMEGA, workloads.LAT_MIN_DEG,
                       workloads.LAT_MAX_DEG)
    dt = 0.1 * 6.371e6 * 0.17 * 2 * np.pi / nlon / 210.0
    ref = oracle.global_forward(grid, torch.as_tensor(x0), dt, 2).numpy()
    ctx = dd.Context(nlon, nlat, dt, 2)
    got = ctx.forward(x0)
    ctx.destroy()
    for v in range(3):
        assert np.max(np.abs(got[:, v] - ref[:, v])) <= 1e-13 * np.max(np.abs(ref[:, v])), v
