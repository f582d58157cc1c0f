"""Roundings that results depend on beyond one run of a kernel."""
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


@pytest.mark.parametrize("nlon,nlat,P1,P2", [(9, 4, 1, 1), (70, 38, 2, 2), (1100, 600, 12, 8)])
def test_forward_run_is_the_background_trajectory(nlon, nlat, P1, P2):
    """dd4dv_forward(x_b) and the background forecast are the same model: equal
    bit for bit, on a grid smaller than a tile and its halo, one of several
    tiles and one that takes a launch per stage."""
    import paper_2205_06649_gb300 as dd
    wl = tiny_workload(nlon=nlon, nlat=nlat, nsteps=5, P1=P1, P2=P2, Q=1, obs_count=20)
    inp = workloads.generate(wl)
    ctx = dd.Context(nlon, nlat, inp["dt"], wl.nsteps)
    ctx.set_background(inp["x_b0"])
    ctx.set_background_error(wl.sigma_b, 0.0, 4)
    so = np.asarray(wl.sigma_o)[inp["obs_var"]]
    ctx.set_observations(inp["obs_level"], inp["obs_var"], inp["obs_fi"], inp["obs_fj"], 0.0 * so, so)
    ctx.set_decomposition(P1, P2, 1, 1, 1, 0, inp["lon_cuts"], inp["lat_cuts"], inp["t_cuts"])
    run, back = ctx.forward(inp["x_b0"]), ctx.boundary_trajectory()
    ctx.destroy()
    assert np.array_equal(run, back)


def test_turkel_zwas_run_drifts_like_the_plain_step():
    """Every operation on h rounds by up to half an ulp (2.3e-13 m), in the RK3
    combination 1/3 X + 2/3 Y to one side, so that the mean of h drifts by the
    order of its operations.  The run's order rounds 1/3 X first and fuses 2/3 Y;
    the oracle's divides and adds.  Their drifts per step, from the same
    combinations of random values, differ by 5e-14 m; fusing 1/3 X instead would
    leave no difference, so half of it is the bar."""
    import oracle
    import paper_2205_06649_gb300 as dd
    nlon, nlat, nsteps = 96, 48, 120
    wl = workloads.preset("small", nlon=nlon, nlat=nlat, nsteps=nsteps)
    inp = workloads.generate(wl)
    ctx = dd.Context(nlon, nlat, inp["dt"], nsteps)
    run = ctx.tz_forward(3, 1, 0.0, inp["x_t0"])[-1, 0]
    ctx.destroy()
    grid = oracle.Grid(nlon, nlat, workloads.RADIUS, workloads.GRAVITY, workloads.OMEGA, workloads.LAT_MIN_DEG,
                       workloads.LAT_MAX_DEG)
    ref = oracle.tz_forward(grid, torch.as_tensor(inp["x_t0"]), inp["dt"], nsteps, 3, 1, 0.0).numpy()[-1, 0]
    rng = np.random.default_rng(0)
    X = 4000.0 + 30.0 * rng.standard_normal(200000)
    Y = X + 0.01 * rng.standard_normal(X.size)
    L = np.longdouble
    fused = (L(2.0 / 3.0) * Y.astype(L) + ((1.0 / 3.0) * X).astype(L)).astype(np.float64)
    want = np.mean(fused - (X / 3.0 + (2.0 / 3.0) * Y))
    got = np.mean(run - ref) / nsteps
    assert -6e-14 < want < -4e-14
    assert abs(got - want) <= 0.5 * abs(want), (got, want)
