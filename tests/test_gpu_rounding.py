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
