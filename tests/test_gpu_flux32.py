"""The mixed form's FP32 fluxes: the 3D direction kernels in every pencil shape, the 1D tile's faces of equal
states, and the 3D mesh filter."""
import numpy as np
import pytest

from oracle import operator as op
from oracle import stepper

from sides import gpu_setup, oracle_setup, to_np
from test_gpu_3d import _box, _mixed_rhs, _xdot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [1, 2, 3, 4])
@pytest.mark.parametrize("n,periodic", [((16, 33, 8), True), ((17, 9, 32), False), ((33, 15, 31), True)])
def test_pencil_shapes_against_oracle(tile, n, periodic):
    """Right-hand sides of a rough state on a moving wavy mesh at the pencils' edges (whole, one node over, one short):
    within 1e-5 of the flux scale, the bound of the form's other right-hand sides."""
    w = _box(*n, periodic, amp=0.01 if periodic else 0.0, seed=n[0])
    sch, _, JU_o, J_o, x = oracle_setup(w)
    dU_o, dJ_o = op.rhs(sch, JU_o, J_o, x, _xdot(w))
    dU, dJ = _mixed_rhs(w, tile)
    h = min(w["dxi"])
    assert np.abs(dU[0].astype(float) - dU_o).sum() < 1e-5 * np.abs(JU_o).sum() / h
    assert np.abs(dJ[0].astype(float) - dJ_o).sum() < 1e-5 * np.abs(J_o).sum() / h


@pytest.mark.parametrize("t_over_tc,ok", [(1.2, True), (0.9, False)])
def test_1d_uniform_state(t_over_tc, ok):
    """A uniform state at the critical density: every face lies between equal nodes, where the dissipation is zero.  Above
    the critical temperature the right-hand sides vanish exactly; below it (p > 0, but inside the spinodal) the state is
    refused as it is between unequal nodes."""
    import torch

    from paper_2407_05568_gb300 import es
    from paper_2407_05568_gb300 import workloads as wl
    w = wl.sine_1d(300)
    g = w["gas"]
    rho = 1.0 / (3.0 * g["b"])
    T = t_over_tc * 8.0 * g["a"] / (27.0 * g["R"] * g["b"])
    w["rho"] = np.full_like(w["rho"], rho)
    w["v"] = np.full_like(w["v"], 0.25)
    w["p"] = np.full_like(w["p"], rho * g["R"] * T / (1.0 - g["b"] * rho) - g["a"] * rho * rho)
    assert w["p"].min() > 0.0
    ctx, JU, J, xt = gpu_setup(w, precision="mixed")
    dU, dJ = torch.empty_like(JU), torch.empty_like(J)
    es.es_rhs(ctx, JU, J, xt, None, dU, dJ)
    assert (es.es_check(ctx) == 0) == ok
    if ok:
        assert not to_np(dU).any()


@pytest.mark.parametrize("n,periodic", [((16, 17, 15), True), ((33, 8, 16), False), ((9, 31, 20), True)])
@pytest.mark.parametrize("passes", [0, 1, 4, 9])
def test_3d_filter_passes(n, periodic, passes):
    """The monitor's filter in float, warps of 32 nodes by two lines and segments of planes with whole, ragged and wrapped
    edges: the mesh velocity within 2e-5 of the oracle's (the bound of the form's redistribution against it)."""
    import torch

    from paper_2407_05568_gb300 import es
    w = _box(*n, periodic, amp=0.005)
    w["moving"] = True
    w["mesh"] = dict(monitor="smooth", alphas=(20.0, 15.0), kappa=2, filter_passes=passes, sweeps=3, eps=0.0)
    sch, mc, JU_o, J_o, x_o = oracle_setup(w)
    xd_o, _, gam_o = stepper.redistribute(sch, mc, JU_o, J_o, x_o, 1e-3)
    ctx, JU, J, xt = gpu_setup(w, precision="mixed")
    xd = torch.empty_like(xt)
    _, gam = es.es_mesh_redistribute(ctx, JU, J, xt, 1e-3, xd)
    assert abs(gam - gam_o) <= 2e-5 * gam_o
    assert np.abs(xd.cpu().numpy() - xd_o).max() <= 2e-5 * np.abs(xd_o).max()


@pytest.mark.parametrize("n", [8, 57, 58, 59, 116, 117, 254, 255, 17632, 17633])
@pytest.mark.parametrize("bc", ["periodic", "outflow"])
def test_1d_tiles_against_oracle(n, bc):
    """The two 1D tiles (58 and 254 nodes) at their edges and at the size where one takes over from the other: right-hand
    sides of a rough state on a moving mesh within 1e-5 of the flux scale, the bound of the form's other right-hand sides."""
    import torch

    from paper_2407_05568_gb300 import es
    from paper_2407_05568_gb300 import workloads as wl
    x, d = wl.uniform_nodes(n, 0.0, 1.0, bc == "periodic")
    w = wl.sine_1d(max(n, 8))
    w.update(bc=(bc,), x=x[None].copy(), dxi=(d,))
    w["rho"], w["v"], w["p"] = wl.rough_state((n,), 3 + n, 1)
    xdot = 0.05 * np.sin(2 * np.pi * x + 0.3)[None]
    if bc != "periodic":
        xdot[:, [0, -1]] = 0.0
    sch, _, JU_o, J_o, x_o = oracle_setup(w)
    dU_o, dJ_o = op.rhs(sch, JU_o, J_o, x_o, xdot)
    ctx, JU, J, xt = gpu_setup(w, precision="mixed")
    dU, dJ = torch.empty_like(JU), torch.empty_like(J)
    es.es_rhs(ctx, JU, J, xt, torch.tensor(xdot, device="cuda"), dU, dJ)
    assert es.es_check(ctx) == 0, es.es_last_error(ctx)
    assert np.abs(to_np(dU) - dU_o).sum() < 1e-5 * np.abs(JU_o).sum() / d
    assert np.abs(to_np(dJ) - dJ_o).sum() < 1e-5 * np.abs(J_o).sum() / d


@pytest.mark.parametrize("n", [200, 239, 256, 278, 280, 300])
def test_2d_cfl_blocks(n):
    """The mixed form's CFL kernel with blocks of up to 256 threads, of up to 512 (one per SM: 196 to 278 squared nodes on 152
    SMs) and of 256 again: the time step of a smooth state on a fixed mesh within 1e-5 of the FP64 form's, and steps run."""
    from paper_2407_05568_gb300 import es
    from paper_2407_05568_gb300 import workloads as wl
    w = wl.sine_2d(n)
    dts = []
    for prec in ("fp64", "mixed"):
        ctx, JU, J, x = es.setup_workload(w, prec)
        dts.append(es.es_cfl_dt(ctx, JU, J, x, None))
        es.es_steps(ctx, JU, J, x, 2, 1e30)
        assert es.es_check(ctx) == 0, es.es_last_error(ctx)
    assert abs(dts[1] - dts[0]) <= 1e-5 * dts[0]
