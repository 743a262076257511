"""The FP64 mesh redistribution's kernels at the edges of their ranges: the tiles of small meshes (filter passes and sweeps
in one launch) and the pass-by-pass kernels of larger ones, every boundary condition, ragged sizes and pass counts."""
import numpy as np
import pytest

from oracle import stepper
from paper_2407_05568_gb300 import workloads as wl

from sides import gpu_setup, oracle_setup

pytestmark = pytest.mark.gpu

BCS = {"periodic": ("periodic", "periodic"), "outflow": ("outflow", "outflow"), "walls": ("reflect", "symmetry_lo"),
       "mixed": ("periodic", "reflect"), "swapped": ("outflow", "periodic")}


def _mesh2d(n1, n2, bc, seed):
    """Density bumps and a moved mesh on [0, 1]^2; periodic directions take a periodic displacement."""
    x1, d1 = wl.uniform_nodes(n1, 0.0, 1.0, bc[0] == "periodic")
    x2, d2 = wl.uniform_nodes(n2, 0.0, 1.0, bc[1] == "periodic")
    X, Y = np.meshgrid(x1, x2)
    rng = np.random.default_rng(seed)
    ph = rng.uniform(0.0, 2 * np.pi, 3)
    bx = np.sin(np.pi * X) if bc[0] != "periodic" else 1.0
    by = np.sin(np.pi * Y) if bc[1] != "periodic" else 1.0
    x = np.stack([X + 0.2 * d1 * bx * by * np.sin(2 * np.pi * (X + Y) + ph[0]),
                  Y + 0.2 * d2 * bx * by * np.cos(2 * np.pi * (X - Y) + ph[1])])
    rho = 0.6 + 0.25 * np.tanh(8.0 * np.sin(2 * np.pi * (X + 0.6 * Y) + ph[2]))
    return dict(gas=wl.UNITS_A, dim=2, n=(n2, n1), dxi=(d1, d2), bc=bc, period=(1.0, 1.0), x=x, rho=rho,
                v=np.stack([0.1 * np.ones_like(X), 0.0 * X]), p=1.0 + 0.05 * np.cos(2 * np.pi * Y), cfl=0.4, moving=True,
                t_end=1e30)


def _compare(w, tol=1e-11):
    import torch

    from paper_2407_05568_gb300 import es
    sch, mc, JU_o, J_o, x_o = oracle_setup(w)
    dt = 1e-3
    xd_o, sw_o, gam_o = stepper.redistribute(sch, mc, JU_o, J_o, x_o, dt)
    ctx, JU, J, xt = gpu_setup(w)
    xd = torch.empty_like(xt)
    sw, gam = es.es_mesh_redistribute(ctx, JU, J, xt, dt, xd)
    assert sw == sw_o
    # x^[mu] - x^n keeps 16 digits of the coordinates, so a few 1e-16 of 1 over the displacements' size
    size = max(np.abs(xd_o).max(), 1e-3 * min(w["dxi"]) / dt)
    assert abs(gam - gam_o) <= 1e-10 * gam_o
    assert np.abs(xd.cpu().numpy() - xd_o).max() <= tol * size


@pytest.mark.parametrize("bc", list(BCS))
@pytest.mark.parametrize("shape,passes,sweeps", [((8, 8), 5, 5), ((9, 31), 1, 1), ((20, 14), 5, 10), ((41, 29), 10, 3),
                                                 ((61, 33), 11, 2), ((33, 61), 0, 11), ((270, 285), 5, 5),
                                                 ((290, 271), 2, 4)])
def test_redistribution_2d(bc, shape, passes, sweeps):
    w = _mesh2d(*shape, BCS[bc], 7 + shape[0])
    w["mesh"] = dict(monitor="vdw", alphas=(1200.0, 1200.0, 1200.0), kappa=2, filter_passes=passes, sweeps=sweeps,
                     eps=0.0)
    _compare(w)


@pytest.mark.parametrize("monitor,kappa,eps", [("smooth", 2, 0.0), ("vdw", 1, 0.0), ("vdw", 2, 0.05)])
def test_redistribution_monitors_and_tolerance(monitor, kappa, eps):
    w = _mesh2d(45, 38, BCS["outflow"], 3)
    w["mesh"] = dict(monitor=monitor, alphas=(20.0, 15.0, 30.0), kappa=kappa, filter_passes=4, sweeps=30,
                     eps=eps * w["dxi"][0])
    _compare(w)


@pytest.mark.parametrize("bc", ["periodic", "outflow", "walls"])
@pytest.mark.parametrize("shape,passes,sweeps,monitor", [((33, 9, 14), 3, 2, "vdw"), ((32, 12, 8), 2, 3, "smooth"),
                                                         ((65, 8, 37), 1, 1, "vdw"), ((8, 31, 9), 5, 4, "smooth")])
def test_redistribution_3d(bc, shape, passes, sweeps, monitor):
    """The filter's warps of 32 nodes by two lines and segments of planes at their edges (one node over, whole, one
    short), and the sweeps with stored weights, every boundary."""
    from test_gpu_3d import _box
    w = _box(*shape, bc == "periodic", amp=0.0 if bc == "walls" else 0.2 / max(shape))
    if bc == "walls":
        w["bc"] = ("reflect", "symmetry_lo", "outflow")
    w["moving"] = True
    w["mesh"] = dict(monitor=monitor, alphas=(1200.0, 1200.0, 1200.0), kappa=2, filter_passes=passes, sweeps=sweeps,
                     eps=0.0)
    _compare(w)


@pytest.mark.parametrize("n", [76000, 380000])
def test_limiter_is_the_least_quotient(n):
    """Delta_gamma is the least of the nodes' quotients room/(2 |dx|), bit for bit, also where many differ by single ulps:
    the same 1D pattern of spacings in every binade from 2^-900 to 2^1000 (one launch of tiles; sweep by sweep), its scale
    varied a little, so that the blocks' quotients are equal but for rounding."""
    import torch

    from paper_2407_05568_gb300 import es
    rng = np.random.default_rng(4)
    blocks, P = 1900, n // 1900
    w = wl.riemann_1d("RP1", n)
    rho = np.tile(rng.uniform(0.3, 1.2, P), blocks)
    w.update(rho=rho, v=np.zeros((1, n)), p=np.full(n, 2.0), bc=("outflow",))
    w["mesh"] = dict(w["mesh"], filter_passes=0, sweeps=1, eps=0.0)
    ctx, JU, J, _ = gpu_setup(w)
    xo = torch.empty((1, n), dtype=torch.float64, device="cuda")
    xd = torch.empty_like(xo)
    q, r = torch.empty_like(xo[0]), torch.empty_like(xo[0])
    for _ in range(500):
        cuts = rng.uniform(0.0, 1.0, 10)                              # a few wide spacings
        at = np.sort(np.concatenate([cuts, rng.choice(cuts, P - 10) + 1e-4 * rng.uniform(size=P - 10)]))
        s = 1.0 + 0.04 * rng.uniform(size=blocks)
        x = (np.ldexp(s, np.arange(blocks) - 900)[:, None] * (1.05 + 0.8 * at)[None, :]).reshape(1, n)
        xt = torch.tensor(x, device="cuda")
        _, gam = es.es_mesh_redistribute(ctx, JU, J, xt, 1.0, xd)
        es.es_mesh_solve(ctx, JU, J, xt, None, xo)
        dx = (xo - xt)[0]
        right = torch.cat([xt[0, 1:], xt[0, -1:]]) - xt[0]
        left = xt[0] - torch.cat([xt[0, :1], xt[0, :-1]])
        two = torch.where(dx == 0, 1.0, 2.0 * dx.abs())
        es.es_selftest_division(torch.where(dx < 0, left, right), two, q, r)       # the kernels' quotient
        least = float(torch.where(dx == 0, 1.0, q).min())
        assert 0.0 < least < 1.0
        assert gam == least


@pytest.mark.parametrize("shape,bc", [((33, 15, 13), "periodic"), ((64, 8, 9), "walls"), ((8, 8, 8), "outflow"),
                                      ((81, 79, 77), "outflow"), ((97, 83, 79), "periodic"), ((97, 83, 79), "walls"),
                                      ((96, 84, 78), "outflow"), ((131, 127, 130), "walls"), ((131, 127, 130), "periodic")])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_3d_filter_kernels(shape, bc, precision):
    """The 3D filter's three forms (node by node; marching with two lines, and with four above 2^21 nodes) on whole and ragged
    meshes: the mesh velocity after two passes and a sweep against the oracle."""
    import torch

    from paper_2407_05568_gb300 import es
    from test_gpu_3d import _box
    if bc == "walls" and precision == "mixed":
        pytest.skip("walls: the FP64 form only")
    w = _box(*shape, bc == "periodic", amp=0.0 if bc == "walls" else 0.2 / max(shape))
    if bc == "walls":
        w["bc"] = ("symmetry_lo", "reflect", "outflow")
    w["moving"] = True
    w["mesh"] = dict(monitor="smooth", alphas=(20.0, 15.0), kappa=2, filter_passes=2, sweeps=1, eps=0.0)
    sch, mc, JU_o, J_o, x_o = oracle_setup(w)
    xd_o, _, gam_o = stepper.redistribute(sch, mc, JU_o, J_o, x_o, 1e-3)
    ctx, JU, J, xt = gpu_setup(w, precision=precision)
    xd = torch.empty_like(xt)
    _, gam = es.es_mesh_redistribute(ctx, JU, J, xt, 1e-3, xd)
    tol = 1e-11 if precision == "fp64" else 2e-5                     # the bounds of the forms' other redistributions
    assert abs(gam - gam_o) <= 10 * tol * gam_o
    assert np.abs(xd.cpu().numpy() - xd_o).max() <= tol * max(np.abs(xd_o).max(), 1e-3 * min(w["dxi"]) / 1e-3)


@pytest.mark.parametrize("bc", ["periodic", "outflow", "reflect", "symmetry_lo"])
@pytest.mark.parametrize("n,passes,sweeps", [(8, 64, 64), (9, 5, 3), (33, 64, 10), (100, 1, 1), (100, 65, 65), (511, 20, 64),
                                             (9728, 5, 4), (9729, 5, 4), (14592, 5, 5), (14593, 64, 5), (19456, 5, 9),
                                             (19457, 5, 9), (29184, 2, 10), (29185, 2, 10)])
def test_redistribution_1d(n, passes, sweeps, bc):
    """The line's tiles (filter passes, and sweeps, in one launch) and the pass-by-pass kernels at the edges of their ranges,
    periodic lines shorter than the halo among them.  A rough state: its second differences are of the size of their factors, so
    that their rounding stays that of the state.  The coordinates, of size 1, are rounded once a sweep; Delta_gamma divides
    such differences by a node's displacement, of a spacing's size."""
    import torch

    from paper_2407_05568_gb300 import es
    x, d = wl.uniform_nodes(n, 0.0, 1.0, bc == "periodic")
    w = wl.sine_1d(max(n, 8))
    w.update(bc=(bc,), x=x[None].copy(), dxi=(d,), moving=True)
    w["rho"], w["v"], w["p"] = wl.rough_state((n,), 5 + n, 1)
    w["mesh"] = dict(monitor="vdw", alphas=(1200.0, 1200.0, 1200.0), kappa=2, filter_passes=passes, sweeps=sweeps, eps=0.0)
    sch, mc, JU_o, J_o, x_o = oracle_setup(w)
    dt = 1e-3
    xd_o, sw_o, gam_o = stepper.redistribute(sch, mc, JU_o, J_o, x_o, dt)
    ctx, JU, J, xt = gpu_setup(w)
    xd = torch.empty_like(xt)
    sw, gam = es.es_mesh_redistribute(ctx, JU, J, xt, dt, xd)
    assert sw == sw_o
    assert abs(gam - gam_o) <= 1e-14 * (4 + sweeps) * n * gam_o
    assert np.abs(xd.cpu().numpy() - xd_o).max() * dt <= 1e-15 * (4 + sweeps)
