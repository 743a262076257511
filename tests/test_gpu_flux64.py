"""The FP64 operator's table-driven logarithm."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_table_log_within_two_ulp():
    """Values over the whole range, the states' range and close to 1 (both sides, where the logarithm is small and must
    keep its relative accuracy), table boundaries, and the arguments that take the library's log(): within 2 ulp of
    numpy's logarithm plus its own half ulp."""
    import torch

    from paper_2407_05568_gb300 import es
    rng = np.random.default_rng(5)
    n = 200_000
    x = np.concatenate([np.exp(rng.uniform(-700.0, 700.0, n)), rng.uniform(0.01, 4.0, n),
                        1.0 + rng.uniform(-1.0, 1.0, n) * np.exp(-30.0 * rng.uniform(size=n)),
                        np.ldexp(1.0 + np.arange(256) / 256.0, -1), np.nextafter(1.0 + np.arange(128) / 128.0, 0.0),
                        [1.0, np.nextafter(1.0, 2.0), 2.0, 0.5, 5e-324, 1e-310, 2.3e-308, np.finfo(float).max]])
    y = torch.empty(x.size, dtype=torch.float64, device="cuda")
    es.es_selftest_log(torch.tensor(x, device="cuda"), y)
    got, ref = y.cpu().numpy(), np.log(x)
    assert got[x == 1.0][0] == 0.0
    assert np.all(np.abs(got - ref) <= 2.5 * np.spacing(np.abs(ref)))


def test_table_log_keeps_the_last_bit():
    """Within 1 ulp of the logarithm in extended precision: the table's constants carry the bits past the double, so one
    rounding of the result's size is left and those of the reduced argument, up to 2^-60 where a result is 2^-7 or more.
    The logarithmic mean of close values divides a difference of two logarithms by as little as 2e-2."""
    import torch

    from paper_2407_05568_gb300 import es
    rng = np.random.default_rng(8)
    n = 400_000
    x = np.concatenate([np.exp(rng.uniform(-700.0, 700.0, n)), rng.uniform(0.01, 4.0, n), 1.0 + rng.uniform(-0.3, 0.3, n)])
    y = torch.empty(x.size, dtype=torch.float64, device="cuda")
    es.es_selftest_log(torch.tensor(x, device="cuda"), y)
    ref = np.log(x.astype(np.longdouble))
    ulp = np.spacing(np.abs(ref.astype(np.float64)))
    off = np.abs(y.cpu().numpy().astype(np.longdouble) - ref) / ulp
    assert off.max() <= 1.0
    # rounding to nearest spreads evenly over half an ulp each way: 0.289 in the mean square, the reduced argument adds little
    assert np.sqrt(np.mean(off.astype(np.float64) ** 2)) <= 0.31


@pytest.mark.parametrize("n", [8, 9, 15, 16, 17, 200, 2432, 2433, 2500, 65536, 65537])
@pytest.mark.parametrize("bc", ["periodic", "outflow", "reflect", "symmetry_lo"])
def test_1d_stage_shapes_vs_oracle(n, bc):
    """The three 1D shapes of the FP64 stage kernel (8-node lines shared by four warps, 62- and 254-node tiles) at the
    edges of their ranges and of their tiles: the right-hand sides of a rough state with a moving mesh, and an RK stage,
    against the oracle to 1e-12 of their size, with the EC flux alone too."""
    import torch

    from oracle import operator as op
    from oracle import stepper
    from paper_2407_05568_gb300 import es
    from paper_2407_05568_gb300 import workloads as wl
    from sides import gpu_setup, oracle_setup
    x, d = wl.uniform_nodes(n, 0.0, 1.0, bc == "periodic")
    w = wl.sine_1d(max(n, 8))
    w.update(bc=(bc,), x=x[None].copy(), dxi=(d,))
    w["rho"], w["v"], w["p"] = wl.rough_state((n,), 3 + n, 1)
    xdot = 0.05 * np.sin(2 * np.pi * x + 0.3)[None]
    if bc != "periodic":
        xdot[:, [0, -1]] = 0.0
    for diss in (True, False):
        sch, _, JU_o, J_o, x_o = oracle_setup(w, dissipation=diss)
        dU_o, dJ_o = op.rhs(sch, JU_o, J_o, x_o, xdot)
        ctx, JU, J, xt = gpu_setup(w, dissipation=diss)
        xd = torch.tensor(xdot, device="cuda")
        dU, dJ = torch.empty_like(JU), torch.empty_like(J)
        es.es_rhs(ctx, JU, J, xt, xd, dU, dJ)
        dt = 0.1 * d
        U1, J1 = torch.empty_like(JU), torch.empty_like(J)
        es.es_rk_stage(ctx, 2, dt, JU, J, JU, J, xt, xd, U1, J1)
        assert es.es_check(ctx) == 0, es.es_last_error(ctx)
        U1_o, J1_o = stepper.rk_stage(sch, 1, dt, JU_o, J_o, JU_o, J_o, x_o, xdot)
        for c in range(3):
            flux = np.abs(JU_o[c]).max() * 4.0 / d                  # the size of a flux difference
            assert np.abs(dU.cpu().numpy()[c] - dU_o[c]).max() < 1e-12 * flux
        assert np.abs(dJ.cpu().numpy() - dJ_o).max() < 1e-12 / d
        assert np.abs(U1.cpu().numpy() - U1_o).max() < 1e-12 * np.abs(U1_o).max()
        assert np.abs(J1.cpu().numpy() - J1_o).max() < 1e-12 * np.abs(J1_o).max()


@pytest.mark.parametrize("n1,n2", [(8, 8), (9, 17), (41, 23), (200, 100), (300, 101)])
@pytest.mark.parametrize("bc", [("periodic", "outflow"), ("reflect", "symmetry_lo")])
def test_2d_small_mesh_shapes(n1, n2, bc):
    """The five shapes of meshes that one wave covers (8 x 8 to 20 x 10 nodes), whole and ragged, and the first size past it:
    right-hand sides of a rough state against the oracle to 1e-12 of a flux difference, the same bits from every shape."""
    import torch

    from oracle import operator as op
    from paper_2407_05568_gb300 import es
    from paper_2407_05568_gb300 import workloads as wl
    from sides import oracle_setup
    x1, d1 = wl.uniform_nodes(n1, 0.0, 1.0, bc[0] == "periodic")
    x2, d2 = wl.uniform_nodes(n2, 0.0, 1.0, bc[1] == "periodic")
    X, Y = np.meshgrid(x1, x2)
    w = wl.sine_2d(16)
    w.update(bc=bc, x=np.stack([X, Y]), dxi=(d1, d2), n=(n2, n1))
    w["rho"], w["v"], w["p"] = wl.rough_state((n2, n1), 3 + n1, 2)
    sch, _, JU_o, J_o, x_o = oracle_setup(w)
    dU_o, dJ_o = op.rhs(sch, JU_o, J_o, x_o, np.zeros_like(x_o))
    outs = []
    for tile in (1, 2, 3, 4, 5):
        ctx = es.es_create(es.make_params(w, tile=tile))
        xt = torch.tensor(np.ascontiguousarray(w["x"]), device="cuda")
        J = torch.empty((n2, n1), dtype=torch.float64, device="cuda")
        es.es_init_mesh(ctx, xt, J)
        JU = torch.empty((4, n2, n1), dtype=torch.float64, device="cuda")
        es.es_prim_to_cons(ctx, torch.tensor(w["rho"], device="cuda"), torch.tensor(w["v"], device="cuda"),
                           torch.tensor(w["p"], device="cuda"), J, JU)
        dU, dJ = torch.empty_like(JU), torch.empty_like(J)
        es.es_rhs(ctx, JU, J, xt, None, dU, dJ)
        assert es.es_check(ctx) == 0, es.es_last_error(ctx)
        outs.append((dU.cpu().numpy(), dJ.cpu().numpy()))
    for c in range(4):
        flux = np.abs(JU_o[c]).max() * 4.0 / min(d1, d2)
        assert np.abs(outs[0][0][c] - dU_o[c]).max() < 1e-12 * flux
    for o in outs[1:]:
        assert np.array_equal(o[0], outs[0][0]) and np.array_equal(o[1], outs[0][1])


def _large_mesh(case):
    """Meshes that 20 x 10 tiles cover with more than 152 tiles: the five shapes of large meshes."""
    from paper_2407_05568_gb300 import workloads as wl
    from test_gpu_parity import _ragged_riemann
    if case == "riemann":
        w = _ragged_riemann(230, 170, seed=6)
        w["xdot"] = np.zeros_like(w["x"])
        return w
    if case == "wavy":
        w = wl.sine_2d(188)
        X, Y = w["x"]
        w["x"], w["xdot"] = wl.wavy_mesh_2d(X, Y), wl.mesh_velocity_2d(X, Y)
        w["rho"], w["v"], w["p"] = wl.rough_state(X.shape, 11, 2)
        return w
    x1, d1 = wl.uniform_nodes(201, 0.0, 1.0, False)
    x2, d2 = wl.uniform_nodes(183, 0.0, 1.0, False)
    X, Y = np.meshgrid(x1, x2)
    w = wl.sine_2d(16)
    w.update(bc=("symmetry_lo", "reflect"), x=np.stack([X, Y]), dxi=(d1, d2), n=(183, 201))
    w["rho"], w["v"], w["p"] = wl.rough_state((183, 201), 5, 2)
    w["xdot"] = 0.05 * np.stack([np.sin(np.pi * X) * np.cos(np.pi * Y), np.sin(np.pi * Y) * np.cos(np.pi * X)])
    w["xdot"][0][:, [0, -1]] = w["xdot"][1][[0, -1]] = 0.0
    w["xdot"][1][:, -1] = 0.0
    return w


@pytest.mark.parametrize("dissipation", [True, False])
@pytest.mark.parametrize("case", ["riemann", "wavy", "walls"])
def test_2d_large_mesh_shapes(case, dissipation):
    """The five shapes of large 2D meshes (among them 32 x 12 nodes, whose directions follow one another): right-hand sides
    and an RK stage with curved metrics and a mesh velocity, the same bits from every shape, and the first against the oracle
    (the bounds of the other parity tests)."""
    import torch

    from oracle import operator as op
    from oracle import stepper
    from paper_2407_05568_gb300 import es
    from sides import gpu_setup, oracle_setup, rel_l1
    w = _large_mesh(case)
    assert -(-w["n"][1] // 20) * -(-w["n"][0] // 10) > 152
    sch, _, JU_o, J_o, x_o = oracle_setup(w, dissipation=dissipation)
    dU_o, dJ_o = op.rhs(sch, JU_o, J_o, x_o, w["xdot"])
    dt = 0.1 * min(w["dxi"])
    U1_o, J1_o = stepper.rk_stage(sch, 1, dt, JU_o, J_o, JU_o, J_o, x_o, w["xdot"])
    _, JU, J, xt = gpu_setup(w, dissipation=dissipation)
    xd = torch.tensor(np.ascontiguousarray(w["xdot"]), dtype=torch.float64, device="cuda")
    outs = []
    for tile in (1, 2, 3, 4, 5):
        ctx = es.es_create(es.make_params(w, dissipation=dissipation, tile=tile))
        out = [torch.empty_like(a) for a in (JU, J, JU, J)]
        es.es_rhs(ctx, JU, J, xt, xd, out[0], out[1])
        es.es_rk_stage(ctx, 2, dt, JU, J, JU, J, xt, xd, out[2], out[3])
        assert es.es_check(ctx) == 0, es.es_last_error(ctx)
        outs.append(out)
    for out in outs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(out, outs[0]))
    dU, dJ, U1, J1 = [a.cpu().numpy() for a in outs[0]]
    h = min(w["dxi"])
    assert np.abs(dU - dU_o).sum() < 1e-12 * np.abs(JU_o).sum() / h
    assert np.abs(dJ - dJ_o).sum() < 1e-12 * np.abs(J_o).sum() / h
    assert rel_l1(U1, U1_o) < 1e-12 and rel_l1(J1, J1_o) < 1e-12


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("shape", [(200,), (3000,), (40, 36), (230, 170)])
def test_nan_state_is_reported_and_stays_local(shape, precision):
    """A NaN in the density or the energy of one node: the state is refused, and right-hand sides out of the stencil's reach
    (three nodes along each direction) are those without it."""
    import torch

    from paper_2407_05568_gb300 import es
    from paper_2407_05568_gb300 import workloads as wl
    from sides import gpu_setup
    w = wl.sine_1d(shape[0]) if len(shape) == 1 else wl.sine_2d(16)
    if len(shape) == 2:
        x1, d1 = wl.uniform_nodes(shape[1], 0.0, 1.0, True)
        x2, d2 = wl.uniform_nodes(shape[0], 0.0, 1.0, True)
        w.update(x=np.stack(np.meshgrid(x1, x2)), dxi=(d1, d2), n=shape)
    w["rho"], w["v"], w["p"] = wl.rough_state(shape, 7, len(shape))
    ctx, JU, J, xt = gpu_setup(w, precision=precision)
    clean = [torch.empty_like(JU), torch.empty_like(J)]
    es.es_rhs(ctx, JU, J, xt, None, *clean)
    assert es.es_check(ctx) == 0
    at = tuple(s // 3 for s in shape)
    far = np.ones(shape, bool)
    for k in range(len(shape)):
        cut = list(at)
        cut[k] = slice(at[k] - 3, at[k] + 4)
        far[tuple(cut)] = False
    far = torch.tensor(far, device="cuda")
    for c in (0, len(shape) + 1):
        bad = JU.clone()
        (bad if precision == "fp64" else bad[0])[(c,) + at] = float("nan")
        dU, dJ = torch.empty_like(JU), torch.empty_like(J)
        es.es_rhs(ctx, bad, J, xt, None, dU, dJ)
        assert es.es_check(ctx) == es.ES_ERR_INADMISSIBLE
        assert torch.equal(dU[..., far], clean[0][..., far])
        assert bool(torch.isnan(dU[(..., c) + at] if precision == "fp64" else dU[(0, c) + at]).all())


@pytest.mark.parametrize("power", [-90, 90])
@pytest.mark.parametrize("shape", [(64,), (200, 24), (9, 10, 11)])
def test_units_of_extreme_size(shape, power):
    """A flow in units in which velocities are 2^+-90 times the usual ones (energies leave the range of FP32, in whose bounds the
    sign switch decides the clear cases): right-hand sides against the oracle to 1e-12 of a flux difference."""
    import torch

    from oracle import operator as op
    from paper_2407_05568_gb300 import es
    from paper_2407_05568_gb300 import workloads as wl
    from sides import gpu_setup, oracle_setup
    dim, u = len(shape), 2.0 ** power
    if dim == 3:
        from test_gpu_3d import _box
        w = _box(*shape[::-1], True, amp=0.005)
    else:
        w = wl.sine_1d(shape[0]) if dim == 1 else wl.sine_2d(16)
        if dim == 2:
            x1, d1 = wl.uniform_nodes(shape[1], 0.0, 1.0, True)
            x2, d2 = wl.uniform_nodes(shape[0], 0.0, 1.0, True)
            w.update(x=np.stack(np.meshgrid(x1, x2)), dxi=(d1, d2), n=shape)
    w["rho"], w["v"], w["p"] = wl.rough_state(shape, 7, dim)
    g = w["gas"]
    w.update(gas=dict(a=g["a"] * u * u, b=g["b"], R=g["R"] * u * u, cv=g["cv"] * u * u), v=w["v"] * u, p=w["p"] * u * u)
    sch, _, JU_o, J_o, x_o = oracle_setup(w)
    dU_o, _ = op.rhs(sch, JU_o, J_o, x_o, np.zeros_like(x_o))
    ctx, JU, J, xt = gpu_setup(w)
    dU, dJ = torch.empty_like(JU), torch.empty_like(J)
    es.es_rhs(ctx, JU, J, xt, None, dU, dJ)
    assert es.es_check(ctx) == 0, es.es_last_error(ctx)
    for c in range(dim + 2):
        flux = np.abs(JU_o[c]).max() * u * 4.0 / min(w["dxi"])
        assert np.abs(dU[c].cpu().numpy() - dU_o[c]).max() < 1e-12 * flux
