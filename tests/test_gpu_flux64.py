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
