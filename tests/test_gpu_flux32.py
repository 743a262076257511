"""The mixed form's 3D direction kernels (FP32 fluxes on double-float node values) in every pencil shape."""
import numpy as np
import pytest

from oracle import operator as op

from sides import oracle_setup
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
