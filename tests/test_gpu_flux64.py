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
