"""Sample statistics of large values: the equal-weight moments are finite where
every weighted term and their sum are, although the plain sums overflow."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def E():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1906_01632_gb300 import build
    build.build()
    from paper_1906_01632_gb300 import elder
    return elder


@pytest.mark.parametrize("S", [2, 8, 67])
def test_sums_beyond_the_largest_double(E, S):
    ctx = E.elder_create(E.elder_config_default(1, 1, 1, bc_mode=2))
    c = np.ones((S, 8))
    c[:, 0] = 1e154   # squares of the differences from the first field: 1e308
    c[:, 1] = 1.7e308  # differences
    c[0, :2] = 0.0
    c[:, 2] = -1e154
    t = torch.tensor(c.ravel(), device="cuda:0")
    mean, var, pe = (v.cpu().numpy() for v in ctx.moments(S, t, threshold=0.5))
    ctx.destroy()
    q = (S - 1) / S
    # sums of S terms, a few roundings per term, at the scale of the terms
    tol = 8 * (S + 8) * 2.0**-53
    assert abs(mean[0] / 1e154 - q) <= tol and abs(var[0] / 1e308 - q / S) <= 4 * tol
    assert abs(mean[1] / 1.7e308 - q) <= tol
    assert mean[2] == -1e154 and var[2] == 0.0
    assert (mean[3:] == 1.0).all() and (var[3:] == 0.0).all()
    assert abs(pe[0] - q) < 1e-15 and abs(pe[1] - q) < 1e-15 and pe[2] == 0.0
