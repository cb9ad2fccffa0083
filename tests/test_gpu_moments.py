"""Sample statistics at the edges of the kernel's split: fewer fields than the
threads of a node, a remainder, a last block of few nodes, equal and given
weights (zeros among them), values around the threshold of either sign."""
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


@pytest.mark.parametrize("dims", [(1, 1, 1), (3, 3, 3), (12, 9, 4)])  # 8, 64, 650 nodes
@pytest.mark.parametrize("S", [1, 2, 5, 32, 67])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("threshold", [0.5, 0.0, -0.25])
def test_moments(E, dims, S, weighted, threshold):
    ctx = E.elder_create(E.elder_config_default(*dims, bc_mode=2))
    rng = np.random.default_rng(S + dims[0])
    c = rng.uniform(-1, 1, (S, ctx.N))
    c[rng.random(c.shape) < 0.2] = threshold
    c[rng.random(c.shape) < 0.1] = -0.0
    w = np.full(S, 1.0 / S)
    if weighted:
        w = rng.random(S) * (rng.random(S) < 0.8)
        w[0] += 0.1
        w /= w.sum()

    def T(a):
        return torch.tensor(np.ascontiguousarray(a).ravel(), device="cuda:0")

    mean, var, pe = ctx.moments(S, T(c), w=T(w) if weighted else None, threshold=threshold)
    ctx.destroy()
    m = w @ c
    # sums of S terms of magnitude <= 4 (squares of differences), a few roundings
    # per term in either order
    tol = 8 * (S + 8) * 2.0**-53
    assert np.abs(mean.cpu().numpy() - m).max() <= tol
    assert np.abs(var.cpu().numpy() - w @ (c - m) ** 2).max() <= 4 * tol
    assert np.abs(pe.cpu().numpy() - w @ (c > threshold)).max() <= tol


def test_moments_of_nonfinite_values(E):
    ctx = E.elder_create(E.elder_config_default(1, 1, 1, bc_mode=2))
    c = np.zeros((4, 8))
    c[1, 0], c[1, 1], c[1, 2] = np.nan, np.inf, -np.inf
    t = torch.tensor(c.ravel(), device="cuda:0")
    mean, var, pe = (v.cpu().numpy() for v in ctx.moments(4, t, threshold=0.5))
    ctx.destroy()
    assert np.isnan(mean[0]) and pe[0] == 0.0 and pe[1] == 0.25 and pe[2] == 0.0
    assert (pe[3:] == 0).all() and (mean[3:] == 0).all()
