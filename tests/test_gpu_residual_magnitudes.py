"""elder_residual where the corners of p of a cell differ so much that its sums are
formed in FP64 beside the fixed-point sums of c (and the other way round), against
the allocation-free entry point's residual (node by node in FP64)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DT = 365.25 * 86400.0 / 12


@pytest.fixture(scope="module")
def E():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1906_01632_gb300 import build
    build.build()
    from paper_1906_01632_gb300 import elder
    return elder


def _both(E, dims, p, c, seed):
    nx, ny, nz = dims
    N, C = (nx + 1) * (ny + 1) * (nz + 1), nx * ny * nz
    rng = np.random.default_rng(seed)
    phi = 0.1 * np.exp(0.2 * rng.standard_normal(C))
    K = 4.845e-13 * (phi / 0.1) ** 3

    def T(a):
        return torch.tensor(np.ascontiguousarray(a).ravel(), dtype=torch.float64, device="cuda:0")

    cfg = E.elder_config_default(nx, ny, nz, bc_mode=3)
    ctx = E.elder_create(cfg)
    a = [T(v) for v in (phi, K, p, c, p, 0.5 * c)]
    R = ctx.residual(1, *a, DT).cpu().numpy().reshape(N, 2)
    Rs, _ = E.elder_residual_norms_static(cfg, 1, *a, DT)
    ctx.destroy()
    return R, Rs.cpu().numpy().reshape(N, 2)


# sums of up to 24 faces and the storage term per row, a few roundings each at the
# scale of the largest term of the grid (not of the residual, in which a hydrostatic
# pressure's terms cancel): 200 units of 2^-53 of the largest term
@pytest.mark.parametrize("dims", [(1, 1, 1), (5, 3, 2), (17, 9, 4), (40, 3, 6)])
@pytest.mark.parametrize("kind", ["top layer", "decades", "zeros", "equal", "tiny c"])
def test_matches_node_sums(E, dims, kind):
    nx, ny, nz = dims
    N = (nx + 1) * (ny + 1) * (nz + 1)
    rng = np.random.default_rng(N)
    k = np.repeat(np.arange(nz + 1), (nx + 1) * (ny + 1))
    p = 1000.0 * 9.81 * (150.0 - k * 150.0 / nz)
    c = rng.uniform(0, 1, N)
    if kind == "top layer":
        p = p + np.where(k == nz, rng.normal(0, 50.0, N), rng.normal(0, 2e3, N))
    elif kind == "decades":
        p = 10.0 ** rng.uniform(-30, 6, N) * np.where(rng.random(N) < 0.3, -1.0, 1.0)
    elif kind == "zeros":
        p = np.where(rng.random(N) < 0.5, 0.0, p)
    elif kind == "equal":
        p = np.full(N, 1.5e6)
    else:
        c = 10.0 ** rng.uniform(-306, -290, N)
    R, Rs = _both(E, dims, p, c, N)
    h = np.array([600.0 / nx, 600.0 / ny, 150.0 / nz])
    shape = 0.25 * h.prod() / h**2  # a quarter face's area over its edge
    rho, K = 1200.0, 4.845e-13 * 8.0  # (largest porosity: below 0.2)
    m = rho * K / 1e-3 * (shape * (np.abs(p).max() + rho * 9.81 * h)).max()
    F = np.abs(c).max() * (m + rho * 0.2 * (3.565e-6 * shape.max() + h.prod() / DT))
    # (one grid of one cell has at least one term of this size; storage of water
    # changes with c too)
    for comp, term in ((0, m + 200.0 * 0.2 * np.abs(c).max() * h.prod() / DT), (1, F)):
        assert np.abs(R[..., comp] - Rs[..., comp]).max() <= 200 * 2.0**-53 * term, (comp, term)


def test_nonfinite_pressures_stay_local_and_nonfinite(E):
    dims = (8, 8, 4)
    N = 9 * 9 * 5
    rng = np.random.default_rng(1)
    for value in (np.nan, np.inf):
        p = 1e6 + rng.normal(0, 2e3, N)
        p[N // 2] = value
        R, Rs = _both(E, dims, p, rng.uniform(0, 1, N), 2)
        assert np.array_equal(np.isfinite(R), np.isfinite(Rs))
        ok = np.isfinite(Rs)
        assert np.abs(R[ok] - Rs[ok]).max() <= 1e-12 * np.abs(Rs[ok]).max()
