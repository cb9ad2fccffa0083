"""elder_residual (cell and edge sums in fixed point) against the allocation-free
entry point's residual (node by node in FP64) where the sums' common unit
matters: zeros, salt fractions over many decades, magnitudes below the fixed
point's range (summed in FP64), non-finite values, ragged grids."""
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


def _both(E, dims, c, c_old, seed, bc_mode=3):
    nx, ny, nz = dims
    N, C = (nx + 1) * (ny + 1) * (nz + 1), nx * ny * nz
    S = c.size // N
    rng = np.random.default_rng(seed)
    k = np.repeat(np.arange(nz + 1), (nx + 1) * (ny + 1))
    p = np.tile(1000.0 * 9.81 * (150.0 - k * 150.0 / nz), S) + rng.normal(0, 2e3, S * N)
    phi = 0.1 * np.exp(0.2 * rng.standard_normal(S * C))
    K = 4.845e-13 * (phi / 0.1) ** 3

    def T(a):
        return torch.tensor(np.ascontiguousarray(a).ravel(), dtype=torch.float64, device="cuda:0")

    cfg = E.elder_config_default(nx, ny, nz, max_samples=S, bc_mode=bc_mode)
    ctx = E.elder_create(cfg)
    a = [T(v) for v in (phi, K, p, c, p, c_old)]
    R = ctx.residual(S, *a, DT).cpu().numpy().reshape(S, N, 2)
    Rs, _ = E.elder_residual_norms_static(cfg, S, *a, DT)
    ctx.destroy()
    return R, Rs.cpu().numpy().reshape(S, N, 2)


# sums of up to 24 terms per row, each a few roundings at the scale of the
# largest term of the grid: 1e-12 of the largest entry per component
@pytest.mark.parametrize("dims,S", [((1, 1, 1), 3), ((5, 3, 2), 2), ((17, 9, 4), 3)])
@pytest.mark.parametrize("kind", ["uniform", "zero", "decades", "tiny"])
def test_matches_node_sums(E, dims, S, kind):
    N = (dims[0] + 1) * (dims[1] + 1) * (dims[2] + 1)
    rng = np.random.default_rng(N)
    c = {"uniform": rng.uniform(0, 1, S * N), "zero": np.zeros(S * N),
         "decades": 10.0 ** rng.uniform(-60, 0, S * N),
         "tiny": 10.0 ** rng.uniform(-306, -290, S * N)}[kind]
    c[rng.random(S * N) < 0.1] = 0.0
    R, Rs = _both(E, dims, c, 0.5 * c, N)
    for comp in (0, 1):
        scale = np.abs(Rs[..., comp]).max()
        assert np.abs(R[..., comp] - Rs[..., comp]).max() <= 1e-12 * scale, (comp, scale)


def test_nonfinite_values_stay_local_and_nonfinite(E):
    dims, S = (8, 8, 4), 1
    N = 9 * 9 * 5
    rng = np.random.default_rng(1)
    for bad in (np.nan, np.inf):
        c = rng.uniform(0, 1, N)
        c[N // 2] = bad
        R, Rs = _both(E, dims, c, c * 0.0, 2)
        assert np.array_equal(np.isfinite(R), np.isfinite(Rs))
        ok = np.isfinite(Rs)
        assert np.abs(R[ok] - Rs[ok]).max() <= 1e-12 * np.abs(Rs[ok]).max()
