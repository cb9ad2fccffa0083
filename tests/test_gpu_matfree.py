"""The matrix-free products of the mixed solver's finest level against the rows
that elder_jacobian assembles (themselves checked against the oracle), on
grids at the edges of the product's tiles: fewer columns than a warp, one and
several tiles along x and z, a last tile of few columns, chunks of rows, odd
batches.  A solve by these products to rtol leaves a residual of the assembled
system within rtol ||b|| and FP32 rounding only if both are the same matrix."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RTOL = 1e-4


@pytest.fixture(scope="module")
def E():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1906_01632_gb300 import build
    build.build()
    from paper_1906_01632_gb300 import elder
    return elder


def _product(J, x, dims, S):
    """Sum over the 27 slots of J[S][27][N][4] times x[S][N][2], and of the magnitudes."""
    nx, ny, nz = dims
    shape = (S, nz + 1, ny + 1, nx + 1)
    J = J.reshape(S, 27, *shape[1:], 2, 2)
    xp = torch.zeros(S, nz + 3, ny + 3, nx + 3, 2, dtype=x.dtype, device=x.device)
    xp[:, 1:-1, 1:-1, 1:-1] = x.reshape(*shape, 2)
    y = torch.zeros(*shape, 2, dtype=x.dtype, device=x.device)
    m = torch.zeros_like(y)
    for s in range(27):
        dx, dy, dz = s % 3, s // 3 % 3, s // 9
        v = xp[:, dz:dz + nz + 1, dy:dy + ny + 1, dx:dx + nx + 1]
        t = J[:, s] * v[..., None, :]
        y += t.sum(-1)
        m += t.abs().sum(-1)
    return y.reshape(S, -1), m.reshape(S, -1)


@pytest.mark.parametrize("dims,S", [((4, 4, 2), 3), ((8, 6, 4), 2), ((30, 6, 10), 2),
                                    ((6, 64, 2), 1), ((64, 8, 64), 1), ((32, 32, 8), 37)])
@pytest.mark.parametrize("bc", [2, 3])
def test_mixed_solve_meets_the_assembled_system(E, dims, S, bc):
    nx, ny, nz = dims
    N, C = (nx + 1) * (ny + 1) * (nz + 1), nx * ny * nz
    g = torch.Generator(device="cuda:0").manual_seed(nx + ny + nz + bc)

    def rand(n):
        return torch.rand(n, generator=g, dtype=torch.float64, device="cuda:0")

    k = torch.arange(N, device="cuda:0") // ((nx + 1) * (ny + 1))
    p = (1000.0 * 9.81 * 150.0 * (1.0 - k.double() / nz)).repeat(S) + 2e3 * (rand(S * N) - 0.5)
    c = 0.5 * rand(S * N)
    phi = 0.08 + 0.04 * rand(S * C)
    K = 4.845e-13 * (phi / 0.1) ** 3
    rhs = 2.0 * rand(2 * S * N) - 1.0
    dt = E.SECONDS_PER_YEAR / 48
    ctx = E.elder_create(E.elder_config_default(nx, ny, nz, max_samples=S, bc_mode=bc,
                                                precision=E.ELDER_MIXED, lin_maxit=400))
    assert ctx.levels > 1
    x, st = ctx.solve(S, phi, K, p, c, dt, rhs, rtol=RTOL)
    J = ctx.jacobian(S, phi, K, p, c, dt)
    ctx.destroy()
    assert (st == 0).all(), st
    y, m = _product(J, x, dims, S)
    b = rhs.reshape(S, -1)
    # rounding of the FP32 solution, vectors and products: a few units of
    # 2^-24 per term of the row sums and per update
    bound = RTOL * b.norm(dim=1) + 30 * 2.0**-24 * m.norm(dim=1)
    assert ((y - b).norm(dim=1) <= 2 * bound).all(), ((y - b).norm(dim=1) / bound).max()
