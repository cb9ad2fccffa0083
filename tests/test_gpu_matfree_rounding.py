"""The matrix-free products to FP32 rounding: a mixed solve to the smallest tolerance
that stays with the FP32 solver (1e-6) meets the assembled rows to that tolerance and
the rounding of its vectors and products, under every boundary set."""
import pytest

from test_gpu_matfree import E, _product  # noqa: F401 (E: the module's fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RTOL = 1e-6


@pytest.mark.parametrize("dims,S", [((8, 8, 4), 3), ((32, 8, 10), 2), ((64, 32, 32), 1),
                                    ((32, 32, 8), 5)])
@pytest.mark.parametrize("bc", [0, 1, 2, 3])
def test_mixed_solve_to_rounding(E, dims, S, bc):  # noqa: F811
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
    # the FP32 vectors, coefficients and products: a few units of 2^-24 per term of
    # the row sums and per update of x
    bound = RTOL * b.norm(dim=1) + 30 * 2.0**-24 * m.norm(dim=1)
    ratio = (y - b).norm(dim=1) / bound
    assert (ratio <= 1).all(), ratio.max()
