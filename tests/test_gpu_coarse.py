"""The dense inverse of the coarsest grid at the sizes where its kernels change:
on a grid that does not coarsen, the V-cycle is that inverse alone, so that
BiCGStab ends after one or two iterations (FP64; the cap of 6 fails a wrong
inverse), or as many as the bfloat16 rounding of the matrix asks for (mixed)."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DT = O.SECONDS_PER_YEAR / 12


@pytest.fixture(scope="module")
def E():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1906_01632_gb300 import build
    build.build()
    from paper_1906_01632_gb300 import elder
    return elder


def T(a):
    return torch.tensor(np.ascontiguousarray(a).ravel(), dtype=torch.float64, device="cuda:0")


# unknowns: 16 (fewer than a warp), 96, 108 | 120, 180 | 252, 432 | 480, 1200 (FP32
# registers of 7 x 16 and 12 x 16 a side; FP64 shares in shared memory up to
# about 440)
@pytest.mark.parametrize("dims", [(1, 1, 1), (5, 3, 1), (5, 2, 2), (4, 3, 2), (5, 4, 2), (6, 5, 2),
                                  (7, 8, 2), (7, 9, 2), (9, 9, 5)])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("transpose", [False, True])
def test_single_level_solve(E, dims, precision, transpose):
    P = O.Problem(*dims, bc_mode=2)
    S = 2
    rng = np.random.default_rng(sum(dims))
    p0, c0 = O.initial_state(P)
    phi = 0.1 * np.exp(0.2 * rng.standard_normal((S, P.C)))
    K = 4.845e-13 * (phi / 0.1) ** 3
    p = p0 + rng.normal(0, 2e3, (S, P.N))
    c = np.clip(c0 + rng.uniform(0, 0.5, (S, P.N)), 0, 1)
    rhs = rng.standard_normal((S, P.N, 2))
    rtol, maxit = (1e-12, 6) if precision == 0 else (1e-5, 60)
    ctx = E.elder_create(E.elder_config_default(*dims, max_samples=S, bc_mode=2, mg_levels=1,
                                                precision=precision, lin_maxit=maxit))
    assert ctx.levels == 1
    x, st = ctx.solve(S, T(phi), T(K), T(p), T(c), DT, T(rhs), transpose=transpose, rtol=rtol)
    ctx.destroy()
    assert (st == 0).all(), st
    x = x.cpu().numpy().reshape(S, 2 * P.N)
    for s in range(S):
        A = O.jacobian_dense(P, phi[s], K[s], p[s], c[s], DT)
        A = A.T if transpose else A
        if precision == 0:
            # against a dense LU, each component to 1e-9 of its largest value
            ref = O.dense_solve(A, rhs[s].ravel())
            scale = np.abs(ref).reshape(-1, 2).max(axis=0)
            err = np.abs(x[s] - ref).reshape(-1, 2).max(axis=0)
            assert (err <= 1e-9 * scale).all(), (err, scale)
        else:
            # the solver bounds the residual's 2-norm by rtol ||b||; the FP32
            # vectors and products add their rounding
            r = A @ x[s] - rhs[s].ravel()
            fp32 = 30 * 2.0**-24 * (np.abs(A) @ np.abs(x[s]))
            assert np.linalg.norm(r) <= 20 * rtol * np.linalg.norm(rhs[s]) + np.linalg.norm(fp32), s
