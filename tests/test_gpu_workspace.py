"""Device memory of a context: elder_create takes what the calls need, so that a
call does not run out of memory in the middle of a run."""
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


def test_rows_of_the_mixed_solver_are_reserved_at_create(E):
    """The calls of a mixed context that need the finest level's assembled rows
    (27 blocks of 4 entries, FP32 and bfloat16: 648 bytes per node, 406 MB here)
    take no device memory of that size."""
    S = 64
    ctx = E.elder_create(E.elder_config_default(32, 32, 8, max_samples=S, precision=E.ELDER_MIXED))
    rows = 648 * ctx.N * S
    p, c = ctx.initial_state(S)
    phi = torch.full((S * ctx.C,), 0.1, dtype=torch.float64, device="cuda:0")
    K = torch.full_like(phi, 4.845e-13)
    rhs = torch.ones(2 * S * ctx.N, dtype=torch.float64, device="cuda:0")
    x = torch.empty_like(rhs)
    dt = E.SECONDS_PER_YEAR / 48
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for call in (lambda: ctx.solve(S, phi, K, p, c, dt, rhs, transpose=True, rtol=1e-4, x=x),
                 lambda: ctx.smoother_apply(S, phi, K, p, c, dt, E.ELDER_SMOOTH_JACOBI, rhs, z=x),
                 lambda: ctx.smoother_apply(S, phi, K, p, c, dt, E.ELDER_SMOOTH_ZLINE, rhs, z=x,
                                            transpose=True)):
        call()
        torch.cuda.synchronize()
        assert free - torch.cuda.mem_get_info()[0] < rows // 8
    ctx.destroy()
