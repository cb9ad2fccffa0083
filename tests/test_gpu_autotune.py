"""The autotuner times the z-line sweep on the level it is tuned for."""
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


def test_sweep_is_timed_on_the_finest_level(E):
    """A sweep from x = 0 over 64x64x16 cells x 128 samples moves 64 bytes per node
    (three line factors, b and x in FP32): 588 MB, of which the 129 MB L2 can hold
    what the launch before left.  No launch moves the rest faster than the 7.9 TB/s
    of the memory, 58 us; the next level's sweep is an eighth of that."""
    S = 128
    ctx = E.elder_create(E.elder_config_default(64, 64, 16, max_samples=S,
                                                precision=E.ELDER_MIXED))
    p, c = ctx.initial_state(S)
    phi = torch.full((S * ctx.C,), 0.1, dtype=torch.float64, device="cuda:0")
    K = torch.full_like(phi, 4.845e-13)
    ctx.step(S, phi, K, p, c, E.SECONDS_PER_YEAR / 48)
    choice = ctx.autotune_choice(E.K_SMOOTH0)
    ctx.destroy()
    ms = [v for v in choice[2] if v > 0]
    least = (64 * 71825 * S - 129e6) / 7.9e12 * 1e3
    assert len(ms) == 3 and min(ms) >= least, (choice, least)
