"""elder_profile_read counts the work of the kernels that run: floating-point
operations of the residual with integer sums and of the line blocks, bytes of the
sweep with three line factors."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DIMS = (32, 16, 8)


@pytest.fixture(scope="module")
def E():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1906_01632_gb300 import build
    build.build()
    from paper_1906_01632_gb300 import elder
    return elder


def _profile(E, precision):
    """{class: (launches, bytes, flops)} of one step of one sample, and the levels'
    node counts."""
    ctx = E.elder_create(E.elder_config_default(*DIMS, precision=precision, bc_mode=2))
    p, c = ctx.initial_state(1)
    phi = torch.full((ctx.C,), 0.1, dtype=torch.float64, device="cuda:0")
    K = torch.full_like(phi, 4.845e-13)
    ctx.profile(True)
    ctx.step(1, phi, K, p, c, E.SECONDS_PER_YEAR / 48)
    ctx.profile(False)
    prof = {k: ctx.profile_read(k) for k in E.KERNEL_CLASSES}
    nodes = [(DIMS[0] // 2**l + 1) * (DIMS[1] // 2**l + 1) * (DIMS[2] // 2**l + 1)
             for l in range(ctx.levels)]
    ctx.destroy()
    return prof, nodes


def _is_multiple(total, one, most):
    """total is n times one, 1 <= n <= most (a launch without an active sample counts 0)."""
    n = round(total / one)
    assert 1 <= n <= most and total == pytest.approx(n * one, rel=1e-9), (total / one, most)


def test_mixed(E):
    prof, nodes = _profile(E, E.ELDER_MIXED)
    levels, C = len(nodes), DIMS[0] * DIMS[1] * DIMS[2]
    r, j, z = (prof[k] for k in (E.K_RESIDUAL, E.K_JACOBIAN, E.K_SMOOTH0))
    _is_multiple(r["flops"], 110 * C + 67 * nodes[0], r["launches"])
    _is_multiple(j["flops"], 1722 * nodes[0] + 2890 * sum(nodes[1:]), j["launches"] / levels)
    # every cycle sweeps each level but the coarsest once
    _is_multiple(z["bytes"], 65 * sum(nodes[:-1]), z["launches"] / (levels - 1))


def test_fp64(E):
    prof, nodes = _profile(E, E.ELDER_FP64)
    C = DIMS[0] * DIMS[1] * DIMS[2]
    r, j = prof[E.K_RESIDUAL], prof[E.K_JACOBIAN]
    _is_multiple(r["flops"], 266 * C + 75 * nodes[0], r["launches"])
    _is_multiple(j["flops"], 2890 * sum(nodes), j["launches"] / len(nodes))


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("smoother", ["zline", "jacobi", "ilu"])
@pytest.mark.parametrize("levels", [0, 1])
def test_bench_model_is_the_library_s(E, precision, smoother, levels):
    """bench.launch_model_bytes of the finest level against the bytes counted: the
    Krylov products run there only; on a single-level grid so does the assembly
    (with rows: a matrix-free level lies above a coarser one)."""
    import argparse

    import bench
    dims = (6, 4, 2)
    a = argparse.Namespace(precision=precision, smoother=smoother, grid=list(dims))
    ctx = E.elder_create(E.elder_config_default(
        *dims, precision=E.ELDER_MIXED if precision == "mixed" else E.ELDER_FP64, bc_mode=2,
        mg_levels=levels,
        smoother={"zline": E.ELDER_SMOOTH_ZLINE, "jacobi": E.ELDER_SMOOTH_JACOBI,
                  "ilu": E.ELDER_SMOOTH_ILU}[smoother]))
    assert ctx.levels == (1 if levels else 2)
    p, c = ctx.initial_state(1)
    phi = torch.full((ctx.C,), 0.1, dtype=torch.float64, device="cuda:0")
    ctx.profile(True)
    ctx.step(1, phi, torch.full_like(phi, 4.845e-13), p, c, E.SECONDS_PER_YEAR / 48)
    ctx.profile(False)
    spmv, jac = ctx.profile_read(E.K_SPMV), ctx.profile_read(E.K_JACOBIAN)
    ctx.destroy()
    if levels == 0:
        _is_multiple(spmv["bytes"], bench.launch_model_bytes(a, "spmv") * 105, spmv["launches"])
    elif smoother != "ilu":  # (no ILU factors on the coarsest level)
        a.smoother = "jacobi"  # the rows' model
        _is_multiple(jac["bytes"], bench.launch_model_bytes(a, "jacobian") * 105, jac["launches"])
