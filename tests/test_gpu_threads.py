"""Calls of two host threads whose kernels are the same but ask for different
amounts of dynamic shared memory: the limit is one value per kernel and device, so
a launch must not lower it for another thread between that thread's setting and
its launch (the launch would be rejected)."""
import threading

import numpy as np
import pytest

import oracle.gpc as G
import oracle as O

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


def _together(*calls):
    """Runs every call in its own thread, all at once; re-raises a failure."""
    gate = threading.Barrier(len(calls))
    errors = []

    def body(call):
        try:
            gate.wait()
            call()
        except Exception as e:  # noqa: BLE001 (handed to the main thread)
            errors.append(e)

    threads = [threading.Thread(target=body, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    if errors:
        raise errors[0]


def T(a):
    return torch.tensor(np.ascontiguousarray(a).ravel(), dtype=torch.float64, device="cuda:0")


def test_projections_of_different_tables(E):
    # tables of 35 KiB, 61 KiB and 97 KiB of one kernel
    beta = torch.tensor(G.multi_indices(3, 4), dtype=torch.int32, device="cuda:0")
    rng = np.random.default_rng(5)
    work = []
    for Nq in (125, 216, 343):
        th, w = T(rng.uniform(-1, 1, (Nq, 3))).reshape(Nq, 3), T(rng.uniform(0, 8 / Nq, Nq))
        u = T(rng.uniform(0, 1, (Nq, 40))).reshape(Nq, 40)
        work.append((th, w, u, E.elder_gpc_project(beta, th, w, u)[0].clone()))
    torch.cuda.synchronize()

    def calls(th, w, u, first):
        def body():
            # (the C call alone: the binding's host work would keep the threads apart)
            coef, mean = torch.empty_like(first), torch.empty(40, dtype=torch.float64, device="cuda:0")
            var = torch.empty_like(mean)
            a = (3, 35, beta.data_ptr(), 4, len(w), th.data_ptr(), w.data_ptr(), 40, u.data_ptr(),
                 coef.data_ptr(), mean.data_ptr(), var.data_ptr(), torch.cuda.Stream().cuda_stream)
            call = E.lib().elder_gpc_project
            assert sum(call(*a) != E.ELDER_OK for _ in range(30000)) == 0
            torch.cuda.synchronize()
            assert torch.equal(coef, first)
        return body

    _together(*(calls(*x) for x in work))


def test_contexts_of_different_coarse_grids(E):
    # single-level grids of 160 and 180 unknowns, two contexts each: eliminations
    # of 100 KiB and 127 KiB of one kernel
    work = []
    for dims in ((4, 3, 3), (5, 4, 2)) * 2:
        P = O.Problem(*dims, bc_mode=2)
        rng = np.random.default_rng(sum(dims))
        p0, c0 = O.initial_state(P)
        phi = 0.1 * np.exp(0.2 * rng.standard_normal(P.C))
        ctx = E.elder_create(E.elder_config_default(*dims, bc_mode=2, mg_levels=1,
                                                    precision=E.ELDER_MIXED))
        a = (T(phi), T(4.845e-13 * (phi / 0.1) ** 3), T(p0), T(c0), O.SECONDS_PER_YEAR / 12,
             E.ELDER_SMOOTH_JACOBI, T(rng.standard_normal(2 * P.N)))
        work.append((ctx, a, ctx.smoother_apply(1, *a).clone()))
    torch.cuda.synchronize()

    def calls(ctx, a, first):
        def body():
            phi, K, p, c, dt, kind, r = a
            z = torch.empty_like(r)
            q = (ctx._h, 1, phi.data_ptr(), K.data_ptr(), p.data_ptr(), c.data_ptr(), dt, kind, 0,
                 r.data_ptr(), z.data_ptr(), torch.cuda.Stream().cuda_stream)
            call = E.lib().elder_smoother_apply
            assert sum(call(*q) != E.ELDER_OK for _ in range(5000)) == 0
            torch.cuda.synchronize()
            assert torch.equal(z, first)
        return body

    _together(*(calls(*x) for x in work))
    for ctx, _, _ in work:
        ctx.destroy()
