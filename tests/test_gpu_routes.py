"""Calls at the sizes where the dispatch changes kernels, against the oracle."""
import numpy as np
import pytest
import torch

import paper_2107_01243_gb300 as sem
import seeded_inputs as si
from tests.helpers import OracleProblem, rel_inf, TWO_PI

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("nel,N", [((12, 8, 8), 3), ((13, 12, 5), 3), ((8, 6, 4), 5),
                                   ((13, 5, 3), 5), ((2, 2, 2), 5)])
@pytest.mark.parametrize("tuned", [False, True])
def test_fp32_element_operator_on_small_boxes(nel, N, tuned):
    """Bulk copies up to 768 elements at N = 3 and 192 at N = 5, unless the caller
    pins the line kernel (the FP32 tolerance of the other kernels' tests)."""
    h = sem.sem_setup(nel, N, length=(TWO_PI,) * 3, deform=0.1)
    o = OracleProblem(nel, N, length=(TWO_PI,) * 3, deform=0.1)
    if tuned:
        sem.sem_set_tuning(h, ax32_kernel="global-load")
    u = si.uniform(o.shape, 61).astype(np.float32).astype(np.float64)
    ud = torch.from_numpy(u).to(DEV, torch.float32).view(-1)
    w = torch.empty_like(ud)
    sem.sem_ax(h, ud, w, 0.7, 1.5)
    assert rel_inf(w.double().cpu().numpy().reshape(o.shape), o.ax(u, 0.7, 1.5)) < 2e-5


@pytest.mark.parametrize("nel", [(8, 19, 1), (9, 17, 1), (2, 2, 2)])
def test_global_operator_n9_around_one_cta_an_sm(nel):
    """152 elements (all of G fetched ahead) and 153, at the tolerance of the
    other orders' parity tests."""
    N = 9
    h = sem.sem_setup(nel, N, length=(TWO_PI,) * 3, deform=0.1)
    o = OracleProblem(nel, N, length=(TWO_PI,) * 3, deform=0.1)
    u = si.uniform((h.n_global,), 62).astype(np.float32).astype(np.float64)
    w = torch.empty(h.n_global, dtype=torch.float32, device=DEV)
    sem.sem_apply_global(h, torch.from_numpy(u).to(DEV, torch.float32), w, 0.7, 1.5)
    ref = np.zeros(h.n_global)
    ref[o.gid.reshape(-1)] = o.matvec(u[o.gid], 0.7, 1.5).reshape(-1)
    assert rel_inf(w.double().cpu().numpy(), ref) < 2e-5


@pytest.mark.parametrize("nel,N", [((15, 20, 8), 1), ((15, 20, 11), 1), ((25, 20, 16), 1),
                                   ((20, 20, 12), 2), ((20, 20, 13), 2), ((25, 20, 16), 2),
                                   ((19, 10, 10), 3), ((16, 15, 13), 3), ((13, 13, 13), 4),
                                   ((14, 14, 15), 5), ((11, 10, 10), 6), ((12, 10, 10), 6),
                                   ((10, 9, 9), 9)])
@pytest.mark.parametrize("precision", [sem.SEM_SOLVE_F64, sem.SEM_SOLVE_MIXED])
def test_solves_around_the_resident_limits(nel, N, precision):
    """Both sides of the element counts where solves stop iterating inside one
    launch, by order and arithmetic."""
    h = sem.sem_setup(nel, N, length=(TWO_PI,) * 3, deform=0.1)
    o = OracleProblem(nel, N, length=(TWO_PI,) * 3, deform=0.1)
    b = o.rhs(si.eval_fourier(si.fourier_modes(31), o.x, o.y, o.z))
    bd = torch.from_numpy(b).to(DEV).view(-1)
    x = torch.full_like(bd, float("nan"))
    info = sem.sem_cg_solve(h, bd, x, h2=0.5, tol=1e-9, precision=precision)
    res = o.residual(x.cpu().numpy().reshape(o.shape), b, h1=1.0, h2=0.5)
    assert info["status"] == "SEM_OK" and res <= 1.05e-9


@pytest.mark.parametrize("nel,N", [((16, 14, 8), 7), ((17, 14, 8), 7), ((16, 16, 16), 5),
                                   ((17, 16, 16), 5)])
def test_fp64_finishing_passes_around_seven_megabytes(nel, N):
    """One pass up to 7 MB of FP64, three beyond: the sums of sem_ax followed by
    sem_dssum to their rounding (eight copies: 4e-15 of the largest value)."""
    h = sem.sem_setup(nel, N, length=(TWO_PI,) * 3, deform=0.1,
                      faces=sem.SEM_FACE_XMIN | sem.SEM_FACE_ZMAX)
    u = torch.from_numpy(si.uniform(h.n_local, 63)).to(DEV)
    w, v = torch.empty_like(u), torch.empty_like(u)
    sem.sem_apply(h, u, w, 1.0, 0.5)
    sem.sem_ax(h, u, v, 1.0, 0.5)
    scale = v.abs().max()
    sem.sem_dssum(h, v)
    assert float((w - v).abs().max() / scale) < 4e-15


def test_bounded_waits_run_out_and_later_solves_are_clean():
    """The self-test's grid barrier is one arrival short: the coarse solve's kernel
    gives up after 20 ms, records it and leaves NaN in its solution (the self-test
    says SEM_OK otherwise).  Solves on the handle, in one launch and with the
    preconditioner, go on as before."""
    h = sem.sem_setup((4, 3, 3), 7, length=(TWO_PI,) * 3, deform=0.1)
    f = torch.from_numpy(si.uniform(h.n_local, 64)).to(DEV)
    b = sem.sem_rhs(h, f, torch.empty_like(f))
    m = sem.sem_schwarz_create(h)
    before = torch.empty_like(b)
    sem.sem_cg_solve(h, b, before, tol=1e-9)
    assert sem.sem_selftest_timeout(h, 20.0) == "SEM_ERR_TIMEOUT"
    sem.sem_sync(h)
    after = torch.empty_like(b)
    assert sem.sem_cg_solve(h, b, after, tol=1e-9)["status"] == "SEM_OK"
    assert torch.equal(before, after)
    info = sem.sem_gmres_solve(h, b, after, tol=1e-9, restart=10, precond=m,
                               precision=sem.SEM_SOLVE_MIXED)
    assert info["status"] == "SEM_OK" and info["rel_res"] <= 1e-9
