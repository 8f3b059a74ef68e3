"""Asynchronous calls recorded into a CUDA graph replay to the eager results:
the Schwarz preconditioner (whose coarse solve is one cluster or one cooperative launch) and
the assembled operators."""
import math

import pytest
import torch

import paper_2107_01243_gb300 as sem

pytestmark = pytest.mark.gpu


def replayed(call, out):
    """out after call() eagerly, then after replaying its capture on cleared memory."""
    call()
    torch.cuda.synchronize()
    eager = out.clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    out.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    return eager, out.clone()


@pytest.mark.parametrize("nel,N", [((3, 4, 5), 5), ((9, 8, 7), 7), ((2, 1, 1), 2),
                                   ((32, 31, 15), 2)])   # 16,896 vertices: a grid
def test_schwarz_apply_captured(nel, N):
    h = sem.sem_setup(nel, N, length=(2 * math.pi,) * 3, deform=0.1)
    m = sem.sem_schwarz_create(h)
    b = torch.empty(h.n_local, dtype=torch.float64, device="cuda")
    sem.sem_rhs(h, torch.rand_like(b), b)
    z = torch.empty_like(b)
    eager, got = replayed(lambda: sem.sem_schwarz_apply(m, b, z), z)
    # the overlapping corrections are added in no fixed order (FP32): 2^-24 of the
    # largest value per addition, at most eight additions and ten coarse iterations
    assert float((got - eager).abs().max()) <= 1e-4 * float(eager.abs().max())


@pytest.mark.parametrize("N", [4, 6, 7])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_apply_captured(N, dtype):
    h = sem.sem_setup((5, 4, 3), N, length=(2 * math.pi,) * 3, deform=0.1)
    u = torch.rand(h.n_local, dtype=dtype, device="cuda")
    w = torch.empty_like(u)
    eager, got = replayed(lambda: sem.sem_apply(h, u, w), w)
    assert torch.equal(eager, got)
