"""Batches whose large problems finish long before the small ones: the element
launches leave finished problems out, and the next solve has them all again."""
import numpy as np
import pytest
import torch

import paper_2107_01243_gb300 as sem
import seeded_inputs as si
from tests.helpers import OracleProblem, TWO_PI

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
PROBLEMS = [((9, 8, 7), 7), ((8, 8, 5), 9), ((3, 2, 2), 7), ((4, 3, 2), 5), ((2, 2, 2), 9)]


@pytest.mark.parametrize("use_graph", [True, False])
@pytest.mark.parametrize("concurrent", [True, False])
def test_finished_problems_leave_the_launches(use_graph, concurrent):
    """First the two large problems have b = 0 (done at once), then a whole order
    has, then none: every solution within the tolerance of the oracle's residual,
    zero where b is zero."""
    hs = [sem.sem_setup(nel, N, length=(TWO_PI,) * 3, deform=0.1) for nel, N in PROBLEMS]
    os = [OracleProblem(nel, N, length=(TWO_PI,) * 3, deform=0.1) for nel, N in PROBLEMS]
    full = [o.rhs(si.eval_fourier(si.fourier_modes(70 + q), o.x, o.y, o.z))
            for q, o in enumerate(os)]
    batch = sem.sem_batch_create(hs)
    sem.sem_batch_set_concurrency(batch, concurrent)
    for zero in ({0, 1}, {1, 4}, set(), {0, 1, 2, 4}):
        bs = [np.zeros_like(b) if q in zero else b for q, b in enumerate(full)]
        bd = [torch.from_numpy(b).to(DEV).view(-1) for b in bs]
        xs = [torch.full_like(b, float("nan")) for b in bd]
        infos = sem.sem_batch_solve(batch, bd, xs, [1.0] * 5, [0.3] * 5, tol=1e-8, check_every=5,
                                    use_graph=use_graph)
        for q, (o, b, x, info) in enumerate(zip(os, bs, xs, infos)):
            assert info["status"] == "SEM_OK"
            xg = x.cpu().numpy().reshape(o.shape)
            if q in zero:
                assert info["iters"] == 0 and not xg.any()
            else:
                assert o.residual(xg, b, h1=1.0, h2=0.3) <= 1.05e-8
