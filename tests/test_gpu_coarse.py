"""The coarse CG of the Schwarz preconditioner at the sizes where its form
changes: one cluster up to 16,384 vertices (full cluster, flat and long boxes,
whose neighbours lie far away and close by), one cooperative grid up to 608
CTAs, and a loop of launches beyond, against the oracle.

Both sides run ten Jacobi-CG iterations, the GPU on FP32 vectors and an
FP32-rounded right-hand side: as for the small boxes of test_gpu_schwarz.py the
results agree to 1e-4 of the largest value."""
import pytest

import paper_2107_01243_gb300 as sem
from oracle import mesh
from tests.helpers import rel_inf
from tests.test_gpu_schwarz import gpu_apply, make, residual_vector

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nel,faces", [((31, 31, 15), mesh.ALL_FACES),     # 16,384 vertices
                                       ((127, 63, 1), mesh.FACE_XMIN),     # 16,384, flat
                                       ((1, 1, 4095), mesh.FACE_ZMAX),     # 16,384, long
                                       ((15, 1, 1), mesh.FACE_YMIN),       # 64: 4 a CTA
                                       ((32, 31, 15), mesh.ALL_FACES),     # 16,896: a grid
                                       ((53, 53, 53), mesh.ALL_FACES)])    # 157,464: launches
def test_coarse_level_at_the_edges_of_its_forms(nel, faces):
    h, o, sw = make(nel, 2, faces, h2=0.4)
    r = residual_vector(o, 121)
    ref = sw.prolong(sw.coarse_solve(sw.restrict(r))) * o.mask
    got = gpu_apply(h, r, sem.SEM_SCHWARZ_COARSE, h2=0.4)
    assert rel_inf(got, ref) < 1e-4
