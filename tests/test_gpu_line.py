"""The line kernel (csrc/ax_line.cu) at the edges of its tiles: element counts
around a CTA's share, vectors without 16-byte alignment, masks and x-pairs of
its fused output, every order, against the oracle."""
import numpy as np
import pytest
import torch

import paper_2107_01243_gb300 as sem
import seeded_inputs as si
from tests.helpers import OracleProblem, rel_inf, TWO_PI

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
# elements per CTA of each order (line_elems; three in FP64 at N = 9)
SHARE = {1: 64, 2: 28, 3: 16, 4: 10, 5: 7, 6: 5, 7: 4, 8: 3, 9: 2, 10: 2}
TOL = {torch.float64: 1e-12, torch.float32: 2e-5}      # as for the other kernels


def unaligned(a, dtype):
    """The values at an address one value past a 16-byte boundary."""
    buf = torch.empty(a.size + 1, dtype=dtype, device=DEV)
    buf[1:] = torch.from_numpy(np.ascontiguousarray(a)).to(DEV, dtype).view(-1)
    return buf[1:]


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("extra", [-1, 0, 1])
@pytest.mark.parametrize("N", range(1, 11))
def test_element_counts_around_a_cta(N, extra, dtype):
    share = 3 if N == 9 and dtype == torch.float64 else SHARE[N]
    nel = (2 * share + extra, 1, 1) if N < 4 else (2 * share + extra, 2, 1)
    faces = sem.SEM_FACE_XMIN | sem.SEM_FACE_ZMAX
    h = sem.sem_setup(nel, N, length=(TWO_PI,) * 3, deform=0.1, faces=faces)
    o = OracleProblem(nel, N, length=(TWO_PI,) * 3, deform=0.1, faces=faces)
    sem.sem_set_f64_kernel(h, sem.SEM_F64_KERNEL_NATIVE)
    cast = np.float32 if dtype == torch.float32 else np.float64
    u = si.uniform(o.shape, 41 + N).astype(cast).astype(np.float64)
    f = si.smooth_coefficient(o.x, o.y, o.z, 42).astype(cast).astype(np.float64)
    ud, fd = unaligned(u, dtype), unaligned(f, dtype)
    w = unaligned(np.zeros(u.size), dtype)
    np_w = lambda: w.double().cpu().numpy().reshape(o.shape)
    sem.sem_ax(h, ud, w, 0.7, 1.5)
    assert rel_inf(np_w(), o.ax(u, 0.7, 1.5)) < TOL[dtype]
    sem.sem_apply(h, ud, w, 0.7, 1.5)
    full = np_w()
    assert rel_inf(full, o.matvec(u, 0.7, 1.5)) < TOL[dtype]
    assert not full[o.mask == 0].any()
    sem.sem_apply(h, ud, w, 0.7, 1.5, phase=sem.SEM_APPLY_LOCAL)
    sem.sem_apply(h, ud, w, 0.7, 1.5, phase=sem.SEM_APPLY_FINISH)
    np.testing.assert_array_equal(np_w(), full)
    sem.sem_apply(h, ud, w, 0.0, 0.5, h1_field=fd)
    assert rel_inf(np_w(), o.matvec(u, 0.0, 0.5, f)) < TOL[dtype]


@pytest.mark.parametrize("N", [2, 6, 7, 8])
def test_infinities_and_nan_stay_in_their_element(N):
    """A non-finite value spreads within its element (and, assembled, to its
    neighbours' shared points), never to another element's interior."""
    nel = (5, 1, 1)
    h = sem.sem_setup(nel, N, length=(TWO_PI,) * 3, deform=0.1)
    sem.sem_set_f64_kernel(h, sem.SEM_F64_KERNEL_NATIVE)
    for dtype in (torch.float64, torch.float32):
        u = torch.rand(h.n_local, dtype=dtype, device=DEV)
        u[2 * (N + 1) ** 3 + 5] = float("inf")
        w = torch.empty_like(u)
        sem.sem_ax(h, u, w)
        finite = torch.isfinite(w).view(5, -1).all(1).cpu().tolist()
        assert finite == [True, True, False, True, True]


@pytest.mark.parametrize("nel,N", [((7, 5, 6), 7), ((9, 4, 5), 6), ((5, 5, 5), 9), ((11, 3, 4), 4),
                                   ((3, 9, 2), 2), ((1, 5, 4), 8), ((6, 1, 5), 5), ((13, 2, 1), 3)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_apply_one_finishing_pass(nel, N, dtype):
    """Boxes whose segments end at different columns of neighbouring rows: the
    single finishing pass leaves every copy of a point with the same value."""
    faces = sem.SEM_FACE_YMIN | sem.SEM_FACE_XMAX
    h = sem.sem_setup(nel, N, length=(TWO_PI,) * 3, deform=0.1, faces=faces)
    o = OracleProblem(nel, N, length=(TWO_PI,) * 3, deform=0.1, faces=faces)
    u = si.uniform(o.shape, 66).astype(np.float32).astype(np.float64)
    ud = torch.from_numpy(u).to(DEV, dtype).view(-1)
    w = torch.empty_like(ud)
    sem.sem_apply(h, ud, w, 0.9, 0.4)
    got = w.double().cpu().numpy().reshape(o.shape)
    assert rel_inf(got, o.matvec(u, 0.9, 0.4)) < TOL[dtype]
    first = np.zeros(int(o.gid.max()) + 1)
    first[o.gid.reshape(-1)] = got.reshape(-1)
    np.testing.assert_array_equal(first[o.gid], got)
