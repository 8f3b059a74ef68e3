"""IEEE FP64 element operators (csrc/ax.cu, ax_line.cu, resident.cu): rounding no
larger than plain dot products', and the sizes at which N = 7 and 9 change
kernels."""
import numpy as np
import pytest
import torch

import paper_2107_01243_gb300 as sem
import seeded_inputs as si
from oracle.gll import deriv_matrix
from tests.helpers import OracleProblem, rel_inf, TWO_PI

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
LD = np.longdouble


def element_operator(D, G, u, mac):
    """D^T G D u by plain dot products, every product-sum made by mac."""
    def lines(M, x, axis):
        x = np.moveaxis(x, axis, -1)
        y = np.zeros_like(x)
        for l in range(M.shape[0]):
            y = mac(M[:, l], x[..., l:l + 1], y)
        return np.moveaxis(y, -1, axis)
    d = [lines(D, u, a) for a in (3, 2, 1)]
    flux = []
    for g in ((0, 3, 4), (3, 1, 5), (4, 5, 2)):
        acc = np.zeros_like(u)
        for c, v in zip(g, d):
            acc = mac(G[:, c], v, acc)
        flux.append(acc)
    out = [lines(D.T, f, a) for f, a in zip(flux, (3, 2, 1))]
    return (out[0] + out[1]) + out[2]


def test_rounding_of_nearly_constant_fields():
    """N = 2, where D's entries are exact: fields of size 3 that vary by 0.05, the
    kind whose large terms cancel.  The split of D into even and odd halves is
    2.7 times as far from the exact result as fused plain dots; the kernel stays
    within 1.5 times."""
    nel, N = (6, 6, 6), 2
    h = sem.sem_setup(nel, N, length=(TWO_PI,) * 3, deform=0.1)
    o = OracleProblem(nel, N, length=(TWO_PI,) * 3, deform=0.1)
    u = 3.0 * si.uniform((o.shape[0], 1, 1, 1), 7) + 0.05 * si.uniform(o.shape, 8)
    G = torch.empty(6 * h.n_local, dtype=torch.float64, device=DEV)
    sem.sem_get_field(h, sem.SEM_FIELD_G, G)
    G = G.cpu().numpy().reshape(o.shape[0], 6, 3, 3, 3)
    D = deriv_matrix(N)
    exact = element_operator(D.astype(LD), G.astype(LD), u.astype(LD), lambda a, b, c: c + a * b)
    fused = element_operator(D, G, u, lambda a, b, c: (LD(1) * a * b + c).astype(np.float64))
    ud = torch.from_numpy(u).to(DEV).view(-1)
    w = torch.empty_like(ud)
    sem.sem_ax(h, ud, w)
    rms = lambda v: float(np.sqrt(((v - exact) ** 2).mean()))
    assert rms(w.cpu().numpy().reshape(u.shape).astype(LD)) <= 1.5 * rms(fused.astype(LD))


@pytest.mark.parametrize("nel,N", [((120, 2, 1), 4), ((60, 2, 1), 6)])
def test_mixed_solve_on_flat_elements_reaches_the_fp64_floor(nel, N):
    """The refinement's FP64 residual rounds at about 9e-13 of b on these elements
    (60 and 120 times as wide as high); a less accurate operator never gets to
    1e-12."""
    h = sem.sem_setup(nel, N)
    f = torch.from_numpy(si.uniform(h.n_local, 3) + 0.5).to(DEV).view(-1)
    b = sem.sem_rhs(h, f, torch.empty_like(f))
    info = sem.sem_cg_solve(h, b, torch.empty_like(b), tol=1e-12, maxit=6000,
                            precision=sem.SEM_SOLVE_MIXED, raise_on_fail=False)
    assert info["status"] == "SEM_OK", info


@pytest.mark.parametrize("nel", [(17, 10, 9), (16, 12, 8)])
@pytest.mark.parametrize("N", [7, 9])
def test_native_kernels_around_their_crossover(nel, N):
    """1,530 elements (one a CTA) and 1,536 (the line kernel), against the
    double-float kernel on the same geometry (both round at 1e-15 of the largest
    flux, whose cancellation leaves 1e-13)."""
    h = sem.sem_setup(nel, N, length=(TWO_PI,) * 3, deform=0.1,
                      faces=sem.SEM_FACE_XMIN | sem.SEM_FACE_YMAX)
    u = torch.from_numpy(si.uniform(h.n_local, 51)).to(DEV)
    got = {}
    for kind in (sem.SEM_F64_KERNEL_NATIVE, sem.SEM_F64_KERNEL_DOUBLEFLOAT):
        sem.sem_set_f64_kernel(h, kind)
        got[kind] = [sem.sem_ax(h, u, torch.empty_like(u), 0.7, 1.5).cpu().numpy(),
                     sem.sem_apply(h, u, torch.empty_like(u), 0.7, 1.5).cpu().numpy()]
    for a, b in zip(*got.values()):
        assert rel_inf(a, b) < 1e-12
