"""Small solves inside one launch (csrc/resident.cu) keep the digits of standard
PCG: as many FP32 iterations as the kernels of one launch per stage, tight FP64
tolerances with IEEE arithmetic, and iterations across launches of 512."""
import numpy as np
import pytest
import torch

import paper_2107_01243_gb300 as sem
import seeded_inputs as si
from tests.helpers import OracleProblem, TWO_PI

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def to_dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV, torch.float64).view(-1)


def staged(h):
    """Solves of this handle run one kernel per stage from here on (a handle with
    replaced multiplicities, here its own, does not iterate inside one launch)."""
    mult = torch.empty(h.n_local, dtype=torch.float64, device=DEV)
    sem.sem_set_multiplicity(h, sem.sem_get_field(h, sem.SEM_FIELD_MULT, mult))
    sem.sem_set_inner_vectors(h, sem.SEM_INNER_LOCAL)


@pytest.mark.parametrize("nel,N,length,deform", [((60, 2, 1), 6, 1.0, 0.0),
                                                 ((8, 8, 8), 7, TWO_PI, 0.1)])
def test_fp32_inner_iterations_as_many_as_staged(nel, N, length, deform):
    """The same recurrences in the same precision differ by rounding alone: within
    4% (recurrences that lose digits take 6 and 18% more)."""
    iters = []
    for force in (False, True):
        h = sem.sem_setup(nel, N, length=(length,) * 3, deform=deform)
        if force:
            staged(h)
        f = to_dev(si.uniform(h.n_local, 3) + 0.5)
        b = sem.sem_rhs(h, f, torch.empty_like(f))
        info = sem.sem_cg_solve(h, b, torch.empty_like(b), tol=1e-11, maxit=6000,
                                precision=sem.SEM_SOLVE_MIXED)
        iters.append(info["iters"])
    assert abs(iters[0] - iters[1]) <= 0.04 * iters[1], iters


@pytest.mark.parametrize("N,field", [(5, True), (6, False), (2, True)])
def test_ieee_solves_to_1e_12(N, field):
    nel = (6, 6, 6) if N > 2 else (12, 12, 12)
    h = sem.sem_setup(nel, N, length=(TWO_PI,) * 3, deform=0.1)
    o = OracleProblem(nel, N, length=(TWO_PI,) * 3, deform=0.1)
    b = o.rhs(si.eval_fourier(si.fourier_modes(31), o.x, o.y, o.z))
    h1f = si.smooth_coefficient(o.x, o.y, o.z, 77) if field else None
    x = torch.empty(h.n_local, dtype=torch.float64, device=DEV)
    info = sem.sem_cg_solve(h, to_dev(b), x, h2=0.5, tol=1e-12,
                            h1_field=to_dev(h1f) if field else None)
    res = o.residual(x.cpu().numpy().reshape(o.shape), b, h1=1.0, h2=0.5, h1_field=h1f)
    assert info["status"] == "SEM_OK" and res <= 1.05e-12, (info, res)


@pytest.mark.parametrize("kind", ["even", "native", "field", "mixed"])
def test_iterations_across_launches(kind):
    """Flat elements take more than 512 iterations: IEEE FP64, a per-point h1 and
    FP32, each as many as the oracle's (2%), and a stop at maxit in the second
    launch."""
    nel, N = (60, 2, 1), 7 if kind == "native" else 6
    h, o = sem.sem_setup(nel, N), OracleProblem(nel, N)
    b = o.rhs(si.uniform((int(o.gid.max()) + 1,), 5)[o.gid])
    kw = {}
    if kind == "native":
        sem.sem_set_f64_kernel(h, sem.SEM_F64_KERNEL_NATIVE)
    h1f = si.smooth_coefficient(o.x, o.y, o.z, 9) if kind == "field" else None
    if kind == "field":
        kw["h1_field"] = to_dev(h1f)
    if kind == "mixed":
        kw.update(precision=sem.SEM_SOLVE_MIXED, inner_tol=1e-6)
    x = torch.empty(h.n_local, dtype=torch.float64, device=DEV)
    info = sem.sem_cg_solve(h, to_dev(b), x, tol=1e-9, **kw)
    res = o.residual(x.cpu().numpy().reshape(o.shape), b, h1_field=h1f)
    assert info["status"] == "SEM_OK" and info["iters"] > 512 and res <= 1.05e-9
    if kind != "mixed":
        ref = o.pcg(b, tol=1e-9, h1_field=h1f)
        assert abs(info["iters"] - ref.iters) <= ref.iters // 50
        info = sem.sem_cg_solve(h, to_dev(b), x, tol=1e-9, maxit=515, raise_on_fail=False, **kw)
        assert info["status"] == "SEM_ERR_NOCONV" and info["iters"] == 515


@pytest.mark.parametrize("N", [3, 2])
def test_right_hand_sides_near_the_largest_double(N):
    """b whose squares reach 2^1020 and more but whose norm is finite: the solution of
    a power of two times b, to the bit pattern's scale (products by powers of two are
    exact).  Few unknowns, so that one square makes up much of the norm."""
    h = sem.sem_setup((1, 1, 1), N)
    f = to_dev(si.uniform(h.n_local, 4) + 1.5)
    b = sem.sem_rhs(h, f, torch.empty_like(f))
    bb = torch.zeros(1, dtype=torch.float64, device=DEV)
    sem.sem_dot(h, b, b, bb)
    k = 511 - int(np.floor(np.log2(float(b.abs().max()))))      # max |b| 2^k in [2^511, 2^512)
    while float(bb) * 2.0 ** (2 * k - 1000) >= 2.0 ** 24:       # <b, b> stays finite
        k -= 1
    assert float(b.abs().max()) ** 2 * 2.0 ** (2 * k - 1000) >= 2.0 ** 20
    x, y = torch.empty_like(b), torch.empty_like(b)
    a = sem.sem_cg_solve(h, b, x, tol=1e-9)
    c = sem.sem_cg_solve(h, b * 2.0 ** k, y, tol=1e-9)
    assert (a["status"], a["iters"]) == (c["status"], c["iters"]) == ("SEM_OK", a["iters"])
    assert float((y * 2.0 ** -k - x).abs().max()) <= 1e-12 * float(x.abs().max())
