"""Solves with one kernel per stage (csrc/cg.cu): what large problems run, here
on small ones (a handle with replaced multiplicities, its own, does not iterate
inside one launch).  Every vector kernel (FP64 and FP32, 16-byte and scalar),
graph and no graph, stops inside a batch, at its end and at maxit with the x that
belongs to them, an initial guess."""
import numpy as np
import pytest
import torch

import paper_2107_01243_gb300 as sem
import seeded_inputs as si
from tests.helpers import OracleProblem, TWO_PI

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
MIXED = dict(precision=sem.SEM_SOLVE_MIXED)


def to_dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV, torch.float64).view(-1)


def problem(nel, N):
    h = sem.sem_setup(nel, N, length=(TWO_PI,) * 3, deform=0.1)
    mult = torch.empty(h.n_local, dtype=torch.float64, device=DEV)
    sem.sem_set_multiplicity(h, sem.sem_get_field(h, sem.SEM_FIELD_MULT, mult))
    sem.sem_set_inner_vectors(h, sem.SEM_INNER_LOCAL)
    o = OracleProblem(nel, N, length=(TWO_PI,) * 3, deform=0.1)
    return h, o, o.rhs(si.eval_fourier(si.fourier_modes(31), o.x, o.y, o.z))


# n_L odd (scalar kernels), even but no multiple of four (FP32 scalar), a multiple
@pytest.mark.parametrize("nel,N", [((3, 3, 3), 4), ((2, 3, 3), 6), ((4, 3, 2), 8), ((3, 3, 2), 7),
                                   ((3, 2, 2), 5), ((5, 4, 3), 1)])
@pytest.mark.parametrize("kind", ["f64", "native", "field", "mixed"])
def test_staged_solves_match_the_oracle(nel, N, kind):
    h, o, b = problem(nel, N)
    if kind == "native":
        sem.sem_set_f64_kernel(h, sem.SEM_F64_KERNEL_NATIVE)
    h1f = si.smooth_coefficient(o.x, o.y, o.z, 77) if kind == "field" else None
    kw = dict(MIXED) if kind == "mixed" else {}
    if h1f is not None:
        kw["h1_field"] = to_dev(h1f)
    x = torch.full((h.n_local,), float("nan"), dtype=torch.float64, device=DEV)
    info = sem.sem_cg_solve(h, to_dev(b), x, h2=0.7, tol=1e-9, **kw)
    res = o.residual(x.cpu().numpy().reshape(o.shape), b, h1=1.0, h2=0.7, h1_field=h1f)
    assert info["status"] == "SEM_OK" and res <= 1.05e-9
    if kind != "mixed":
        ref = o.pcg(b, h2=0.7, tol=1e-9, h1_field=h1f)
        assert abs(info["iters"] - ref.iters) <= 1


@pytest.mark.parametrize("nel,N", [((3, 3, 3), 4), ((3, 3, 2), 7)])
@pytest.mark.parametrize("kw", [{}, MIXED])
def test_graphs_and_batches_give_the_same_x(nel, N, kw):
    """The kernels and their order do not depend on how they are launched."""
    h, o, b = problem(nel, N)
    xs = []
    for graph in (True, False):
        for every in (1, 7, 16, 1000):
            x = torch.full((h.n_local,), float("nan"), dtype=torch.float64, device=DEV)
            info = sem.sem_cg_solve(h, to_dev(b), x, tol=1e-9, use_graph=graph, check_every=every,
                                    **kw)
            xs.append((info["iters"], x.cpu().numpy()))
    for it, x in xs[1:]:
        assert it == xs[0][0]
        np.testing.assert_array_equal(x, xs[0][1])


@pytest.mark.parametrize("nel,N", [((3, 3, 3), 4), ((3, 3, 2), 7), ((2, 3, 3), 6)])
@pytest.mark.parametrize("graph", [True, False])
@pytest.mark.parametrize("maxit", [1, 16, 20])
def test_stop_at_maxit_keeps_the_last_x(nel, N, graph, maxit):
    """x after maxit iterations: the oracle's to rounding (1e-10 of its size), the
    residual that the call reports."""
    h, o, b = problem(nel, N)
    x = torch.full((h.n_local,), float("nan"), dtype=torch.float64, device=DEV)
    info = sem.sem_cg_solve(h, to_dev(b), x, tol=1e-13, maxit=maxit, use_graph=graph,
                            raise_on_fail=False)
    assert info["status"] == "SEM_ERR_NOCONV" and info["iters"] == maxit
    got = x.cpu().numpy().reshape(o.shape)
    assert abs(info["rel_res"] - o.residual(got, b)) <= 1e-12 + 1e-10 * info["rel_res"]
    ref = o.pcg(b, tol=1e-13, maxit=maxit).x
    assert np.abs(got - ref).max() <= 1e-10 * np.abs(ref).max()


@pytest.mark.parametrize("kw", [{}, MIXED])
def test_initial_guess(kw):
    h, o, b = problem((3, 3, 2), 7)
    x = torch.empty(h.n_local, dtype=torch.float64, device=DEV)
    cold = sem.sem_cg_solve(h, to_dev(b), x, tol=1e-9, **kw)
    x2 = torch.empty_like(x)
    warm = sem.sem_cg_solve(h, to_dev(b), x2, tol=1e-9, x0=x * (1.0 + 1e-4), **kw)
    assert warm["status"] == "SEM_OK" and warm["iters"] < cold["iters"]
    assert o.residual(x2.cpu().numpy().reshape(o.shape), b) <= 1.05e-9
