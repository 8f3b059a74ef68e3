"""Small solves that iterate inside one launch (csrc/resident.cu), judged by
the oracle: every order and arithmetic, one element per CTA and several, more
iterations than one launch runs, face subsets, the status codes; and the
integer sums it reduces with (csrc/fixsum.cuh, on the CPU)."""
import math
import os
import shutil
import subprocess

import numpy as np
import pytest
import torch

import paper_2107_01243_gb300 as sem
import seeded_inputs as si
from tests.helpers import OracleProblem, TWO_PI

DEV = "cuda:0"
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def to_dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV, torch.float64).view(-1)


def problem(nel, N, faces=sem.SEM_FACE_ALL):
    h = sem.sem_setup(nel, N, length=(TWO_PI,) * 3, deform=0.1, faces=faces)
    o = OracleProblem(nel, N, length=(TWO_PI,) * 3, deform=0.1, faces=faces)
    return h, o, o.rhs(si.eval_fourier(si.fourier_modes(31), o.x, o.y, o.z))


def solve(h, o, b, tol, **kw):
    x = torch.full((h.n_local,), float("nan"), dtype=torch.float64, device=DEV)
    h1f = kw.pop("h1_field", None)
    info = sem.sem_cg_solve(h, to_dev(b), x, tol=tol,
                            h1_field=None if h1f is None else to_dev(h1f), **kw)
    xg = x.cpu().numpy().reshape(o.shape)
    res = o.residual(xg, b, h1=kw.get("h1", 1.0), h2=kw.get("h2", 0.0), h1_field=h1f)
    return info, xg, res


# the oracle's stopping test with the 5% the other solve tests allow for the
# recurrence residual against the true one
@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["auto", "native", "field", "mixed"])
@pytest.mark.parametrize("N", range(1, 11))
def test_every_order_matches_the_oracle(N, kind):
    nel = (3, 2, 2) if N > 1 else (5, 4, 3)
    h, o, b = problem(nel, N)
    kw = dict(h2=0.7)
    if kind == "native":
        sem.sem_set_f64_kernel(h, sem.SEM_F64_KERNEL_NATIVE)
    if kind == "field":
        kw["h1_field"] = si.smooth_coefficient(o.x, o.y, o.z, 77)
    if kind == "mixed":
        kw["precision"] = sem.SEM_SOLVE_MIXED
    tol = 1e-9
    info, xg, res = solve(h, o, b, tol, **kw)
    assert info["status"] == "SEM_OK" and res <= 1.05 * tol
    assert abs(info["rel_res"] - res) < 1e-12
    ref = o.pcg(b, h2=0.7, tol=tol, h1_field=kw.get("h1_field"))
    if kind != "mixed":
        assert abs(info["iters"] - ref.iters) <= 1


@pytest.mark.gpu
@pytest.mark.parametrize("nel,N,faces", [
    ((1, 1, 1), 7, sem.SEM_FACE_ALL), ((1, 1, 3), 4, sem.SEM_FACE_XMIN),
    ((2, 1, 1), 9, sem.SEM_FACE_ZMAX | sem.SEM_FACE_YMIN),
    ((13, 11, 5), 2, sem.SEM_FACE_ALL),                # more elements than CTAs
    ((9, 9, 9), 3, sem.SEM_FACE_XMAX | sem.SEM_FACE_YMAX), ((1, 40, 16), 3, 0)])
@pytest.mark.parametrize("precision", [sem.SEM_SOLVE_F64, sem.SEM_SOLVE_MIXED])
def test_box_shapes_and_faces(nel, N, faces, precision):
    h, o, b = problem(nel, N, faces)
    tol = 1e-9
    info, xg, res = solve(h, o, b, tol, h2=1.3, precision=precision)
    assert info["status"] == "SEM_OK" and res <= 1.05 * tol


@pytest.mark.gpu
def test_more_iterations_than_one_launch_and_maxit():
    """Flat elements (the oracle takes 1688 iterations): the state crosses the
    launches of 512 iterations."""
    nel, N = (60, 2, 1), 7
    h = sem.sem_setup(nel, N)
    o = OracleProblem(nel, N)
    b = o.rhs(si.uniform((int(o.gid.max()) + 1,), 5)[o.gid])
    ref = o.pcg(b, tol=1e-11)
    info, xg, res = solve(h, o, b, 1e-11)
    assert ref.iters > 512 and abs(info["iters"] - ref.iters) <= ref.iters // 50
    assert res <= 1.05e-11
    info, _, _ = solve(h, o, b, 1e-11, maxit=515, raise_on_fail=False)
    assert info["status"] == "SEM_ERR_NOCONV" and info["iters"] == 515


@pytest.mark.gpu
def test_results_repeat_bit_for_bit():
    for N in (6, 7):
        h, o, b = problem((5, 4, 3), N)
        x = [solve(h, o, b, 1e-10)[1] for _ in range(2)]
        assert np.array_equal(x[0], x[1])


def test_integer_sums_on_the_host(tmp_path):
    """fixsum.cuh: a value survives the trip through its integer exactly, and a
    sum is within one rounding plus 2^-56 of the largest term a piece."""
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    src = tmp_path / "fx.cpp"
    src.write_text(r'''
#include "fixsum.cuh"
#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <vector>
using namespace sem;
static unsigned long long bits(double x) { unsigned long long b; memcpy(&b, &x, 8); return b; }
int main() {
  std::mt19937_64 g(1);
  for (int t = 0; t < 300000; ++t) {
    unsigned long long b = g();
    if (t % 7 == 0) b &= ~(0x7FFull << 52);            // subnormals
    if (((b >> 52) & 0x7FF) == 0x7FF) continue;
    const int e = fx_exp(b);
    const long long m = fx_mant(b, e);
    const double r = fx_round(m >> 32, (long long)(unsigned)m, e);
    if (bits(r) != b && !(r == 0 && !(b << 1))) return 1;
  }
  for (int t = 0; t < 30000; ++t) {
    const int n = 1 + g() % 700, spread = g() % 80;
    std::vector<double> v(n);
    long double s = 0;
    int e = 1;
    for (auto& x : v) {
      x = std::ldexp((double)(g() >> 11) * 0x1p-53 + 0.1, (int)(g() % (spread + 1)) - 30);
      if (t % 2 && (g() & 1)) x = -x;
      s += x;
      e = std::max(e, fx_exp(bits(x)));
    }
    long long hi = 0, lo = 0;
    for (double x : v) {
      const long long m = fx_mant(bits(x), e);
      hi += m >> 32;
      lo += (long long)(unsigned)m;
    }
    const long double err = fabsl((long double)fx_round(hi, lo, e) - s);
    if (err > 0x1p-52L * fabsl(s) + n * std::ldexp(1.0L, e - 1023 - 56)) return 2;
  }
  return std::isnan(fx_round(1, 1, kFxBad)) && fx_round(0, 0, 9) == 0.0 ? 0 : 3;
}
''')
    exe = str(tmp_path / "fx")
    csrc = os.path.join(ROOT, "paper_2107_01243_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-D__host__=", "-D__device__=", "-I", csrc,
                    str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0
