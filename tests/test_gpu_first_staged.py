"""Staged solves captured into CUDA graphs as the first library call of a process:
the line kernels' attributes are set by sem_setup, not inside the capture.  (Small
solves iterate inside one launch; replaced multiplicities, the handle's own, make
these ones stage.)"""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json, sys
import torch
sys.path.insert(0, sys.argv[1])
import paper_2107_01243_gb300 as sem
import seeded_inputs as si

case, N, nel = sys.argv[2], int(sys.argv[3]), json.loads(sys.argv[4])
h = sem.sem_setup(nel, N, length=(6.0,) * 3, deform=0.1)
mult = torch.empty(h.n_local, dtype=torch.float64, device="cuda:0")
sem.sem_set_multiplicity(h, sem.sem_get_field(h, sem.SEM_FIELD_MULT, mult))
f = torch.from_numpy(si.uniform(h.n_local, 13)).to("cuda:0")
b = sem.sem_rhs(h, f, torch.empty_like(f))
if case == "native":
    sem.sem_set_f64_kernel(h, sem.SEM_F64_KERNEL_NATIVE)
if case == "local":
    sem.sem_set_inner_vectors(h, sem.SEM_INNER_LOCAL)
if case == "global":
    sem.sem_set_inner_vectors(h, sem.SEM_INNER_GLOBAL)
prec = sem.SEM_SOLVE_MIXED if case in ("local", "global") else sem.SEM_SOLVE_F64
info = sem.sem_cg_solve(h, b, torch.empty_like(b), tol=1e-8, precision=prec, use_graph=True)
print(json.dumps(info))
"""


@pytest.mark.parametrize("case,N,nel", [("native", 7, [16, 12, 8]), ("native", 9, [3, 3, 3]),
                                        ("f64", 6, [4, 3, 3]), ("local", 6, [4, 3, 3]),
                                        ("local", 7, [4, 3, 3]), ("global", 9, [4, 3, 3])])
def test_staged_solve_as_first_call(case, N, nel):
    out = subprocess.run([sys.executable, "-c", CHILD, ROOT, case, str(N), json.dumps(nel)],
                         cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert out.returncode == 0, out.stderr[-3000:]
    info = json.loads(out.stdout.strip().splitlines()[-1])
    assert info["status"] == "SEM_OK" and info["rel_res"] <= 1.0001e-8, info
