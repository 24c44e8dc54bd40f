"""Structured energies at the limits of what their kernels take.

Requests of shared memory around the 48 KB that a launch gets without asking,
each in a process of its own (an earlier, larger request on the device would
have raised the limit already).
"""
import os
import subprocess
import sys

import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PHI = """
import sys
sys.path[:0] = ["tests", "."]
from test_gpu_energy_gram import test_energy_of_one_tucker_potential as check
check((20, 18, 17), {r}, {rho})
"""
FP64 = """
import sys
sys.path[:0] = ["tests", "."]
import numpy as np, torch, synth
import paper_1212_3509_gb300 as D
from oracle.energy import energy_from_m
n, r, h = (20, 18, 17), {r}, (1 / 20,) * 3
rng = np.random.default_rng(3)
core, V = rng.standard_normal((3, r[2], r[1], r[0])), rng.standard_normal(3 * sum(a * b for a, b in zip(r, n)))
m, at = [], 0
for q in range(3):
    U = []
    for p in range(3):
        U.append(V[at:at + r[p] * n[p]].reshape(r[p], n[p]))
        at += r[p] * n[p]
    m.append(np.einsum("cba,ax,by,cz->zyx", core[q], *U, optimize=True))
P = D.demag_build_factors(n, h, 21)
e = torch.empty((), dtype=torch.float64, device="cuda")
D.demag_energy_tucker_fp64(P, r, torch.tensor(core.ravel()).cuda(), torch.tensor(V).cuda(), e)
ref = energy_from_m(np.stack(m), n, h, 21)
assert abs(e.item() - ref) <= 1e-10 * abs(ref), (e.item(), ref)
"""


# Grams, intermediates and core of 44688, 44800 and 44776 bytes beside 4496 of static memory: just over 48 KB
@pytest.mark.parametrize("r,rho", [((8, 8, 8), (14, 13, 15)), ((10, 10, 10), (15, 12, 13)), ((1, 12, 58), (1, 12, 58))])
def test_ranks_whose_request_crosses_the_default_limit(r, rho):
    subprocess.run([sys.executable, "-c", PHI.format(r=r, rho=rho)], cwd=ROOT, check=True, timeout=300)


def test_fp64_ranks_whose_request_crosses_the_default_limit():
    subprocess.run([sys.executable, "-c", FP64.format(r=(1, 12, 58))], cwd=ROOT, check=True, timeout=300)
