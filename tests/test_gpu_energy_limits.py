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


def _energy(n, r, core, V, rho, C, U):
    import numpy as np
    import paper_1212_3509_gb300 as D
    from gpu_helpers import dev
    import torch
    P = D.demag_build_factors(n, (1 / 50, 1 / 40, 1 / 30), 5)
    e = torch.empty((), dtype=torch.float64, device="cuda")
    D.demag_energy_tucker_phi(P, r, dev(core.ravel()), dev(np.concatenate([v.ravel() for q in V for v in q])), rho,
                              dev(C.ravel()), dev(np.concatenate([u.ravel() for u in U])), e)
    P.close()
    return e.item()


def test_lane_sums_beyond_float32():
    """Columns whose FP32 products fit over 32 columns but not over a warp's 1024: the sum is FP64's."""
    import numpy as np
    from test_gpu_energy_gram import _apply_d
    n, h, r, rho = (1024, 5, 4), (1 / 50, 1 / 40, 1 / 30), (3, 1, 1), (2, 1, 1)
    rng = np.random.default_rng(5)
    one = np.ones
    core, C = one((3, 1, 1, 3), np.float32), one((1, 1, 2), np.float32)
    V = [[(1.5e18 * rng.uniform(0.9, 1, (3, n[0]))).astype(np.float32)] +
         [rng.standard_normal((1, n[p])).astype(np.float32) for p in (1, 2)] for _ in range(3)]
    U = [(1.5e18 * rng.uniform(0.9, 1, (2, n[0]))).astype(np.float32)] + \
        [rng.standard_normal((1, n[p])).astype(np.float32) for p in (1, 2)]
    ref = mag = 0.0
    for q in range(3):
        G = []
        for p in range(3):
            W = U[p].astype(np.float64)
            W = _apply_d(W, h[p]) if p == q else W
            G.append((V[q][p].astype(np.float64) @ W.T, np.abs(V[q][p]).astype(np.float64) @ np.abs(W).T))
        ref += np.prod([g.sum() for g, _ in G])
        mag += np.prod([g.sum() for _, g in G])
    half = 0.5 * h[0] * h[1] * h[2]
    assert mag > 3.4e38 * 10  # beyond float32
    assert abs(_energy(n, r, core, V, rho, C, U) - half * ref) <= 2e-6 * half * mag


@pytest.mark.parametrize("bad,want", [(float("inf"), "inf"), (float("-inf"), "-inf"), (float("nan"), "nan")])
def test_infinities_stay_infinite(bad, want):
    """An infinite entry at the end of an axis, all else positive: every Gram that meets it is infinite of one
    sign (its differences at the last two cells are), and so is the energy."""
    import numpy as np
    n, r, rho = (40, 5, 4), (9, 1, 1), (1, 1, 1)
    rng = np.random.default_rng(6)
    core, C = np.ones((3, 1, 1, 9), np.float32), np.ones((1, 1, 1), np.float32)
    grow = [np.arange(1, n[p] + 1, dtype=np.float32)[None] for p in range(3)]  # positive differences
    V = [[rng.uniform(0.5, 1, (r[p], n[p])).astype(np.float32) for p in range(3)] for _ in range(3)]
    U = [g.copy() for g in grow]
    U[0][0, -1] = bad
    assert str(_energy(n, r, core, V, rho, C, U)) == want
