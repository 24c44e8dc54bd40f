"""Structured formats at every transform length of the register kernel and around it.

Columns of 129 to 2048 cells transform in registers, two nodes at a time, with
32 to 256 threads per column; shorter and longer ones by in-place passes.
Odd and even node numbers and ranks, columns that do and do not fill their
blocks, against the FP64 oracle, node by node; and that neither a column's
neighbours nor the rest of a batch bear on it.
"""
import numpy as np
import pytest

import synth
from gpu_helpers import dev, host
from oracle import structured as ost

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _apply(D, n, r, lam, U, R):
    P = D.demag_build_factors(n, (1.0 / max(n),) * 3, R)
    B = len(lam)
    w = torch.full((B, P.M, 3, r), float("nan"), device="cuda")
    out = torch.full((B, P.M * 3 * r * sum(n)), float("nan"), device="cuda")
    D.demag_apply_cp_batched(P, B, r, dev(np.stack(lam).astype(np.float32)), dev(np.stack(U)), w, out)
    torch.cuda.synchronize()
    M = P.M
    P.close()
    return M, host(out)


# A column's error lies within eps log2(L) of |t|_1 |x|_2 (forward, product and inverse of a normwise
# stable transform, t the generator), with |t|_1 the larger of the two nodes that share a transform;
# relative to y itself it is not bounded, since a flat generator can sum a column to nearly nothing.
@pytest.mark.parametrize("n,r,R", [((129, 256, 128), 1, 7), ((257, 300, 512), 3, 9), ((513, 1000, 1024), 2, 5),
                                   ((1025, 2048, 140), 1, 7), ((2049, 4096, 3000), 1, 5), ((4097, 200, 1), 1, 5)])
def test_cp_vs_oracle(n, r, R):
    import paper_1212_3509_gb300 as D
    lam, U = synth.cp_inputs(n, r, 70 + sum(n))
    h = (1.0 / max(n),) * 3
    M, got = _apply(D, n, r, [lam], [U.ravel()], R)
    _, ref = ost.apply_cp(lam, U.ravel(), n, h, R)
    V = ost._split_blocks(U.ravel(), n, (r, r, r))
    _, hh = ost.scaled_spacing(n, h)
    tau = ost.sinc_nodes(M, 2.15)[2]
    at = 0
    for p in range(3):
        size, L = M * 3 * r * n[p], 1 << (2 * n[p] - 1).bit_length()
        g, e = got[0][at:at + size].reshape(M, 3, r, n[p]), ref[p]
        at += size
        for q in range(3):
            gen = ost.gen_F if ost.factor_kind(p, q) == "F" else ost.gen_E
            t1 = [np.abs(gen(tau[k], hh[p], n[p])).sum() for k in range(M)]
            x = np.linalg.norm(V[q][p], axis=1)
            for k in range(M):
                bound = 2.0 ** -24 * np.log2(L) * max(t1[k], t1[min(k ^ 1, M - 1)]) * x
                assert (np.linalg.norm(g[k, q] - e[k, q], axis=1) <= bound).all(), (p, k, q)


def test_columns_do_not_meet():
    import paper_1212_3509_gb300 as D
    n, r, R, B = (200, 300, 1100), 1, 9, 3
    items = [synth.cp_inputs(n, r, 80 + i) for i in range(B)]
    lam, U = [i[0] for i in items], [i[1].ravel().astype(np.float32) for i in items]
    M, alone = _apply(D, n, r, lam[1:2], U[1:2], R)
    scaled = [U[0] * np.float32(1e30), U[1], np.full_like(U[2], np.nan)]
    _, both = _apply(D, n, r, lam, scaled, R)
    assert np.array_equal(both[1], alone[0])
    assert np.isnan(both[2]).all()
