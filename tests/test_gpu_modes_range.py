"""The CUDA-core mode products over the whole range of float32.

The halves' operands are sums and differences of two field values; neither they
nor their factors may leave the range that the values and the results keep.
"""
import numpy as np
import pytest

import synth
from gpu_helpers import TOL, assert_close, dev, host
from oracle import full as ofull
from oracle import nonuniform as onu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# values up to 3e38, near the largest float32 (3.4e38), and down to 1e-30
@pytest.mark.parametrize("scale", [3e38, 1e-30])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n,uniform", [((17, 12, 33), True), ((40, 64, 9), True), ((11, 20, 8), False)])
def test_values_of_any_size(n, uniform, prec, scale):
    import paper_1212_3509_gb300 as D
    R = 21
    m = synth.random_unit_m(n, 90)
    m /= np.abs(m).max()
    if uniform:
        h = (1 / max(n),) * 3
        P = D.demag_build_factors(n, h, R)
        ref, adj = ofull.apply_full(m, n, h, R), ofull.apply_adjoint(m[0], n, h, R)
    else:
        rng = np.random.default_rng(8)
        edges = [np.concatenate([[0.0], np.cumsum(0.5 + rng.random(v))]) / (2 * max(n)) for v in n]
        P = D.demag_build_factors_nonuniform(edges, R)
        ref, adj = onu.apply_full(m, edges, R), onu.apply_full(m[0], edges, R, transpose=True)
    phi = torch.empty(n[2], n[1], n[0], device="cuda")
    D.demag_apply_full(P, dev((m * scale).astype(np.float32)), phi, prec)
    g = torch.empty(3, n[2], n[1], n[0], device="cuda")
    D.demag_apply_adjoint(P, dev((m[0] * scale).astype(np.float32)), g, prec)
    P.close()
    assert_close(host(phi).astype(np.float64) / scale, ref, TOL[prec], "forward")
    assert_close(host(g).astype(np.float64) / scale, adj, TOL[prec], "adjoint")
