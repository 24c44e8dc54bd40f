"""The CUDA-core mode products (FP32 / FP64) at the edges of their tiles.

Axis lengths around the halves' tile widths (16, 32, 64 columns), the
contraction steps of 8, odd lengths (whose middle cell pairs with itself) and
axes of one to three cells, forward, adjoint and analytic field, uniform and
non-uniform, against the FP64 oracle at the tolerances of the forms.
"""
import numpy as np
import pytest

import synth
from gpu_helpers import TOL, assert_close, dev, host
from oracle import field as ofield
from oracle import full as ofull
from oracle import nonuniform as onu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (2, 1, 3), (1, 70, 2), (7, 8, 9), (15, 16, 17), (31, 33, 32), (64, 5, 65), (66, 34, 3),
          (4, 129, 6), (2, 3, 131), (130, 2, 18)]


@pytest.fixture(scope="module")
def D():
    import paper_1212_3509_gb300 as D
    return D


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n", SHAPES)
@pytest.mark.parametrize("R", [5, 41])
def test_forward_adjoint_field_vs_oracle(D, n, prec, R):
    h = (1 / max(n),) * 3
    P = D.demag_build_factors(n, h, R)
    m = synth.random_unit_m(n, 77)
    phi = torch.full((n[2], n[1], n[0]), float("nan"), device="cuda")
    D.demag_apply_full(P, dev(m), phi, prec)
    assert_close(host(phi), ofull.apply_full(m, n, h, R), TOL[prec], "forward")
    y = np.ascontiguousarray(m[0] * m[1] + m[2])
    g = torch.full((3, n[2], n[1], n[0]), float("nan"), device="cuda")
    D.demag_apply_adjoint(P, dev(y), g, prec)
    assert_close(host(g), ofull.apply_adjoint(y, n, h, R), TOL[prec], "adjoint")
    hd = torch.full_like(g, float("nan"))
    D.demag_stray_field_exact(P, dev(m), hd, prec)
    assert_close(host(hd), ofield.apply_field(m, n, h, R), TOL[prec], "field")
    P.close()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [(1, 2, 3), (17, 16, 33), (65, 3, 9), (5, 70, 31)])
def test_nonuniform_vs_oracle(D, n, prec):
    R = 41
    rng = np.random.default_rng(5)
    edges = [np.concatenate([[0.0], np.cumsum(0.5 + rng.random(v))]) for v in n]
    P = D.demag_build_factors_nonuniform(edges, R)
    m = synth.random_unit_m(n, 78)
    phi = torch.full((n[2], n[1], n[0]), float("nan"), device="cuda")
    D.demag_apply_full(P, dev(m), phi, prec)
    assert_close(host(phi), onu.apply_full(m, edges, R), TOL[prec], "forward")
    y = np.ascontiguousarray(m[0] - m[1] * m[2])
    g = torch.full((3, n[2], n[1], n[0]), float("nan"), device="cuda")
    D.demag_apply_adjoint(P, dev(y), g, prec)
    assert_close(host(g), onu.apply_full(y, edges, R, transpose=True), TOL[prec], "adjoint")
    P.close()
