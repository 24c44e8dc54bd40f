"""The 3D FFT passes at every transform length and at the edges of their tiles.

FFT lengths 32 to 512 run in registers with 2 to 32 lanes per fibre and 16 to
128 fibres per block, shorter and longer ones by in-place passes; each axis
takes each length here, with fibre counts around and between whole blocks, for
the potential and the field, against the FP64 oracle.
"""
import pytest

import synth
from gpu_helpers import TOL, assert_close, dev, host
from oracle import field as ofield
from oracle import full as ofull

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# lengths per axis: 16/32/64, 64/32/128, 128/256/32, 256/32/64, 512/64/16, 32/512/64, 32/64/512, 128/128/128, 4/256/256, 1024/32/32
SHAPES = [(8, 9, 17), (32, 16, 33), (64, 65, 12), (128, 15, 31), (129, 20, 7), (16, 256, 18), (10, 31, 256),
          (33, 64, 60), (2, 100, 127), (257, 9, 16)]


@pytest.mark.parametrize("n", SHAPES)
def test_potential_and_field_vs_oracle(n):
    import paper_1212_3509_gb300 as D
    h, R = (1 / max(n),) * 3, 21
    P = D.demag_build_factors(n, h, R)
    m = synth.random_unit_m(n, 60 + sum(n))
    phi = torch.full((n[2], n[1], n[0]), float("nan"), device="cuda")
    D.demag_apply_full_fft(P, dev(m), phi)
    assert_close(host(phi), ofull.apply_full(m, n, h, R), TOL["fp32"], "potential")
    hd = torch.full((3, n[2], n[1], n[0]), float("nan"), device="cuda")
    D.demag_stray_field_fft(P, dev(m), hd)
    assert_close(host(hd), ofield.apply_field(m, n, h, R), TOL["fp32"], "field")
    P.close()
