"""Tile widths and CTAs per SM of the tensor-core launches, and the node sum's groups.

Tiles of at most 128 columns run two CTAs per SM, wider ones one; a batch cuts
wide tiles where they are the minority.  Neither changes the MMA sequence of an
output element, so batched and single applications agree bit for bit; the node
sum of a grid of few rows is split into more groups, checked against the oracle.
"""
import pytest

import synth
from gpu_helpers import TOL, assert_close, dev, host
from oracle import full as ofull

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    import paper_1212_3509_gb300 as D
    return D


# halves of 128 / 129 (the two widths), of one tile and more, of few rows
@pytest.mark.parametrize("prec", ["bf16x3", "tf32x3"])
@pytest.mark.parametrize("n", [(256, 20, 18), (257, 18, 20), (18, 260, 17), (17, 20, 300), (24, 24, 24), (17, 17, 17),
                               (600, 17, 18)])
def test_single_application_vs_oracle(D, n, prec):
    h = (1 / max(n),) * 3
    P = D.demag_build_factors(n, h, 41)
    m = synth.random_unit_m(n, 31)
    phi = torch.full((n[2], n[1], n[0]), float("nan"), device="cuda")
    for _ in range(2):  # the second call finds the work counters as the first one left them
        phi.fill_(float("nan"))
        D.demag_apply_full(P, dev(m), phi, prec)
    D.demag_sync_status(P)
    assert_close(host(phi), ofull.apply_full(m, n, h, 41), TOL[prec])
    P.close()


@pytest.mark.parametrize("prec", ["bf16x3", "tf32x3"])
@pytest.mark.parametrize("shapes", [[(300, 40, 20), (64, 64, 64), (80, 70, 60)],    # wide tiles cut
                                    [(300, 300, 20), (24, 24, 24)]])                # wide tiles kept
def test_batch_equals_single_calls(D, shapes, prec):
    plans = [D.demag_build_factors(n, (1 / max(n),) * 3, 21) for n in shapes]
    ms = [dev(synth.random_unit_m(n, 40 + i)) for i, n in enumerate(shapes)]
    single = [torch.empty(n[2], n[1], n[0], device="cuda") for n in shapes]
    for P, m, o in zip(plans, ms, single):
        D.demag_apply_full(P, m, o, prec)
    out = [torch.full_like(o, float("nan")) for o in single]
    D.demag_apply_full_batched(plans, ms, out, prec)
    for a, b in zip(out, single):
        assert torch.equal(a, b)
    for P in plans:
        D.demag_sync_status(P)
        P.close()
