"""Which schedule an application on tensor cores takes: tuned or by size.

Told apart by the launches of one call.  Forward: operand split, three stages or
the fused kernel and its mode-3 stage, reduction (5 or 4); adjoint the same;
stray field: split, eight stages or three times two, three reductions (12 or 10).
"""
import json

import pytest

import synth
from gpu_helpers import dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CHAIN, FUSED = (5, 5, 12), (4, 4, 10)


@pytest.fixture(scope="module")
def D():
    import paper_1212_3509_gb300 as D
    return D


def _launches(D, P):
    """Launches of the second forward, adjoint and stray-field call (the first ones prepare)."""
    n = P.n
    m = dev(synth.random_unit_m(n, 3))
    phi = torch.empty(n[2], n[1], n[0], device="cuda")
    v = torch.empty(3, n[2], n[1], n[0], device="cuda")
    calls = (lambda: D.demag_apply_full(P, m, phi, "bf16x3"), lambda: D.demag_apply_adjoint(P, phi, v, "bf16x3"),
             lambda: D.demag_stray_field_exact(P, m, v, "bf16x3"))
    out = []
    for call in calls:
        call()
        before = D.demag_launch_count(P)
        call()
        out.append(D.demag_launch_count(P) - before)
    D.demag_sync_status(P)
    return tuple(out)


@pytest.mark.parametrize("fused", [0, 1])
def test_every_direction_follows_the_tuned_choice(D, fused, tmp_path):
    n, R = (64, 48, 40), 11  # by size: the chain
    path = tmp_path / "tune.jsonl"
    P = D.demag_build_factors(n, (1 / 64,) * 3, R)
    D.demag_autotune(P, True)
    D.demag_reserve_workspace(P, "bf16x3")
    D.demag_autotune_save(P, str(path))
    chosen = [e["value"] for e in (D.demag_autotune_entry(P, i) for i in range(D.demag_autotune_count(P)))
              if e["kind"] == "bf16x3_schedule"]
    assert len(chosen) == 1
    assert _launches(D, P) == (FUSED if chosen[0] else CHAIN)
    P.close()
    lines = [json.loads(t) for t in path.read_text().splitlines()]
    for t in lines:
        if t["kind"] == 9:
            t["value"] = fused
    path.write_text("".join(json.dumps(t, separators=(",", ":")) + "\n" for t in lines))
    P = D.demag_build_factors(n, (1 / 64,) * 3, R)
    assert D.demag_autotune_load(P, str(path)) == len(lines)
    assert _launches(D, P) == (FUSED if fused else CHAIN)
    P.close()


# forward line 4.5e6 of ext1^2 ext2 (with fewer than 8 nodes 1.5e6 and 2^20 cells), the others' 1.2e7; grids
# whose number of cells says otherwise among them
@pytest.mark.parametrize("n,R,forward,others", [
    ((160, 160, 17), 41, 0, 0), ((128, 96, 96), 41, 0, 0), ((53, 204, 181), 41, 0, 0),  # 4.1e6, 1.6e6, 0.9e6
    ((176, 160, 20), 41, 1, 0), ((240, 208, 20), 17, 1, 0),                             # 5.0e6, 11.98e6
    ((240, 224, 20), 17, 1, 1), ((256, 256, 17), 5, 1, 1),                              # 12.9e6, 16.8e6
    ((128, 96, 96), 15, 1, 0), ((128, 96, 96), 17, 0, 0), ((128, 96, 64), 15, 0, 0),    # 7 and 8 nodes; few cells
    ((53, 204, 181), 11, 0, 0), ((96, 128, 128), 11, 0, 0)])                            # many cells, short first axis
def test_untuned_choice_by_size(D, n, R, forward, others):
    P = D.demag_build_factors(n, (1 / max(n),) * 3, R)
    got = _launches(D, P)
    assert D.demag_forward_schedule(P, "bf16x3") == forward
    P.close()
    assert got == ((FUSED if forward else CHAIN)[0],) + (FUSED if others else CHAIN)[1:]
