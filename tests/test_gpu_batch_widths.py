"""Column tiles with neighbours leave each other's columns alone.

The tensor-core epilogue stores whole boxes of 32 columns where the output goes
through TMA (the next axis a multiple of 32 cells in the split layout; axis 3:
axis 1).  A launch of several column tiles per half therefore needs widths that
are multiples of 32: in a batch that cuts a wide tile, and in a width read from
a tuning cache.  Tile widths do not change an output element's arithmetic, so
the results equal those of single, untuned calls bit for bit.
"""
import json

import numpy as np
import pytest

import synth
from gpu_helpers import dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    import paper_1212_3509_gb300 as D
    return D


def _plan(D, n, uniform, R):
    if uniform:
        return D.demag_build_factors(n, (1 / max(n),) * 3, R)
    rng = np.random.default_rng(sum(n))
    return D.demag_build_factors_nonuniform([np.concatenate(([0.0], np.cumsum(rng.uniform(0.5, 1.5, v)))) / max(n)
                                             for v in n], R)


# the wide axis first (halves of 150, 200, 132; 150 cells of a non-uniform grid), second and third;
# the other grid carries most of the output, so that the wide tiles are cut
@pytest.mark.parametrize("prec", ["bf16x3", "tf32x3"])
@pytest.mark.parametrize("n,uniform", [((300, 64, 64), True), ((400, 64, 32), True), ((264, 32, 20), True),
                                       ((40, 300, 64), True), ((64, 40, 300), True), ((150, 64, 40), False)])
def test_cut_tiles_equal_single_calls(D, n, uniform, prec):
    shapes = [(n, uniform), ((128, 128, 128), True)]
    plans = [_plan(D, s, u, 11) for s, u in shapes]
    ms = [dev(synth.random_unit_m(s, 50 + i)) for i, (s, _) in enumerate(shapes)]
    single = [torch.empty(s[2], s[1], s[0], device="cuda") for s, _ in shapes]
    for P in plans:
        D.demag_set_fused(P, False)
    for P, m, o in zip(plans, ms, single):
        D.demag_apply_full(P, m, o, prec)
    for _ in range(3):
        out = [torch.full_like(o, float("nan")) for o in single]
        D.demag_apply_full_batched(plans, ms, out, prec)
        for a, b in zip(out, single):
            assert torch.equal(a, b)
    for P in plans:
        D.demag_sync_status(P)
        P.close()


def test_cached_width_that_splits_a_store_box_is_not_taken(D, tmp_path):
    n, R = (300, 64, 64), 11
    m = dev(synth.random_unit_m(n, 60))
    path = tmp_path / "tune.jsonl"
    P = _plan(D, n, True, R)
    a = torch.empty(n[2], n[1], n[0], device="cuda")
    D.demag_apply_full(P, m, a, "bf16x3")
    P.close()
    P = _plan(D, n, True, R)
    D.demag_autotune(P, True)
    b = torch.empty_like(a)
    D.demag_apply_full(P, m, b, "bf16x3")
    D.demag_autotune_save(P, str(path))
    kinds = [D.demag_autotune_entry(P, i) for i in range(D.demag_autotune_count(P))]
    P.close()
    assert torch.equal(a, b)
    assert any(e["kind"] == "bf16x3_tile_width" and e["key"][0] == 0 for e in kinds)
    lines = [json.loads(t) for t in path.read_text().splitlines()]
    for t in lines:
        if t["kind"] == 1:  # BF16x3 tile width: 80 columns would end inside a box
            t["value"] = 80
    path.write_text("".join(json.dumps(t, separators=(",", ":")) + "\n" for t in lines))
    P = _plan(D, n, True, R)
    assert D.demag_autotune_load(P, str(path)) == len(lines)
    for _ in range(3):
        b.fill_(float("nan"))
        D.demag_apply_full(P, m, b, "bf16x3")
        assert torch.equal(a, b)
    P.close()


@pytest.mark.parametrize("shapes", [[((256, 256, 300), True), ((300, 300, 12), False), ((64, 64, 64), False)],
                                    [((256, 256, 40), True), ((300, 20, 18), False)],
                                    [((512, 512, 4), False), ((128, 64, 64), True)]])
def test_batch_of_fused_grids_films_and_chains(D, shapes):
    """Only the groups that run decide how wide tiles are taken: the mode-3 stage of a fused grid, not its
    unused chain stages; the stages of a film without its last one."""
    plans = [_plan(D, n, True, 11) for n, _ in shapes]
    ms = [dev(synth.random_unit_m(n, 70 + i)) for i, (n, _) in enumerate(shapes)]
    single = [torch.empty(n[2], n[1], n[0], device="cuda") for n, _ in shapes]
    for P, (_, fused), m, o in zip(plans, shapes, ms, single):
        D.demag_set_fused(P, fused)
        D.demag_apply_full(P, m, o, "bf16x3")
    out = [torch.full_like(o, float("nan")) for o in single]
    D.demag_apply_full_batched(plans, ms, out, "bf16x3")
    for a, b in zip(out, single):
        assert torch.equal(a, b)
    for P in plans:
        D.demag_sync_status(P)
        P.close()
