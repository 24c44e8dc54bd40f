"""The structured energies at the edges of their Gram blocks.

Ranks around the 8 x 8 output blocks, contractions inside and beyond shared
memory, columns past one pass of the block (8192), axes of one and two cells,
against the contraction written out in float64 numpy.  FP32 factors, products
summed in FP32 over at most 32 columns: relative error of each Gram entry below
32 * 2^-24 * sum |a b|, so of the energy below 2e-6 * the same sum of absolute
values; the bound below is that sum.
"""
import numpy as np
import pytest

from gpu_helpers import dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _difference(n, h):
    A = np.zeros((n, n))
    if n == 2:
        A[:] = [[-1 / h, 1 / h]] * 2
    elif n > 2:
        i = np.arange(1, n - 1)
        A[i, i + 1], A[i, i - 1] = 0.5 / h, -0.5 / h
        A[0, :3] = np.array([-3.0, 4.0, -1.0]) / (2 * h)
        A[-1, -3:] = np.array([1.0, -4.0, 3.0]) / (2 * h)
    return A


def _apply_d(w, h):
    """Rows of w differenced without forming the matrix for long axes."""
    n = w.shape[1]
    if n < 3:
        return w @ _difference(n, h).T
    d = np.empty_like(w)
    d[:, 1:-1] = (w[:, 2:] - w[:, :-2]) / (2 * h)
    d[:, 0] = (-3 * w[:, 0] + 4 * w[:, 1] - w[:, 2]) / (2 * h)
    d[:, -1] = (3 * w[:, -1] - 4 * w[:, -2] + w[:, -3]) / (2 * h)
    return d


@pytest.mark.parametrize("n,r,rho", [((40, 33, 20), (1, 8, 9), (7, 9, 1)), ((64, 300, 65), (16, 17, 15), (17, 16, 64)),
                                     ((257, 2, 1), (8, 2, 1), (9, 2, 1)), ((9001, 5, 4), (3, 2, 2), (2, 3, 1)),
                                     ((70, 66, 64), (64, 64, 33), (64, 9, 64))])
def test_energy_of_one_tucker_potential(n, r, rho):
    import paper_1212_3509_gb300 as D
    rng = np.random.default_rng(11)
    h = (1 / 50, 1 / 40, 1 / 30)
    P = D.demag_build_factors(n, h, 5)
    core = rng.standard_normal((3, r[2], r[1], r[0])).astype(np.float32)
    V = [[rng.standard_normal((r[p], n[p])).astype(np.float32) for p in range(3)] for _ in range(3)]
    C = rng.standard_normal((rho[2], rho[1], rho[0])).astype(np.float32)
    U = [rng.standard_normal((rho[p], n[p])).astype(np.float32) for p in range(3)]
    e = torch.empty((), dtype=torch.float64, device="cuda")
    D.demag_energy_tucker_phi(P, r, dev(core.ravel()), dev(np.concatenate([V[q][p].ravel() for q in range(3)
                                                                            for p in range(3)])),
                              rho, dev(C.ravel()), dev(np.concatenate([u.ravel() for u in U])), e)
    ref = mag = 0.0
    for q in range(3):
        G, Ga = [], []
        for p in range(3):
            W = U[p].astype(np.float64)
            Wd = _apply_d(W, h[p]) if p == q else W
            G.append(V[q][p].astype(np.float64) @ Wd.T)
            Ga.append(np.abs(V[q][p].astype(np.float64)) @ np.abs(Wd).T)
        args = ("cba,ax,by,cz,zyx->",)
        ref += np.einsum(*args, core[q].astype(np.float64), *G, C.astype(np.float64), optimize=True)
        mag += np.einsum(*args, np.abs(core[q]).astype(np.float64), *Ga, np.abs(C).astype(np.float64), optimize=True)
    half = 0.5 * h[0] * h[1] * h[2]
    assert abs(e.item() - half * ref) <= 2e-6 * half * mag
    again = torch.empty_like(e)
    D.demag_energy_tucker_phi(P, r, dev(core.ravel()), dev(np.concatenate([V[q][p].ravel() for q in range(3)
                                                                            for p in range(3)])),
                              rho, dev(C.ravel()), dev(np.concatenate([u.ravel() for u in U])), again)
    assert again.item() == e.item()  # summed in a fixed order
    P.close()


def test_energy_on_two_streams_and_captured():
    """One plan's energies in flight on two streams, and in a graph: the same bits."""
    import paper_1212_3509_gb300 as D
    import synth
    n, r = (60, 40, 30), (3, 5, 20)
    P = D.demag_build_factors(n, (1 / 60,) * 3, 21)
    core, V = synth.tucker_inputs(n, r, 3)
    c, v = dev(core.ravel()), dev(V)
    tot = sum(a * b for a, b in zip(r, n))
    w, o = torch.empty(P.M * 3, device="cuda"), torch.empty(P.M * 3 * tot, device="cuda")
    D.demag_apply_tucker(P, r, v, w, o)
    e = [torch.zeros((), dtype=torch.float64, device="cuda") for _ in range(4)]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        D.demag_energy_tucker(P, r, c, v, w, o, e[0])
    g.replay()
    torch.cuda.synchronize()
    other = torch.cuda.Stream()
    other.wait_stream(torch.cuda.current_stream())
    for _ in range(3):
        D.demag_energy_tucker(P, r, c, v, w, o, e[1])
        D.demag_energy_tucker(P, r, c, v, w, o, e[2], stream=other)
        D.demag_energy_tucker(P, r, c, v, w, o, e[3])
    torch.cuda.synchronize()
    assert len({x.item() for x in e}) == 1
    del g  # the graph owns its scratch: gone before the plan
    P.close()
