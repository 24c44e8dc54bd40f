"""Each node of a structured application is as exact as its own generator allows.

Two nodes share a complex transform in the register kernel, and a transform's
rounding errors are relative to the whole of it; neighbouring nodes differ by a
factor of up to 40 (F at the last nodes of R = 61, 129 cells).  A column's error
must all the same lie within eps log2(L) |t_k|_1 |x|_2 of the node's own
generator t_k (forward, product and inverse of a normwise stable transform).
"""
import numpy as np
import pytest

from gpu_helpers import dev, host
from oracle import structured as ost

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,R", [(129, 61), (129, 41), (160, 61), (256, 61), (400, 61), (1024, 61), (2048, 41),
                                 (129, 63)])
@pytest.mark.parametrize("kind", ["random", "smooth", "constant"])
def test_every_node_within_its_own_bound(n, R, kind):
    import paper_1212_3509_gb300 as D
    r, dims = 3, (n, n, 20)
    rng = np.random.default_rng(n + R)

    def columns(length):
        if kind == "random":
            return rng.standard_normal((r, length))
        x = (np.arange(length) + 0.5) / length
        return np.cos(np.pi * np.arange(1, r + 1)[:, None] * x) if kind == "smooth" else np.ones((r, length))

    U = np.concatenate([columns(dims[p]).ravel() for _ in range(3) for p in range(3)]).astype(np.float32)
    h = (1.0 / n,) * 3
    P = D.demag_build_factors(dims, h, R)
    M = P.M
    w = torch.empty(1, M, 3, r, device="cuda")
    out = torch.full((1, M * 3 * r * sum(dims)), float("nan"), device="cuda")
    D.demag_apply_cp_batched(P, 1, r, dev(np.ones((1, 3, r), np.float32)), dev(U[None]), w, out)
    got = host(out)[0]
    P.close()
    V = ost._split_blocks(U, dims, (r, r, r))
    _, hh = ost.scaled_spacing(dims, h)
    tau = ost.sinc_nodes(M, 2.15)[2]
    at = 0
    for p in range(2):  # the two axes of n cells: types F and E at components 0 and 1
        size, L = M * 3 * r * n, 1 << (2 * n - 1).bit_length()
        g = got[at:at + size].reshape(M, 3, r, n).astype(np.float64)
        at += size
        for q in range(2):
            gen = ost.gen_F if ost.factor_kind(p, q) == "F" else ost.gen_E
            X = np.fft.rfft(V[q][p], 2 * L)
            for k in range(M):
                t = gen(tau[k], hh[p], n)
                c = np.zeros(2 * L)
                c[:n], c[2 * L - n + 1:] = t[n - 1:], t[:n - 1]
                ref = np.fft.irfft(np.fft.rfft(c) * X)[:, :n]
                bound = 2.0 ** -24 * np.log2(L) * np.abs(t).sum() * np.linalg.norm(V[q][p], axis=1)
                assert (np.linalg.norm(g[k, q] - ref, axis=1) <= bound).all(), (p, q, k)


def test_symbols_of_a_short_axis_beside_a_long_one():
    """The register kernel's table follows its own axes: 200 cells beside 4096 cost a few MB and not the
    table of the long axis once more (25 MB at M = 128)."""
    import paper_1212_3509_gb300 as D
    used = []
    for n1 in (100, 200, 100, 200):  # 100 cells have no such table; the first two load what is loaded once
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        P = D.demag_build_factors((n1, 4096, 1), (1 / 4096,) * 3, 257)
        torch.cuda.synchronize()
        used.append(free - torch.cuda.mem_get_info()[0])
        P.close()
    assert used[3] - used[2] < 8 << 20, used
