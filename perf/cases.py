"""What the library is measured on: the calls of a micromagnetic program, by use.

Twelve listed cases and a generator of more of the same ranges.  Full tensors
in every arithmetic (FP32 is the default of the Python entry points and of the
autograd energy, FP64 the form others are checked against, BF16x3 / TF32x3 the
tensor-core forms), forward and adjoint, single grids and a batch of uneven
ones; the FFT convolution for the potential and the stray field; and the CP,
TT and Tucker formats.  Sizes go from 16 cells per axis, where a call is all
latency, to 256^3 cells and 4096 cells per axis, with odd and ragged sizes and
thin films among them.

`exact` restates the operator in 64-bit torch: the sinc-quadrature kernel is
summed in real space and applied by one zero-padded FFT convolution, the
structured formats by 1D convolutions of their factor columns.
"""
import math
import random

import torch

import paper_1212_3509_gb300 as D

C0 = 2.15


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest call: one application on a 16^3 test grid, where launches and latency count
        dict(name="full_16_fp32", kind="full", precision="fp32", n1=16, n2=16, n3=16, R=41),
        # one application in the default arithmetic on an everyday cube
        dict(name="full_128_fp32", kind="full", precision="fp32", n1=128, n2=128, n3=128, R=41),
        # one step of an energy minimisation through autograd (default arithmetic, ragged grid): forward and backward
        dict(name="gradient_75x60x45_fp32", kind="gradient", precision="fp32", n1=75, n2=60, n3=45, R=41),
        # a reference application in FP64, the form that other results are checked against
        dict(name="full_64_fp64", kind="full", precision="fp64", n1=64, n2=64, n3=64, R=41),
        # the headline: the largest full-format grid on tensor cores
        dict(name="full_256_bf16x3", kind="full", precision="bf16x3", n1=256, n2=256, n3=256, R=41),
        # the adjoint map of an optimisation with a field loss, FP32-grade tensor-core arithmetic, ragged grid
        dict(name="adjoint_115x96x70_tf32x3", kind="adjoint", precision="tf32x3", n1=115, n2=96, n3=70, R=41),
        # a parameter study: cubes and thin films of many sizes in one call
        dict(name="uneven_batch_16_bf16x3", kind="batch", precision="bf16x3", count=16, shapes=5, R=41),
        # the potential of the largest grid by one FFT convolution (its cost does not depend on R)
        dict(name="potential_fft_256", kind="potential_fft", n1=256, n2=256, n3=256, R=41),
        # the stray field of a time integrator's step on a ragged grid, by FFT
        dict(name="field_fft_150x100x60", kind="field_fft", n1=150, n2=100, n3=60, R=41),
        # CP tensors on 4096 cells per axis, many magnetizations at once
        dict(name="cp_4096_r4_b64", kind="cp", n1=4096, n2=4096, n3=4096, r=4, batch=64, R=61),
        # tensor trains on 1024 cells per axis
        dict(name="tt_1024_r8_b16", kind="tt", n1=1024, n2=1024, n3=1024, r1=8, r2=8, batch=16, R=61),
        # a single Tucker magnetization: its potential and its energy, no full tensor formed
        dict(name="tucker_energy_1024_r8", kind="tucker_energy", n1=1024, n2=1024, n3=1024, r1=8, r2=8, r3=8, R=61),
    ]


def _size(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _sizes(rng, lo, hi):
    return dict(n1=_size(rng, lo, hi), n2=_size(rng, lo, hi), n3=_size(rng, lo, hi))


def draw(rng):
    kind = rng.choice(["full", "gradient", "full64", "tensor", "tensor", "batch", "potential_fft", "field_fft", "cp",
                       "tt", "tucker_energy"])
    odd_R = 2 * rng.randint(10, 20) + 1
    if kind == "full":
        return dict(kind="full", precision="fp32", R=odd_R, **_sizes(rng, 8, 128))
    if kind == "gradient":
        return dict(kind="gradient", precision="fp32", R=odd_R, **_sizes(rng, 8, 75))
    if kind == "full64":
        return dict(kind="full", precision="fp64", R=odd_R, **_sizes(rng, 8, 64))
    if kind == "tensor":
        n = dict(n1=_size(rng, 17, 256), n2=_size(rng, 17, 256), n3=_size(rng, 3, 256))
        if rng.random() < 0.5:
            return dict(kind="full", precision="bf16x3", R=odd_R, **n)
        return dict(kind="adjoint", precision=rng.choice(["tf32x3", "bf16x3"]), R=odd_R,
                    **{p: min(v, 115) for p, v in n.items()})
    if kind == "batch":
        return dict(kind="batch", precision="bf16x3", count=rng.randint(3, 12), shapes=rng.randint(100, 999), R=odd_R)
    if kind in ("potential_fft", "field_fft"):
        return dict(kind=kind, R=odd_R, **_sizes(rng, 12, 256 if kind == "potential_fft" else 150))
    odd_R = 2 * rng.randint(20, 30) + 1
    if kind == "cp":
        n = _sizes(rng, 100, 4096)
        r = rng.randint(1, 6)
        room = 12288 * 4 * 64 // (r * sum(n.values()))
        return dict(kind="cp", r=r, batch=_size(rng, 1, max(1, min(64, room))), R=odd_R, **n)
    if kind == "tt":
        n = _sizes(rng, 100, 1024)
        return dict(kind="tt", r1=rng.randint(1, 8), r2=rng.randint(1, 8), batch=_size(rng, 1, 16), R=odd_R, **n)
    n = _sizes(rng, 100, 1024)
    return dict(kind="tucker_energy", r1=rng.randint(1, 8), r2=rng.randint(1, 8), r3=rng.randint(1, 8), R=odd_R, **n)


def _n(case):
    return case["n1"], case["n2"], case["n3"]


def _h(n):
    return (1.0 / max(n),) * 3  # cubic cells, longest edge 1


def _shapes(case):
    """The grids of a batch: cubes of 32 to 192 cells and two kinds of film, a fixed list per case."""
    rng = random.Random(case["shapes"])
    out = []
    for i in range(case["count"]):
        if i % 8 == 3:
            out.append((512, 512, 4))
        elif i % 8 == 7:
            out.append((256, 64, 8))
        else:
            out.append((rng.choice(range(32, 193, 16)),) * 3)
    return out


# ---------------------------------------------------------------- inputs

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _magnetization(n, seed):
    """A vortex about the domain's centre with 5% Gaussian noise, |m| = 1: float32 [3][n3][n2][n1]."""
    n1, n2, n3 = n
    h = _h(n)[0]
    x = ((torch.arange(n1, device="cuda", dtype=torch.float64) + 0.5 - 0.5 * n1) * h).view(1, 1, n1).expand(n3, n2, n1)
    y = ((torch.arange(n2, device="cuda", dtype=torch.float64) + 0.5 - 0.5 * n2) * h).view(1, n2, 1).expand(n3, n2, n1)
    m = torch.stack([-y, x, torch.full_like(x, 0.1)])
    m = m / m.norm(dim=0, keepdim=True)
    m = m + 0.05 * torch.randn(m.shape, generator=_generator(seed), device="cuda", dtype=torch.float64)
    return (m / m.norm(dim=0, keepdim=True)).float().contiguous()


def _smooth(n, rows, g):
    """Rows sum_s a_s sin(2 pi s x + t_s) over 8 harmonics at the cell centres of [0, 1]: float32 [rows][n]."""
    s = torch.arange(1, 9, device="cuda", dtype=torch.float64)
    a = torch.randn(rows, 8, generator=g, device="cuda", dtype=torch.float64) / s
    t = 2 * math.pi * torch.rand(rows, 8, generator=g, device="cuda", dtype=torch.float64)
    x = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n
    out = torch.zeros(rows, n, device="cuda", dtype=torch.float64)
    for i in range(8):
        out += a[:, i:i + 1] * torch.sin(2 * math.pi * s[i] * x + t[:, i:i + 1])
    return out.float()


def _factors(case, ranks, batch, seed):
    """Smooth factor columns, per item blocks (component, mode) of [rank][n_p]; also as {(q, p): [batch][rank][n_p]}."""
    g = _generator(seed)
    n = _n(case)
    blocks = {(q, p): _smooth(n[p], batch * ranks[p], g).view(batch, ranks[p], n[p]) for q in range(3) for p in range(3)}
    flat = torch.cat([blocks[q, p].reshape(batch, -1) for q in range(3) for p in range(3)], dim=1).contiguous()
    return flat, blocks


def _inputs(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_magnetization(n, seed + 1000003 * i) for i, n in enumerate(_shapes(case))]
    n = _n(case)
    if kind == "adjoint":  # a scalar field: a residual of order one, smooth part and noise
        m = _magnetization(n, seed)
        return (m[0] * m[1] + m[2]).contiguous()
    if kind == "cp":
        g = _generator(seed + 1)
        lam = 1.0 + 0.25 * torch.randn(case["batch"], 3, case["r"], generator=g, device="cuda")
        return (lam,) + _factors(case, (case["r"],) * 3, case["batch"], seed)
    if kind == "tt":
        g = _generator(seed)
        r1, r2, b = case["r1"], case["r2"], case["batch"]
        shapes = ((r1, n[0]), (r1 * r2, n[1]), (r2, n[2]))
        return tuple(torch.randn(b, 3, *s, generator=g, device="cuda") / math.sqrt((r1, r2, r2)[i])
                     for i, s in enumerate(shapes))
    if kind == "tucker_energy":
        r = (case["r1"], case["r2"], case["r3"])
        core = torch.randn(3, r[2], r[1], r[0], generator=_generator(seed + 1), device="cuda")
        return (core,) + _factors(case, r, 1, seed)
    return _magnetization(n, seed)


def prepare(case, seed):
    """The plan(s) with their workspace, the inputs and the output buffers that a program reuses from call to call."""
    kind = case["kind"]
    x = _inputs(case, seed)
    s = dict(case=case, x=x)
    if kind == "batch":
        s["plans"] = [D.demag_build_factors(n, _h(n), case["R"], C0) for n in _shapes(case)]
        for plan in s["plans"]:
            D.demag_reserve_workspace(plan, case["precision"])
        s["out"] = [torch.empty_like(m[0]) for m in x]
        return s
    n = _n(case)
    s["plan"] = plan = D.demag_build_factors(n, _h(n), case["R"], C0)
    if kind in ("full", "adjoint", "gradient"):
        D.demag_reserve_workspace(plan, case["precision"])
    if kind in ("full", "potential_fft"):
        s["out"] = torch.empty_like(x[0])
    elif kind == "adjoint":
        s["out"] = torch.empty(3, *x.shape, device="cuda")
    elif kind == "gradient":
        s["x"] = x.requires_grad_(True)
    elif kind == "field_fft":
        s["out"] = torch.empty_like(x)
    elif kind == "cp":
        b, r = case["batch"], case["r"]
        s["out"] = torch.empty(b, plan.M, 3, r, device="cuda"), torch.empty(b, plan.M * 3 * r * sum(n), device="cuda")
    elif kind == "tt":
        s["out"] = (torch.empty(case["batch"], plan.M, 3, device="cuda"),) + tuple(
            torch.empty(case["batch"], plan.M, *g.shape[1:], device="cuda") for g in x)
    elif kind == "tucker_energy":
        r = (case["r1"], case["r2"], case["r3"])
        s["out"] = (torch.empty(plan.M, 3, device="cuda"),
                    torch.empty(plan.M * 3 * sum(a * b for a, b in zip(r, n)), device="cuda"),
                    torch.empty((), dtype=torch.float64, device="cuda"))
    return s


def run(s):
    case, x = s["case"], s["x"]
    kind = case["kind"]
    if kind == "full":
        D.demag_apply_full(s["plan"], x, s["out"], case["precision"])
    elif kind == "adjoint":
        D.demag_apply_adjoint(s["plan"], x, s["out"], case["precision"])
    elif kind == "gradient":
        x.grad = None
        e = D.demag_energy_fn(x, s["plan"], case["precision"])
        e.backward()
        # the energy of FP32 fields is recorded beside them in their own precision
        return {"gradient": x.grad, "energy": e.detach().float()}
    elif kind == "batch":
        D.demag_apply_full_batched(s["plans"], x, s["out"], case["precision"])
    elif kind == "potential_fft":
        D.demag_apply_full_fft(s["plan"], x, s["out"])
    elif kind == "field_fft":
        D.demag_stray_field_fft(s["plan"], x, s["out"])
    elif kind == "cp":
        D.demag_apply_cp_batched(s["plan"], case["batch"], case["r"], x[0], x[1], *s["out"])
    elif kind == "tt":
        D.demag_apply_tt_batched(s["plan"], case["batch"], (case["r1"], case["r2"]), *x, *s["out"])
    elif kind == "tucker_energy":
        r = (case["r1"], case["r2"], case["r3"])
        w, v, e = s["out"]
        D.demag_apply_tucker(s["plan"], r, x[1], w, v)
        D.demag_energy_tucker(s["plan"], r, x[0], x[1], w, v, e)
        return {"weights": w, "factors": v, "energy": e.float()}
    return s["out"]


# ---------------------------------------------------------------- what a pass cannot do without

def _mode_products(n, M, per_axis):
    """Multiply-adds (2 flops) of the mode products; the even / odd halves of a Toeplitz factor need half of them."""
    return M * n[0] * n[1] * n[2] * sum(a * b for a, b in zip(per_axis, n))


def _fft3(n, fields):
    L = [max(2, 1 << (2 * v - 2).bit_length()) for v in n]
    pts = L[0] * L[1] * L[2]
    return fields * 2.5 * pts * math.log2(pts), L


def work(case):
    kind, M = case["kind"], (case["R"] - 1) // 2
    if kind == "batch":
        s = _shapes(case)
        return dict(bytes=sum(16 * a * b * c for a, b, c in s), flops=sum(_mode_products(n, M, (3, 3, 2)) for n in s))
    n = _n(case)
    N = n[0] * n[1] * n[2]
    if kind == "full":
        return dict(bytes=16 * N, flops=_mode_products(n, M, (3, 3, 2)))
    if kind == "adjoint":
        return dict(bytes=16 * N, flops=_mode_products(n, M, (2, 3, 3)))
    if kind == "gradient":
        return dict(bytes=24 * N, flops=_mode_products(n, M, (5, 6, 5)))
    if kind in ("potential_fft", "field_fft"):
        field = kind == "field_fft"
        flops, L = _fft3(n, 6 if field else 4)
        octant = (L[0] // 2 + 1) * (L[1] // 2 + 1) * (L[2] // 2 + 1)
        return dict(bytes=(24 if field else 16) * N + (24 if field else 12) * octant, flops=flops)
    if kind == "cp":
        cols = [case["r"]] * 3
    elif kind == "tt":
        cols = [case["r1"], case["r1"] * case["r2"], case["r2"]]
    else:
        cols = [case["r1"], case["r2"], case["r3"]]
    batch = case.get("batch", 1)
    entries = 3 * batch * sum(a * b for a, b in zip(cols, n))
    # one real transform of length 2n forward per column, one back per column and node
    flops = sum(3 * batch * a * (M + 1) * 2.5 * 2 * b * math.log2(2 * b) for a, b in zip(cols, n))
    return dict(bytes=4 * entries * (M + 1), flops=flops)


# ---------------------------------------------------------------- the same in 64 bits, by plain torch

def _nodes(R):
    M = (R - 1) // 2
    theta = C0 * math.log(M) / M
    t = theta * torch.arange(1, M + 1, device="cuda", dtype=torch.float64)
    return torch.sinh(t), 2 * theta * torch.cosh(t) * torch.sinh(t) ** 2 / (2 * math.pi ** 1.5)  # tau, c omega


def _generators(n, hh, tau):
    """E, F and their derivatives along the axis for d = -(n-1) .. n-1: [M][2n-1] each."""
    d = torch.arange(-(n - 1), n, device="cuda", dtype=torch.float64)
    t = tau[:, None]
    a, b = ((d.abs() - 0.5) * hh)[None, :], ((d.abs() + 0.5) * hh)[None, :]
    sign = torch.sign(d)[None, :]
    E = math.sqrt(math.pi) / (2 * t) * torch.where(a < 0, 2 * torch.special.erf(t * b),
                                                   torch.special.erfc(t * a) - torch.special.erfc(t * b))
    F = sign * torch.exp(-(t * a) ** 2) * -torch.expm1(-t * t * (2 * d.abs() * hh * hh)[None, :]) / (2 * t * t)
    dE = -2 * t * t * F
    dF = b * torch.exp(-(t * b) ** 2) - a * torch.exp(-(t * a) ** 2)
    return E, F, dE, dF


def _scale(n):
    h = _h(n)[0]
    s = max(n) * h
    return h / s, s


def _spectra(n, R, along=None):
    """The Fourier kernels of the three components; `along`: of the derivative of the potential along that axis."""
    hh, s = _scale(n)
    tau, w = _nodes(R)
    gens = [_generators(v, hh, tau) for v in n]
    L = [1 << (2 * v - 2).bit_length() for v in n]
    for q in range(3):
        T = []
        for p in range(3):
            g = gens[p][(1 if p == q else 0) + (2 if p == along else 0)]
            z = torch.zeros(len(tau), L[p], device="cuda", dtype=torch.float64)
            z[:, :n[p]] = g[:, n[p] - 1:]
            if n[p] > 1:
                z[:, L[p] - n[p] + 1:] = g[:, :n[p] - 1]
            T.append(z)
        plane = (T[1][:, :, None] * T[0][:, None, :]).reshape(len(tau), -1)
        K = ((w * (1.0 if along is not None else s))[:, None] * T[2]).T @ plane
        yield torch.fft.rfftn(K.view(L[2], L[1], L[0]))


def _spectrum(f, n):
    L = [1 << (2 * v - 2).bit_length() for v in n]
    return torch.fft.rfftn(f.double(), s=(L[2], L[1], L[0]))


def _back(S, n):
    L = [1 << (2 * v - 2).bit_length() for v in n]
    return torch.fft.irfftn(S, s=(L[2], L[1], L[0]))[:n[2], :n[1], :n[0]].contiguous()


def _potential(m, n, R, along=None):
    acc = None
    for q, K in enumerate(_spectra(n, R, along)):
        term = K * _spectrum(m[q], n)
        acc = term if acc is None else acc + term
    return _back(acc, n)


def _adjoint(y, n, R):
    Y = _spectrum(y, n)
    return torch.stack([-_back(K * Y, n) for K in _spectra(n, R)])


def _difference(n, h):
    """The second-order difference matrix: central inside, one-sided at the ends."""
    A = torch.zeros(n, n, device="cuda", dtype=torch.float64)
    if n == 2:
        A[:, 0], A[:, 1] = -1 / h, 1 / h
    elif n > 2:
        i = torch.arange(1, n - 1, device="cuda")
        A[i, i + 1], A[i, i - 1] = 0.5 / h, -0.5 / h
        A[0, :3] = torch.tensor([-3.0, 4.0, -1.0], dtype=torch.float64, device="cuda") / (2 * h)
        A[-1, -3:] = torch.tensor([1.0, -4.0, 3.0], dtype=torch.float64, device="cuda") / (2 * h)
    return A


_ALONG = ("ij,abj->abi", "ij,ajb->aib", "ij,jab->iab")


def _gradient(m, n, R):
    h = _h(n)[0]
    A = [_difference(v, h) for v in n]
    m = m.detach().double()
    phi = _potential(m, n, R)
    d = torch.stack([torch.einsum(_ALONG[p], A[p], phi) for p in range(3)])
    dtm = sum(torch.einsum(_ALONG[p], A[p].T, m[p]) for p in range(3))
    half = 0.5 * h ** 3
    return {"gradient": half * (d + _adjoint(dtm, n, R)), "energy": half * (m * d).sum()}


def _columns(v, n, hh, tau, kind):
    """T_k v for every node: v [batch][rows][n] -> [batch][M][rows][n]."""
    g = _generators(n, hh, tau)[kind]
    L = 1 << (2 * n - 2).bit_length()
    z = torch.zeros(len(tau), L, device="cuda", dtype=torch.float64)
    z[:, :n] = g[:, n - 1:]
    z[:, L - n + 1:] = g[:, :n - 1]
    S = torch.fft.rfft(z)
    X = torch.fft.rfft(v.double(), n=L)
    out = torch.empty(v.shape[0], len(tau), v.shape[1], n, device="cuda", dtype=torch.float64)
    for b in range(v.shape[0]):
        out[b] = torch.fft.irfft(S[:, None, :] * X[b][None], n=L)[..., :n]
    return out


def _mode(blocks, p, n, hh, tau):
    """Output block of mode p: [batch][M][3][rows][n_p] from {(q, p): [batch][rows][n_p]}."""
    return torch.stack([_columns(blocks[q, p], n[p], hh, tau, 1 if q == p else 0) for q in range(3)], dim=2)


def _structured(blocks, n, R):
    hh, s = _scale(n)
    tau, w = _nodes(R)
    return w * s, [_mode(blocks, p, n, hh, tau) for p in range(3)]


def exact(case, seed):
    kind, R = case["kind"], case["R"]
    x = _inputs(case, seed)
    if kind == "batch":
        return [_potential(m, n, R) for m, n in zip(x, _shapes(case))]
    n = _n(case)
    if kind in ("full", "potential_fft"):
        return _potential(x, n, R)
    if kind == "adjoint":
        return _adjoint(x, n, R)
    if kind == "gradient":
        return _gradient(x, n, R)
    if kind == "field_fft":
        return torch.stack([-_potential(x, n, R, along=p) for p in range(3)])
    if kind == "tt":
        blocks = {(q, p): x[p][:, q] for q in range(3) for p in range(3)}
        w, modes = _structured(blocks, n, R)
        return (w[None, :, None].expand(case["batch"], -1, 3).contiguous(), *modes)
    blocks = x[2]
    w, modes = _structured(blocks, n, R)
    flat = torch.cat([v.reshape(v.shape[0], -1) for v in modes], dim=1)
    if kind == "cp":
        return w[None, :, None, None] * x[0].double()[:, None], flat
    # Tucker: E = 1/2 V sum_q <m_q, D_q phi>, phi = sum_(k, q') w_k [[core_q'; T_(k, q', p) V_(q', p)]]
    h = _h(n)[0]
    core = x[0].double()
    energy = torch.zeros((), device="cuda", dtype=torch.float64)
    A = [_difference(v, h) for v in n]
    for q in range(3):
        V = [blocks[q, p][0].double() for p in range(3)]
        V[q] = V[q] @ A[q]  # <V, D W> = <D^T V, W>
        for q2 in range(3):
            G = [torch.einsum("an,kbn->kab", V[p], modes[p][0, :, q2]) for p in range(3)]
            t = torch.einsum("cba,kax->kcbx", core[q], G[0])
            t = torch.einsum("kcbx,kby->kcyx", t, G[1])
            t = torch.einsum("kcyx,kcz->kzyx", t, G[2])
            energy += (w[:, None, None, None] * t * core[q2][None]).sum()
    return {"weights": w[:, None].expand(-1, 3).contiguous(), "factors": flat[0], "energy": 0.5 * h ** 3 * energy}
