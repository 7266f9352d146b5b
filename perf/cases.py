"""The work a user of the library has it do, as measured cases.

Every case goes through the package's public calls (`Plan`, `polyspectrum`, `estimate_batched`): a
seeded density field in device memory, a plan that the program keeps, one call, whole outputs.

The kinds of call:
- "estimate": `Plan.estimate`, the polyspectrum of one field (order 2 to 5, any precision, `ell` > 0 a
  redshift-space multipole);
- "connected": `Plan.estimate` and `Plan.disconnected`, what a user subtracts for the connected trispectrum;
- "backward": `Plan.backward`, the gradient of a weighted sum of the bins;
- "train": the autograd op `polyspectrum`, forward and backward, as in a field-level fit;
- "mocks": `estimate_batched` over realisations of three grid sizes;
- "fullshape": `Plan.trispectrum_full` of one shell quadruple.

`exact` restates the estimator in plain torch, in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1904_11055_gb300 as ps

L = 1000.0  # box side; only the normalisation depends on it
GRIDS = (16, 24, 32, 48, 64, 96, 128, 160, 256)


# ------------------------------------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest useful call: a quick look at a small simulation; latency and launches count
        dict(name="bispec32_bf16", kind="estimate", N=32, order=3, nshell=8, width=1.0, prec="split_bf16", ell=0),
        # the plain method in double precision on a small Gaussian field: the reference run of a pipeline
        dict(name="bispec64_fp64", kind="estimate", N=64, order=3, nshell=16, width=1.0, prec="fp64", ell=0),
        # a batch of mock catalogues of mixed grid sizes, for a covariance
        dict(name="mocks_bf16", kind="mocks", N=128, order=3, nshell=32, width=1.0, prec="split_bf16", ell=0),
        # the bispectrum of a large simulation, the headline workload, and the same on the CUDA cores
        dict(name="bispec256_bf16", kind="estimate", N=256, order=3, nshell=64, width=1.0, prec="split_bf16", ell=0),
        dict(name="bispec256_fp32", kind="estimate", N=256, order=3, nshell=64, width=1.0, prec="fp32", ell=0),
        # the trispectrum of a large simulation in wide shells
        dict(name="trispec256_bf16", kind="estimate", N=256, order=4, nshell=32, width=1.5, prec="split_bf16", ell=0),
        # the connected trispectrum of a middle-sized one in plain single precision
        dict(name="trispec128_fp32", kind="connected", N=128, order=4, nshell=20, width=1.5, prec="fp32", ell=0),
        # the gradient at the headline size, and a fit's forward and backward at a middle one
        dict(name="grad256_bf16", kind="backward", N=256, order=3, nshell=64, width=1.0, prec="split_bf16", ell=0),
        dict(name="train128_fp32", kind="train", N=128, order=3, nshell=40, width=1.0, prec="fp32", ell=0),
        # the redshift-space quadrupole
        dict(name="quad160_bf16", kind="estimate", N=160, order=3, nshell=48, width=1.0, prec="split_bf16", ell=2),
        # a higher order
        dict(name="pent128_bf16", kind="estimate", N=128, order=5, nshell=20, width=1.0, prec="split_bf16", ell=0),
        # one full-shape trispectrum bin, 22 x 22 diagonal bins
        dict(name="full256", kind="fullshape", N=256, order=4, nshell=32, width=1.5, prec="split_bf16", ell=0,
             k1=10, k2=10, k3=10, k4=10, ndiag=22, dwidth=1.5),
    ]


def _kmax(nshell, width):
    """The largest integer wavevector component inside the outermost shell."""
    e2 = (width * (nshell + 0.5)) ** 2
    K = int(math.sqrt(e2)) + 1
    while K * K >= e2:
        K -= 1
    return K


def draw(rng):
    """One more case of the same ranges: any grid and order, 3 shells to as many as the grid resolves without
    wrapped closures, unit and wider shells, every precision and call."""
    top = _cost(max(listed(), key=_cost))
    while True:
        kind = rng.choice(["estimate"] * 5 + ["connected", "backward", "backward", "train", "train", "mocks", "fullshape"])
        prec = rng.choice(["split_bf16", "split_bf16", "fp32", "fp64"])
        order = rng.choice([2, 3, 3, 3, 4, 4, 5])
        ell = rng.choice([0, 0, 0, 2, 4]) if kind == "estimate" and order in (3, 4) else 0
        if kind in ("connected", "fullshape"):
            order = 4
        if kind in ("backward", "train"):
            order = rng.choice([3, 3, 4])
        if kind == "mocks":
            order, prec = 3, "fp32" if prec == "fp32" else "split_bf16"
        N = 128 if kind == "mocks" else rng.choice(GRIDS)
        width = rng.choice([1.0, 1.0, 1.25, 1.5, 2.0])
        wrap_at = 96 if kind == "mocks" else N
        hi = 1  # the most shells whose closures do not wrap
        while order * _kmax(hi + 1, width) < wrap_at and 2 * _kmax(hi + 1, width) + 1 <= wrap_at and hi < 64:
            hi += 1
        if order == 5:
            hi = min(hi, 20)
        if order == 4 and prec == "split_bf16":
            hi = min(hi, 16 if ell else 34)  # the tensor-core path takes no more
        if hi < 3:
            continue
        nshell = min(hi, int(round(math.exp(rng.uniform(math.log(3.0), math.log(hi + 0.49))))))
        case = dict(kind=kind, N=N, order=order, nshell=nshell, width=width, prec=prec, ell=ell)
        if kind == "fullshape":
            m = min(nshell, 12)
            for t in ("k1", "k2", "k3", "k4"):
                case[t] = rng.randint(max(1, m // 2), m)
            # diagonals up to about the longest that the quadrilaterals have, in bins of about the shells' width
            case["dwidth"] = width * rng.choice([0.5, 1.0, 1.0, 2.0])
            case["ndiag"] = min(64, int(width * (case["k1"] + max(case["k2"], case["k3"]) + 1) / case["dwidth"]) + 1)
        if kind == "estimate" and order == 2 and N < 32:
            continue  # a power spectrum of a few hundred cells is no one's workload
        if _cost(case) <= top:
            return case


# ------------------------------------------------------------------------------------------------ inputs
def _edges(case):
    return case["width"] * (np.arange(case["nshell"] + 1) + 0.5)


def _field(N, seed, dtype):
    """A lognormal density contrast with P ~ k^-1.5 exp(-(k / (N/4))^2), unit variance before the map."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    w = torch.randn((N, N, N), generator=g, device="cuda", dtype=torch.float64)
    m = torch.fft.fftfreq(N, device="cuda", dtype=torch.float64) * N
    mz = torch.arange(N // 2 + 1, device="cuda", dtype=torch.float64)
    k2 = m[:, None, None] ** 2 + m[None, :, None] ** 2 + mz[None, None, :] ** 2
    amp = k2.clamp(min=1.0) ** -0.375 * torch.exp(-0.5 * k2 / (N / 4.0) ** 2)
    amp[0, 0, 0] = 0.0
    x = torch.fft.irfftn(torch.fft.rfftn(w) * amp, s=(N, N, N))
    x = (x - x.mean()) / x.std()
    return (torch.exp(x - 0.5) - 1.0).to(dtype)


def _mock_grids(case):
    """(grid, realisations) of a batch."""
    return ((128, 4), (96, 2), (160, 2))


def _weights(case, bins, seed):
    """dL/dB of a fit: a normal residual per bin over the bin's expected scatter, prod_t sqrt(P(k_t) / k_t)."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 77_777)
    r = torch.randn(len(bins), generator=g, device="cuda", dtype=torch.float64)
    k = case["width"] * torch.as_tensor(np.asarray(bins, dtype=np.float64), device="cuda")
    return r * torch.exp(0.5 * (2.5 * torch.log(k) + (k / (case["N"] / 4.0)) ** 2)).prod(dim=1)


def _dtype(case):
    return torch.float64 if case["prec"] == "fp64" else torch.float32


def prepare(case, seed):
    e, kind = _edges(case), case["kind"]
    if kind == "mocks":
        plans, fields = [], []
        for i, (N, count) in enumerate(_mock_grids(case)):
            plan = ps.Plan(N, L, case["order"], e, case["prec"], ps.POLY_ALLOW_ALIAS)
            for r in range(count):
                plans.append(plan)
                fields.append(_field(N, seed * 101 + 10 * i + r, _dtype(case)))
        outs = [torch.empty(p.nbins, dtype=torch.float64, device="cuda") for p in plans]
        return dict(kind=kind, plans=plans, fields=fields, outs=outs)
    plan = ps.Plan(case["N"], L, case["order"], e, case["prec"], 0, case["ell"])
    state = dict(kind=kind, plan=plan, delta=_field(case["N"], seed, _dtype(case)))
    if kind in ("backward", "train"):
        state["w"] = _weights(case, plan.bins, seed)
    if kind == "train":
        state["delta"].requires_grad_(True)
    if kind == "fullshape":
        state["k"] = [case["k1"], case["k2"], case["k3"], case["k4"]]
        state["dedges"] = case["dwidth"] * np.arange(case["ndiag"] + 1)
    return state


def run(state):
    kind = state["kind"]
    if kind == "mocks":
        return ps.estimate_batched(state["plans"], state["fields"], state["outs"])
    plan, delta = state["plan"], state["delta"]
    if kind == "estimate":
        return plan.estimate(delta)
    if kind == "connected":
        return {"B": plan.estimate(delta), "disc": plan.disconnected(delta)}
    if kind == "backward":
        return plan.backward(delta, state["w"])
    if kind == "train":
        delta.grad = None
        B = ps.polyspectrum(delta, plan)
        B.backward(state["w"])
        return {"B": B.detach(), "grad": delta.grad}
    T, C = plan.trispectrum_full(delta, state["k"], state["dedges"])
    return {"T": T, "counts": C}


# ------------------------------------------------------------------------------------------------ work
def _bins(case):
    """The bins in the library's order: k1 >= ... >= kn, kn fastest, polygon rule on the shell centres."""
    ns, n = case["nshell"], case["order"]
    b = np.arange(1, ns + 1)[:, None]
    for _ in range(n - 1):
        rep = b[:, -1]
        head = np.repeat(b, rep, axis=0)
        first = np.cumsum(rep) - rep
        last = np.arange(rep.sum()) - np.repeat(first, rep) + 1
        b = np.concatenate([head, last[:, None]], axis=1)
    return b[b[:, 0] <= b[:, 1:].sum(axis=1) + 1e-9 * b[:, 0]] if n > 1 else b


def _distinct(a):
    return 0 if a.shape[1] < 2 else len(np.unique(a, axis=0))


def _fft_flops(N, count):
    return count * 2.5 * N ** 3 * math.log2(float(N) ** 3)  # real transforms


def _sum_flops(case, N):
    """Products of each row and column formed once, one multiply-add per bin and cell."""
    b, n = _bins(case), case["order"]
    ra = {2: 1, 3: 2, 4: 2, 5: 2, 6: 3}[n]
    prods = _distinct(b[:, :ra]) * (ra - 1) + _distinct(b[:, ra:]) * (n - ra - 1)
    return float(N) ** 3 * (prods + 2.0 * len(b))


def _grad_flops(case, N):
    """One multiply-add per distinct (shell, other shells) and cell; the products of the others formed once."""
    b, n = _bins(case), case["order"]
    ent = np.concatenate([np.concatenate([b[:, t:t + 1], np.delete(b, t, axis=1)], axis=1) for t in range(n)])
    return float(N) ** 3 * (2.0 * len(np.unique(ent, axis=0)) + _distinct(np.unique(ent[:, 1:], axis=0)) * (n - 2))


def _shell_modes(case, s):
    e = _edges(case)
    K = _kmax(case["nshell"], case["width"])
    m = np.arange(-K, K + 1)
    x, y, z = np.meshgrid(m, m, m, indexing="ij")
    q2 = (x * x + y * y + z * z).astype(np.float64)
    at = (q2 >= e[s - 1] ** 2) & (q2 < e[s] ** 2) & (q2 > 0)
    return np.stack([x[at], y[at], z[at]], axis=1)


def _quads(case):
    """Closed quadrilaterals of the full-shape bin, from the pair sums' histograms."""
    S = [_shell_modes(case, case[t]) for t in ("k1", "k2", "k3", "k4")]
    K = max(int(np.abs(s).max()) for s in S)
    M = 4 * K + 1
    hat = []
    for s in S:
        a = np.zeros((M, M, M), dtype=np.float32)
        a[s[:, 0] % M, s[:, 1] % M, s[:, 2] % M] = 1.0
        hat.append(np.fft.rfftn(a))
    return float(np.fft.irfftn(hat[0] * hat[1] * hat[2] * hat[3], s=(M, M, M))[0, 0, 0])


def work(case):
    N, ns, kind = case["N"], case["nshell"], case["kind"]
    es = 8 if case["prec"] == "fp64" else 4
    nb = len(_bins(case))
    if kind == "mocks":
        byt = fl = 0.0
        for G, count in _mock_grids(case):
            byt += count * (es * float(G) ** 3 + 8 * nb)
            fl += count * (_sum_flops(case, G) + _fft_flops(G, 1 + ns))
        return {"bytes": byt, "flops": fl}
    grid = es * float(N) ** 3
    if kind == "fullshape":
        # per quadrilateral a real part of a complex product and its sum, and the diagonal's length
        return {"bytes": grid + 16 * case["ndiag"] ** 2, "flops": _fft_flops(N, 1) + 10.0 * _quads(case)}
    fields = 2 * ns if case["ell"] else ns
    est = _sum_flops(case, N) + _fft_flops(N, 1 + fields)
    if kind == "estimate":
        return {"bytes": grid + 8 * nb, "flops": est}
    if kind == "connected":
        return {"bytes": grid + 16 * nb, "flops": est}
    grad = _grad_flops(case, N) + _fft_flops(N, 2 + ns)
    if kind == "backward":
        return {"bytes": 2 * grid + 8 * nb, "flops": grad + _fft_flops(N, ns)}
    return {"bytes": 2 * grid + 16 * nb, "flops": est + grad}


def _cost(case):
    """Time in arbitrary units: flops over the rate of the units that the precision runs on."""
    rate = {"fp64": 1.0, "fp32": 70.0, "split_bf16": 70.0 if case["order"] == 4 and case["kind"] in ("backward", "train")
            else 400.0}[case["prec"]]
    return work(case)["flops"] / rate


# ------------------------------------------------------------------------------------------------ tolerances
def tolerance(case):
    """About four times the largest distances from `exact` seen over the listed and a hundred drawn cases (2-norm:
    fp64 3e-15, fp32 6e-7, split_bf16 4.3e-5 and its gradients 3.4e-6; "max", one value's over the outputs' root
    mean square or itself: 1.5e-14, 2.7e-6, 1.1e-4 and 4.6e-5)."""
    if case["kind"] == "fullshape":  # FP32 in the split-BF16 plans too
        return {"fp64": {"rel": 2e-14, "max": 1e-13}}.get(case["prec"], {"rel": 2.5e-6, "max": 1e-5})
    if case["kind"] == "backward" and case["prec"] == "split_bf16":
        return {"rel": 1.4e-5, "max": 2e-4}
    return {"fp64": {"rel": 2e-14, "max": 1e-13}, "fp32": {"rel": 2.5e-6, "max": 1e-5},
            "split_bf16": {"rel": 1.7e-4, "max": 4.5e-4}}[case["prec"]]


# ------------------------------------------------------------------------------------------------ exact
def _shell_of(N, e):
    """Shell index of every mode of the half spectrum of an N^3 real field (-1: none), and q_z / |q|."""
    m = torch.round(torch.fft.fftfreq(N, device="cuda", dtype=torch.float64) * N)
    mz = torch.arange(N // 2 + 1, device="cuda", dtype=torch.float64)
    q2 = m[:, None, None] ** 2 + m[None, :, None] ** 2 + mz[None, None, :] ** 2
    s = torch.bucketize(q2, torch.as_tensor(e ** 2, device="cuda"), right=True) - 1
    s[(s >= len(e) - 1) | (q2 == 0)] = -1
    return s, mz[None, None, :] / q2.clamp(min=1.0).sqrt()


def _legendre(ell, mu):
    p0, p1 = torch.ones_like(mu), mu
    for n in range(1, ell):
        p0, p1 = p1, ((2 * n + 1) * mu * p1 - n * p0) / (n + 1)
    return p1 if ell else p0


def _shell_fields(F, shell, ns, N, weight=None):
    """D_s(x) = sum over the shell's modes of F e^{+iqx} (unnormalised), [ns, N^3]."""
    D = torch.empty((ns, N ** 3), dtype=torch.float64, device="cuda")
    for s in range(ns):
        G = torch.where(shell == s, F if weight is None else F * weight, 0.0)
        D[s] = torch.fft.irfftn(G, s=(N, N, N), norm="forward").reshape(-1)
    return D


def _groups(bins):
    """For every k2 (or k1 for n = 2): its rows (first legs), columns (the other legs) and the places of its bins."""
    n = bins.shape[1]
    ra = 1 if n == 2 else 2
    for k in np.unique(bins[:, ra - 1]):
        at = np.flatnonzero(bins[:, ra - 1] == k)
        rows, ri = np.unique(bins[at, :ra], axis=0, return_inverse=True)
        cols, ci = np.unique(bins[at, ra:], axis=0, return_inverse=True)
        yield rows - 1, cols - 1, at, ri.reshape(-1), ci.reshape(-1)


def _sums(bins, D, D1, w=None, step=1 << 19):
    """S_b = sum_x prod_t D_{b_t}(x), the first leg from D1; w: cell weights."""
    S = torch.zeros(len(bins), dtype=torch.float64, device="cuda")
    groups = [(r, c, torch.as_tensor(a, device="cuda"), torch.as_tensor(i, device="cuda"), torch.as_tensor(j, device="cuda"))
              for r, c, a, i, j in _groups(bins)]
    step = min(step, max(1 << 14, (1 << 30) // max(1, max(len(g[0]) + len(g[1]) for g in groups))))
    for x in range(0, D.shape[1], step):
        d, d1 = D[:, x:x + step], D1[:, x:x + step]
        for rows, cols, at, ri, ci in groups:
            A = d1[rows[:, 0]]
            if rows.shape[1] > 1:
                A = A * d[rows[:, 1]]
            if w is not None:
                A = A * w[x:x + step]
            Bc = d[cols[:, 0]]
            for t in range(1, cols.shape[1]):
                Bc = Bc * d[cols[:, t]]
            S[at] += (A @ Bc.T)[ri, ci]
    return S


def _count_sums(bins, case, N):
    """sum_x prod_t iota_{b_t}(x) over one cell of each orbit of the cube's symmetries, with the orbits' sizes."""
    shell, _ = _shell_of(N, _edges(case))
    h = N // 2
    i = torch.arange(h + 1, device="cuda")
    x, y, z = torch.meshgrid(i, i, i, indexing="ij")
    at = (x <= y) & (y <= z)
    x, y, z = x[at], y[at], z[at]
    perms = torch.where((x == y) & (y == z), 1.0, torch.where((x == y) | (y == z), 3.0, 6.0)).double()
    for v in (x, y, z):
        perms = perms * torch.where((v == 0) | (2 * v == N), 1.0, 2.0)
    cell = (x * N + y) * N + z
    one = torch.ones((N, N, N // 2 + 1), dtype=torch.complex128, device="cuda")
    iota = torch.empty((case["nshell"], len(cell)), dtype=torch.float64, device="cuda")
    for s in range(case["nshell"]):
        f = torch.fft.irfftn(torch.where(shell == s, one, 0.0), s=(N, N, N), norm="forward").reshape(-1)
        iota[s] = f[cell]
    return _sums(bins, iota, iota, perms)


def _norm(case, N):
    return (2 * case["ell"] + 1) * (L ** 3) ** (case["order"] - 1) / float(N) ** (3 * case["order"])


def _exact_estimate(case, N, delta, sums=True):
    bins = _bins(case)
    shell, mu = _shell_of(N, _edges(case))
    F = torch.fft.rfftn(delta.double())
    D = _shell_fields(F, shell, case["nshell"], N)
    D1 = D if case["ell"] == 0 else _shell_fields(F, shell, case["nshell"], N, _legendre(case["ell"], mu))
    C = _count_sums(bins, case, N)
    B = torch.where(C.abs() > 0.5 * N ** 3, _norm(case, N) * _sums(bins, D, D1) / C, 0.0) if sums else None
    return B, D, C, shell, F


def _exact_grad(case, N, D, C, shell, g, step=1 << 18):
    """sum_m irfft(mask_m rfft(G_m)), G_m = dL/dD_m by automatic differentiation of the products, slab by slab."""
    bins = _bins(case)
    w = torch.where(C.abs() > 0.5 * N ** 3, _norm(case, N) * g / C, 0.0)
    groups = [(r, c, torch.as_tensor(i, device="cuda"), torch.as_tensor(j, device="cuda"), torch.as_tensor(a, device="cuda"))
              for r, c, a, i, j in _groups(bins)]
    G = torch.zeros_like(D)
    for x in range(0, D.shape[1], step):
        d = D[:, x:x + step].detach().clone().requires_grad_(True)
        for rows, cols, ri, ci, at in groups:
            W = torch.zeros((len(rows), len(cols)), dtype=torch.float64, device="cuda")
            W[ri, ci] = w[at]
            A = d[rows[:, 0]] * d[rows[:, 1]] if rows.shape[1] > 1 else d[rows[:, 0]]
            Bc = d[cols[:, 0]] * d[cols[:, 1]] if cols.shape[1] > 1 else d[cols[:, 0]]
            (A * (W @ Bc)).sum().backward()
        G[:, x:x + step] = d.grad
    H = torch.zeros((N, N, N // 2 + 1), dtype=torch.complex128, device="cuda")
    for s in range(case["nshell"]):
        H += torch.where(shell == s, torch.fft.rfftn(G[s].reshape(N, N, N)), 0.0)
    return torch.fft.irfftn(H, s=(N, N, N), norm="forward")


def _exact_disc(case, N, C, shell, F):
    bins = _bins(case)
    twice = torch.full((N // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
    twice[0] = 1.0
    p2 = (F.real ** 2 + F.imag ** 2) * twice
    P = torch.stack([torch.where(shell == s, p2, 0.0).sum() for s in range(case["nshell"])])
    b = torch.as_tensor(bins - 1, device="cuda")
    k1, k2, k3, k4 = b[:, 0], b[:, 1], b[:, 2], b[:, 3]
    pair = ((k1 == k2) & (k3 == k4)) * P[k1] * P[k3] + ((k1 == k3) & (k2 == k4)) * P[k1] * P[k2] \
        + ((k1 == k4) & (k2 == k3)) * P[k1] * P[k2]
    return torch.where(C.abs() > 0.5 * N ** 3, _norm(case, N) * float(N) ** 3 * pair / C, 0.0)


def _exact_full(case, delta):
    """T and counts of the full-shape bin: every (q1, q2) pair against the (q3, q4) pairs that close it."""
    N, nd = case["N"], case["ndiag"]
    S = [torch.as_tensor(_shell_modes(case, case[t]), device="cuda") for t in ("k1", "k2", "k3", "k4")]
    F = torch.fft.fftn(delta.double())
    M = 4 * max(int(s.abs().max()) for s in S) + 1
    if M > N:
        return None  # closures that wrap around the grid are left to the library's own tests
    f = [F[s[:, 0] % N, s[:, 1] % N, s[:, 2] % N] for s in S]
    key = lambda q: ((q[..., 0] + M // 2) * M + q[..., 1] + M // 2) * M + q[..., 2] + M // 2  # noqa: E731
    k34 = key(-(S[2][:, None, :] + S[3][None, :, :])).reshape(-1)
    p34 = (f[2][:, None] * f[3][None, :]).reshape(-1)
    i3 = torch.arange(len(S[2]), device="cuda").repeat_interleave(len(S[3]))
    order = torch.argsort(k34)
    p34, i3 = p34[order], i3[order]
    have = torch.bincount(k34, minlength=M ** 3)
    first = torch.cumsum(have, 0) - have
    e2 = torch.as_tensor((case["dwidth"] * np.arange(nd + 1)) ** 2, device="cuda")
    T = torch.zeros(nd * nd, dtype=torch.float64, device="cuda")
    C = torch.zeros(nd * nd, dtype=torch.int64, device="cuda")
    bin_of = lambda q: torch.bucketize((q * q).sum(-1).double(), e2, right=True) - 1  # noqa: E731
    d13 = bin_of(S[0][:, None, :] - S[2][None, :, :])
    for i in range(len(S[0])):
        k12 = key(S[0][i] + S[1])
        d1 = bin_of(S[0][i] - S[1])
        n = torch.where((d1 >= 0) & (d1 < nd), have[k12], 0)
        j = torch.arange(len(S[1]), device="cuda").repeat_interleave(n)
        at = first[k12][j] + torch.arange(len(j), device="cuda") - (torch.cumsum(n, 0) - n)[j]
        d2 = d13[i][i3[at]]
        keep = (d2 >= 0) & (d2 < nd)
        cell = torch.where(keep, d1[j] * nd + d2, nd * nd)
        v = ((f[0][i] * f[1])[j] * p34[at]).real
        T += torch.bincount(cell, weights=torch.where(keep, v, 0.0), minlength=nd * nd + 1)[:-1]
        C += torch.bincount(cell, minlength=nd * nd + 1)[:-1]
    norm = (L ** 3) ** 3 / float(N) ** 12
    return {"T": torch.where(C > 0, norm * T / C.clamp(min=1), 0.0).reshape(nd, nd), "counts": C.reshape(nd, nd)}


def exact(case, seed):
    kind, N = case["kind"], case["N"]
    state = prepare(case, seed)  # the same inputs
    if kind == "mocks":
        return [_exact_estimate(case, f.shape[0], f)[0] for f in state["fields"]]
    delta = state["delta"].detach()
    if kind == "fullshape":
        return _exact_full(case, delta)
    B, D, C, shell, F = _exact_estimate(case, N, delta, sums=kind != "backward")
    if kind == "estimate":
        return B
    if kind == "connected":
        return {"B": B, "disc": _exact_disc(case, N, C, shell, F)}
    grad = _exact_grad(case, N, D, C, shell, state["w"])
    return grad if kind == "backward" else {"B": B, "grad": grad}
