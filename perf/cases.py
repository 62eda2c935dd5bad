"""What the framework's users have it do, as cases that can be timed one by one.

Every case goes through ``paper_2601_08077_gb300.df``, the library's binding, the way an SCF program does: the DF
tensor B of a molecule, its context and its output buffers are made once (``prepare``) and each pass (``run``) is one
call sequence on them.  A case's ``kind`` says which:

* ``scf``       the Coulomb and exchange build of one density and its energies (one SCF iteration at a Table 1 level);
* ``k``         the exchange build alone;
* ``geometry``  a new geometry: B split into its digit planes, then the first build;
* ``batch``     many molecules at once: their Coulomb builds, then their exchange builds, as captured graphs;
* ``gemm``      a stand-alone FP64-emulated product A B^T over INT8 slices;
* ``crt``       the same through residues, for a Gram matrix X X^T;
* ``mlp``       loss and gradients of the slice-count network over a training set.

The molecules are the synthetic ones the repository uses everywhere: atoms at random in a cube of constant density (or
along a chain), 5 s-type AO and 10 or 15 auxiliary exponents per atom, B from closed-form Coulomb integrals.  They are
made here on the GPU, in seconds less than the integral generator takes on the host; to keep that quick the metric is
factored in groups of 16 atoms (B's values then spread over the same range, with full FP64 mantissas).
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

GROUP_ATOMS = 16
LEVEL_SLICES = (3, 4, 5, 6)  # Table 1's levels 4..1


def listed():
    return [
        # the smallest molecule of the tests, early SCF iterations (level 4): launches and latency
        {"name": "scf-20atom-s3", "kind": "scf", "atoms": 20, "aux": 15, "nocc": 20, "s": 3, "shape": "cube", "packed": False},
        # a small molecule in mid-SCF (level 2); one 64-row tile of orbitals would hold its 60
        {"name": "scf-60atom-s5", "kind": "scf", "atoms": 60, "aux": 15, "nocc": 60, "s": 5, "shape": "cube", "packed": False},
        # odd nao, naux and nocc, B as packed triangles, level 3
        {"name": "scf-87atom-s4-packed", "kind": "scf", "atoms": 87, "aux": 15, "nocc": 87, "s": 4, "shape": "cube", "packed": True},
        # the 120-atom molecule at the first level that meets 1e-10
        {"name": "scf-120atom-s5", "kind": "scf", "atoms": 120, "aux": 15, "nocc": 120, "s": 5, "shape": "cube", "packed": False},
        # the benchmark's nao and nocc (240 atoms), with the smaller auxiliary set of 2 functions per AO
        {"name": "scf-240atom-s5", "kind": "scf", "atoms": 240, "aux": 10, "nocc": 250, "s": 5, "shape": "cube", "packed": False},
        # a Schwarz-screened chain: block-sparse B, the two builds in order
        {"name": "scf-chain160-s5", "kind": "scf", "atoms": 160, "aux": 15, "nocc": 160, "s": 5, "shape": "chain", "packed": False},
        # the exchange build at 8 slices, the FP64-like last iterations; odd nocc
        {"name": "k-100atom-s8", "kind": "k", "atoms": 100, "aux": 15, "nocc": 101, "s": 8, "shape": "cube", "packed": False},
        # a step of a geometry optimisation: new B, digit planes for every level, first iteration at level 4
        {"name": "geometry-90atom-s3", "kind": "geometry", "atoms": 90, "aux": 15, "nocc": 90, "s": 3, "shape": "cube", "packed": False},
        # a batch of uneven molecules
        {"name": "batch-16mol-s5", "kind": "batch", "molecules": 16, "low": 30, "high": 100, "mix": 1, "s": 5},
        # a square FP64-accurate product
        {"name": "gemm-2048-s7", "kind": "gemm", "m": 2048, "n": 2048, "k": 2048, "s": 7},
        # one auxiliary block's K_b of the 120-atom molecule by the CRT variant, at the accuracy of level 2
        {"name": "crt-gram-600x15360-n12", "kind": "crt", "m": 600, "k": 15360, "moduli": 12},
        # the slice-count network on the training set of 200 molecules
        {"name": "mlp-grad-6992", "kind": "mlp", "rows": 6992},
    ]


def _log(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    kind = rng.choice(("scf", "scf", "scf", "scf", "k", "geometry", "batch", "gemm", "crt", "mlp"))
    if kind in ("scf", "k", "geometry"):
        shape = "chain" if kind == "scf" and rng.random() < 0.2 else "cube"
        atoms = _log(rng, 60, 160) if shape == "chain" else _log(rng, 16, 160)
        nocc = max(8, int(round(atoms * rng.uniform(0.8, 1.1))))
        s = rng.choice((3, 4, 5, 6, 8)) if kind == "k" else rng.choice(LEVEL_SLICES)
        return {"kind": kind, "atoms": atoms, "aux": rng.choice((10, 15)), "nocc": nocc, "s": s, "shape": shape,
                "packed": kind == "scf" and shape == "cube" and rng.random() < 0.25}
    if kind == "batch":
        low = rng.randint(16, 50)
        return {"kind": "batch", "molecules": rng.randint(4, 16), "low": low, "high": low + rng.randint(10, 50),
                "mix": rng.randint(2, 1 << 20), "s": rng.choice(LEVEL_SLICES)}
    if kind == "gemm":
        return {"kind": "gemm", "m": _log(rng, 100, 6000), "n": _log(rng, 100, 3000), "k": _log(rng, 100, 3000),
                "s": rng.choice((3, 4, 5, 6, 7, 8))}
    if kind == "crt":
        return {"kind": "crt", "m": _log(rng, 100, 1000), "k": _log(rng, 1000, 32000), "moduli": rng.choice((8, 10, 12, 14))}
    return {"kind": "mlp", "rows": _log(rng, 300, 20000)}


# --- inputs -------------------------------------------------------------------

def _geometry(n, shape, rng):
    if shape == "chain":
        x = np.cumsum(rng.uniform(1.6, 2.2, n))
        return np.column_stack([x - x[0], rng.uniform(-0.4, 0.4, (n, 2))])
    edge = 10.0 * (n / 20.0) ** (1.0 / 3.0)
    pts = np.empty((n, 3))
    k = 0
    while k < n:
        p = rng.uniform(0.0, edge, 3)
        if k == 0 or np.min(((pts[:k] - p) ** 2).sum(1)) >= 1.5 ** 2:
            pts[k] = p
            k += 1
    return pts


def _tensor(atoms, aux, shape, rng):
    """B [naux, nao, nao] (every B_P exactly symmetric) of a molecule on the GPU."""
    dev, f64 = "cuda", torch.float64
    xyz = torch.from_numpy(_geometry(atoms, shape, rng)).to(dev)
    a = torch.from_numpy(np.tile(np.geomspace(0.1, 10.0, 5), atoms)).to(dev)
    c = torch.from_numpy(np.tile(np.geomspace(0.05, 20.0, aux), atoms)).to(dev)
    A, R = xyz.repeat_interleave(5, 0), xyz.repeat_interleave(aux, 0)
    nao, naux = a.numel(), c.numel()
    na, nc = (2.0 * a / math.pi) ** 0.75, (2.0 * c / math.pi) ** 0.75
    p = a[:, None] + a[None, :]
    wa = a[:, None, None] * A[:, None, :]
    ctr = (wa + wa.transpose(0, 1)) / p[:, :, None]
    r2 = ((A[:, None, :] - A[None, :, :]) ** 2).sum(-1)
    pair = (na[:, None] * na[None, :]) * torch.exp(-(a[:, None] * a[None, :]) / p * r2)
    if shape == "chain":  # Schwarz screening of the AO pairs at 1e-12
        best = ((2.0 * c / math.pi) ** 1.5 * 2.0 * math.pi ** 2.5 / (c * c * torch.sqrt(2.0 * c))).max()
        keep = torch.sqrt(pair ** 2 * 2.0 * math.pi ** 2.5 / (p * p * torch.sqrt(2.0 * p)) * best) >= 1e-12
        pair = torch.where(keep & keep.T, pair, torch.zeros_like(pair))

    def boys(t):
        u = torch.sqrt(torch.clamp(t, min=1e-12))
        return torch.where(t < 1e-8, 1.0 - t / 3.0, (0.5 * math.sqrt(math.pi)) * torch.erf(u) / u)

    B = torch.empty((naux, nao, nao), dtype=f64, device=dev)
    step = max(1, (1 << 26) // (nao * nao))
    for P0 in range(0, naux, step):
        q = c[P0:P0 + step, None, None]
        ps = p[None] + q
        d2 = torch.zeros((q.shape[0], nao, nao), dtype=f64, device=dev)
        for x in range(3):
            d2 += (ctr[None, :, :, x] - R[P0:P0 + step, x, None, None]) ** 2
        B[P0:P0 + step] = boys(p[None] * q / ps * d2) * pair[None] * (2.0 * math.pi ** 2.5) * nc[P0:P0 + step, None, None] / (
            p[None] * q * torch.sqrt(ps))
        del ps, d2
    size = GROUP_ATOMS * aux
    for P0 in range(0, naux, size):
        cg, Rg, ng = c[P0:P0 + size], R[P0:P0 + size], nc[P0:P0 + size]
        s = cg[:, None] + cg[None, :]
        V = boys(cg[:, None] * cg[None, :] / s * ((Rg[:, None, :] - Rg[None, :, :]) ** 2).sum(-1)) * (
            2.0 * math.pi ** 2.5) * ng[:, None] * ng[None, :] / (cg[:, None] * cg[None, :] * torch.sqrt(s))
        L = torch.linalg.cholesky(V)
        G = B[P0:P0 + size]
        G.copy_(torch.linalg.solve_triangular(L, G.reshape(cg.numel(), -1), upper=False).view_as(G))
        half = max(1, (1 << 27) // (nao * nao))
        for k in range(0, cg.numel(), half):
            H = G[k:k + half]
            H.copy_(0.5 * (H + H.transpose(1, 2)))
    return B


def _orbitals(nao, nocc, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    C = torch.linalg.qr(torch.randn((nao, nocc), generator=g, dtype=torch.float64, device="cuda"))[0].contiguous()
    D = 2.0 * C @ C.T
    return C, (0.5 * (D + D.T)).contiguous()


def _molecule(case, seed):
    B = _tensor(case["atoms"], case["aux"], case["shape"], np.random.default_rng(int(seed)))
    C, D = _orbitals(B.shape[1], case["nocc"], seed)
    return B, C, D


def _atoms(case):
    r = random.Random(case["mix"])
    return [r.randint(case["low"], case["high"]) for _ in range(case["molecules"])]


def _batch(case, seed):
    for i, n in enumerate(_atoms(case)):
        yield _molecule({"atoms": n, "aux": 15, "shape": "cube", "nocc": n}, 1000 * int(seed) + i)


def _rows(m, k, seed):
    """Rows of an X block: entries of a few orders of magnitude, one scale per row."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    x = torch.randn((m, k), generator=g, dtype=torch.float64, device="cuda")
    return (x * torch.exp2(4.0 * torch.randn((m, 1), generator=g, dtype=torch.float64, device="cuda"))).contiguous()


def _training_set(case, seed):
    """Block features in their scaled ranges, the slice counts as classes, a He-initialised network."""
    rng = np.random.default_rng(int(seed))
    X = rng.uniform(-1.0, 1.0, (case["rows"], 16)).astype(np.float32)
    X[:, 15] = 1.0
    y = rng.integers(1, 7, case["rows"]).astype(np.int32)
    parts = []
    for rows, cols in ((64, 16), (64, 64), (8, 64)):
        parts += [rng.standard_normal((rows, cols)) * np.sqrt(2.0 / cols), 0.1 * rng.standard_normal(rows)]
    return X, y, np.concatenate([q.ravel() for q in parts]).astype(np.float32)


# --- the passes ---------------------------------------------------------------

def prepare(case, seed):
    from paper_2601_08077_gb300 import df
    kind = case["kind"]
    if kind in ("scf", "k", "geometry"):
        B, C, D = _molecule(case, seed)
        naux, nao, _ = B.shape
        ctx = df.Context(nao, naux, case["nocc"], 6 if kind == "geometry" else case["s"])
        if case["packed"]:
            iu = torch.triu_indices(nao, nao, device=B.device)
            B = B[:, iu[0], iu[1]].contiguous()
            ctx.setup_packed(B)
        elif kind != "geometry":
            ctx.setup(B)
        J, K = torch.empty_like(D), torch.empty_like(D)
        rho = torch.empty(naux, dtype=torch.float64, device=D.device)
        return {"case": case, "ctx": ctx, "B": B, "C": C, "D": D, "J": J, "K": K, "rho": rho}
    if kind == "batch":
        ctxs, Cs, Ds, Js, Ks = [], [], [], [], []
        for B, C, D in _batch(case, seed):
            ctx = df.Context(B.shape[1], B.shape[0], C.shape[1], case["s"])
            ctx.setup(B)
            ctxs.append(ctx)
            Cs.append(C)
            Ds.append(D)
            Js.append(torch.empty_like(D))
            Ks.append(torch.empty_like(D))
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        return {"case": case, "batch": df.Batch(ctxs), "stream": stream, "C": Cs, "D": Ds, "J": Js, "K": Ks}
    if kind == "gemm":
        return {"case": case, "A": _rows(case["m"], case["k"], seed), "B": _rows(case["n"], case["k"], seed + 1000003)}
    if kind == "crt":
        return {"case": case, "A": _rows(case["m"], case["k"], seed)}
    X, y, params = _training_set(case, seed)
    return {"case": case, "net": df.MLP(params), "X": torch.from_numpy(X).cuda(), "y": torch.from_numpy(y).cuda()}


def run(state):
    from paper_2601_08077_gb300 import df
    case = state["case"]
    kind = case["kind"]
    if kind == "k":
        K, _ = state["ctx"].build_K(state["C"], case["s"], state["K"])
        return {"K": K}
    if kind in ("scf", "geometry"):
        ctx = state["ctx"]
        if kind == "geometry":
            ctx.setup(state["B"])
        J, rho, K, _ = ctx.build_JK(state["D"], state["C"], case["s"], state["J"], state["rho"], state["K"])
        return {"J": J, "rho": rho, "K": K, "E": list(ctx.energy(state["D"], J, K, rho))}
    if kind == "batch":
        b, st = state["batch"], state["stream"]
        b.build_J(state["D"], state["J"], stream=st)
        b.build_K(state["C"], case["s"], state["K"], stream=st)
        return {"J": state["J"], "K": state["K"]}
    if kind == "gemm":
        return df.emulated_gemm(state["A"], state["B"], case["s"])
    if kind == "crt":
        return df.emulated_gemm_crt(state["A"], state["A"], case["moduli"])
    grad, loss = state["net"].gradients(state["X"], state["y"])
    return {"grad": grad, "loss": loss}


def _sizes(case):
    return 5 * case["atoms"], case["aux"] * case["atoms"], case["nocc"]


def _build_work(nao, naux, nocc, s, coulomb):
    """B's upper triangles, the orbitals (and the density) in, K (and J, rho) out; the slice products of the exchange."""
    half = nao * (nao + 1) // 2
    by = 8.0 * (naux * half + nao * nocc + nao * nao)
    if coulomb:
        by += 8.0 * (2 * nao * nao + naux)
    return {"bytes": by, "flops": s * (s + 1) // 2 * (2.0 * nocc * nao * nao * naux + 2.0 * half * naux * nocc)}


def work(case):
    kind = case["kind"]
    if kind in ("scf", "k", "geometry"):
        nao, naux, nocc = _sizes(case)
        w = _build_work(nao, naux, nocc, case["s"], kind != "k")
        if kind == "geometry":  # the dense B in, six digit planes (one byte a digit) and the row exponents out
            w["bytes"] += 4.0 * naux * nao * (nao - 1) + 6.0 * naux * nao * nao + 4.0 * naux * nao
        if case["shape"] == "chain":  # about 60 neighbours of each AO survive the screening
            kept = min(1.0, 60.0 / nao)
            w = {"bytes": kept * w["bytes"], "flops": w["flops"] * (1.0 + kept) / 2.0}
        return w
    if kind == "batch":
        ws = [_build_work(5 * n, 15 * n, n, case["s"], True) for n in _atoms(case)]
        return {"bytes": sum(w["bytes"] for w in ws), "flops": sum(w["flops"] for w in ws)}
    if kind == "gemm":
        m, n, k, s = case["m"], case["n"], case["k"], case["s"]
        return {"bytes": 8.0 * (m * k + n * k + m * n), "flops": s * (s + 1) // 2 * 2.0 * m * n * k}
    if kind == "crt":
        m, k = case["m"], case["k"]
        return {"bytes": 8.0 * (m * k + m * m), "flops": case["moduli"] * 2.0 * m * m * k}
    return {"bytes": 4.0 * (17 * case["rows"] + 2 * 5768), "flops": 6.0 * 5632 * case["rows"]}


# --- the same in 64 bits --------------------------------------------------------

def _exact_build(B, C, D):
    naux, nao, _ = B.shape
    rho = B.reshape(naux, -1) @ D.reshape(-1)
    J = (rho @ B.reshape(naux, -1)).view(nao, nao)
    K = torch.zeros_like(J)
    step = max(1, (1 << 28) // (nao * C.shape[1]))
    for P0 in range(0, naux, step):
        X = (B[P0:P0 + step].reshape(-1, nao) @ C).view(-1, nao, C.shape[1]).transpose(0, 1).reshape(nao, -1)
        K += X @ X.T
    return J, rho, K


def exact(case, seed):
    kind = case["kind"]
    if kind in ("scf", "k", "geometry"):
        B, C, D = _molecule(case, seed)
        J, rho, K = _exact_build(B, C, D)
        if kind == "k":
            return {"K": K}
        E = [0.5 * float((D * J).sum()), 0.5 * float((rho * rho).sum()), -0.5 * float((D * K).sum())]
        return {"J": J, "rho": rho, "K": K, "E": E}
    if kind == "batch":
        got = [_exact_build(*m) for m in _batch(case, seed)]
        return {"J": [g[0] for g in got], "K": [g[2] for g in got]}
    if kind == "gemm":
        return _rows(case["m"], case["k"], seed) @ _rows(case["n"], case["k"], seed + 1000003).T
    if kind == "crt":
        A = _rows(case["m"], case["k"], seed)
        return A @ A.T
    X, y, params = _training_set(case, seed)
    p, ws, at = torch.from_numpy(params).double().cuda(), [], 0
    for shape in ((64, 16), (64,), (64, 64), (64,), (8, 64), (8,)):
        n = math.prod(shape)
        ws.append(p[at:at + n].view(shape).requires_grad_())
        at += n
    h = torch.from_numpy(X).double().cuda()
    h = torch.relu(h @ ws[0].T + ws[1])
    h = torch.relu(h @ ws[2].T + ws[3])
    loss = torch.nn.functional.cross_entropy(h @ ws[4].T + ws[5], torch.from_numpy(y).long().cuda())
    grads = torch.autograd.grad(loss, ws)
    return {"grad": torch.cat([g.reshape(-1) for g in grads]), "loss": float(loss.detach())}
