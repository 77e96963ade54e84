"""The work that programs have this library do, as cases that can be timed and compared.

A case is a dict of plain values; prepare() makes what a program has in hand before the call
(inputs on the GPU and a handle), run() is one pass through the public entry points, work() what
one pass cannot do without, exact() the result in 64 bits by plain torch.

Products: the cores of a train are fixed only up to a change of basis on every bond, so a product
is returned as the tensor that its cores stand for, contracted as a program does that evaluates
the field on its grid. The sizes are such that this tensor fits in memory.

Kinds of input trains:
  random    Gaussian cores, left-canonical (the small and the batched products, the losses);
  spectral  right-canonical with a 1/k profile on every bond (the benchmark's inputs);
  field     a random-phase field with an energy spectrum k^(-5/3) and a viscous cut-off on a
            periodic grid of d^L points (1, 2 or 3 dimensions for d = 2, 4, 8, digits interleaved,
            coarsest first), compressed to bond chi.
"""

import math

import numpy as np
import torch

import paper_2410_19747_gb300 as ttm


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


# ---------------------------------------------------------------- cases

def listed():
    return [
        # The smallest product in use: ten sites, bond 8, nothing truncated. Bound by launches.
        {"name": "random_small", "op": "multiply", "kind": "random", "L": 10, "d": 2, "chiA": 8, "chiB": 8,
         "eps": 0.0, "chi_max": 0, "chi_out": 0, "prec": "fp64", "graph": 0},
        # A time stepper that multiplies fields of one shape again and again: captured once, replayed.
        {"name": "field1d_graph", "op": "multiply", "kind": "field", "L": 12, "d": 2, "chiA": 12, "chiB": 12,
         "eps": 1e-12, "chi_max": 24, "chi_out": 24, "prec": "fp64", "graph": 1},
        # A long one-dimensional field, middling bonds, float64.
        {"name": "field1d", "op": "multiply", "kind": "field", "L": 20, "d": 2, "chiA": 48, "chiB": 48,
         "eps": 1e-14, "chi_max": 64, "chi_out": 64, "prec": "fp64", "graph": 0},
        # Two-dimensional turbulence on 1024 x 1024, the product u v at bond 64, float64.
        {"name": "field2d", "op": "multiply", "kind": "field", "L": 10, "d": 4, "chiA": 64, "chiB": 64,
         "eps": 1e-14, "chi_max": 64, "chi_out": 64, "prec": "fp64", "graph": 0},
        # Three-dimensional advective term, uneven bonds, mixed mode.
        {"name": "field3d", "op": "multiply", "kind": "field", "L": 6, "d": 8, "chiA": 96, "chiB": 70,
         "eps": 1e-14, "chi_max": 96, "chi_out": 96, "prec": "bf16_split", "graph": 0},
        # The benchmark's inputs and options (mixed mode, the cap binds) on a shorter train.
        {"name": "spectral_large", "op": "multiply", "kind": "spectral", "L": 18, "d": 2, "chiA": 160, "chiB": 160,
         "eps": 1e-14, "chi_max": 160, "chi_out": 160, "prec": "bf16_split", "graph": 0},
        # Eight pairs of uneven bonds in one batched call, mixed mode.
        {"name": "batch_uneven", "op": "batch", "kind": "random", "n": 8, "L": 12, "d": 2, "chi_lo": 16, "chi_hi": 64,
         "eps": 1e-14, "chi_max": 48, "chi_out": 0, "prec": "bf16_split"},
        # Odd sizes throughout, wide Swaps and a final rounding to a smaller output bond.
        {"name": "rounded_odd", "op": "multiply", "kind": "field", "L": 11, "d": 3, "chiA": 27, "chiB": 23,
         "eps": 1e-13, "chi_max": 45, "chi_out": 21, "prec": "fp64", "graph": 0},
        # The overlap of two large trains (norms, distances, the error measure of a compression).
        {"name": "inner_large", "op": "inner", "L": 30, "d": 2, "chiA": 512, "chiB": 300},
        # A training step on <W, A o B>: value and the gradients of every core of A and B.
        {"name": "grad_inner", "op": "grad", "loss": "inner", "L": 20, "d": 4, "chiA": 64, "chiB": 64, "chiW": 64},
        # A training step on || A o B - C ||^2 at small bonds.
        {"name": "grad_sqdist", "op": "grad", "loss": "sqdist", "L": 10, "d": 4, "chiA": 12, "chiB": 12, "chiW": 12},
        # The plain matrix product on the tensor cores at float64 accuracy.
        {"name": "gemm_split", "op": "gemm", "M": 1500, "N": 1024, "K": 2000, "prec": "bf16_split"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges. Sizes stay below those of the largest listed case."""
    op = rng.choice(["multiply"] * 6 + ["batch", "inner", "grad", "gemm"])
    if op == "multiply":
        kind = rng.choice(["random", "field", "field", "field", "spectral"])
        prec = rng.choice(["fp64", "bf16_split"])
        graph = 1 if rng.random() < 0.2 else 0
        if kind == "random":
            L = rng.randint(6, 12)
            return {"op": op, "kind": kind, "L": L, "d": 2, "chiA": _log_int(rng, 3, 12), "chiB": _log_int(rng, 3, 12),
                    "eps": 0.0, "chi_max": 0, "chi_out": 0, "prec": prec, "graph": graph}
        if kind == "spectral":
            chi = _log_int(rng, 24, 128)
            return {"op": op, "kind": kind, "L": rng.randint(14, 17), "d": 2, "chiA": chi, "chiB": max(4, chi - rng.randint(0, 9)),
                    "eps": 1e-14, "chi_max": chi, "chi_out": chi, "prec": prec, "graph": graph}
        d = rng.choice([2, 2, 3, 4, 4, 8])
        L = {2: rng.randint(12, 20), 3: rng.randint(7, 11), 4: rng.randint(6, 10), 8: rng.randint(4, 6)}[d]
        chi = _log_int(rng, 8, {2: 64, 3: 48, 4: 64, 8: 64}[d])
        return {"op": op, "kind": kind, "L": L, "d": d, "chiA": chi, "chiB": max(4, chi - rng.randint(0, chi // 3)),
                "eps": rng.choice([1e-14, 1e-13, 1e-12, 1e-10]), "chi_max": chi + rng.randint(0, chi // 2),
                "chi_out": rng.choice([0, chi]), "prec": prec, "graph": graph}
    if op == "batch":
        lo = rng.randint(4, 16)
        return {"op": op, "kind": "random", "n": rng.randint(2, 8), "L": rng.randint(8, 12), "d": 2, "chi_lo": lo,
                "chi_hi": lo + rng.randint(4, 40), "eps": 1e-14, "chi_max": rng.randint(24, 48), "chi_out": 0,
                "prec": rng.choice(["fp64", "bf16_split"])}
    if op == "inner":
        return {"op": op, "L": rng.randint(10, 30), "d": rng.choice([2, 3, 4]), "chiA": _log_int(rng, 16, 256),
                "chiB": _log_int(rng, 16, 256)}
    if op == "grad":
        if rng.random() < 0.5:
            return {"op": op, "loss": "inner", "L": rng.randint(8, 20), "d": rng.choice([2, 4]), "chiA": _log_int(rng, 8, 60),
                    "chiB": _log_int(rng, 8, 60), "chiW": _log_int(rng, 8, 60)}
        return {"op": op, "loss": "sqdist", "L": rng.randint(6, 10), "d": rng.choice([2, 3, 4]), "chiA": _log_int(rng, 4, 12),
                "chiB": _log_int(rng, 4, 12), "chiW": _log_int(rng, 4, 12)}
    return {"op": op, "M": _log_int(rng, 64, 2000), "N": _log_int(rng, 64, 1000), "K": _log_int(rng, 64, 1500),
            "prec": rng.choice(["fp64", "bf16_split", "bf16_split"])}


# ---------------------------------------------------------------- inputs

def _bonds(L, d, chi):
    return [min(d ** i, d ** (L - i), chi) for i in range(L + 1)]


def _generator(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, dtype=torch.float64, device=_device())


def _random_train(L, d, chi, g):
    """Gaussian cores, made left-canonical; the norm sits in the last core."""
    D = _bonds(L, d, chi)
    out, carry = [], torch.ones(1, 1, dtype=torch.float64, device=_device())
    for k in range(L):
        c = torch.einsum("ij,jsk->isk", carry, _normal(g, D[k], d, D[k + 1]))
        if k == L - 1:
            out.append(c.contiguous())
            break
        q, carry = torch.linalg.qr(c.reshape(c.shape[0] * d, -1))
        out.append(q.reshape(c.shape[0], d, -1).contiguous())
    return out


def _spectral_train(L, d, chi, g):
    """Right-orthonormal random cores with a normalised 1/k profile on every bond, right-canonical, norm 1."""
    D = _bonds(L, d, chi)
    cores = []
    for k in range(L):
        q, _ = torch.linalg.qr(_normal(g, d * D[k + 1], D[k]))
        c = q.T.reshape(D[k], d, D[k + 1])
        if k:
            s = 1.0 / torch.arange(1, D[k] + 1, dtype=torch.float64, device=_device())
            c = (s / s.norm())[:, None, None] * c
        cores.append(c)
    for k in range(L - 1, 0, -1):
        Dl = cores[k].shape[0]
        q, r = torch.linalg.qr(cores[k].reshape(Dl, -1).T)
        cores[k] = q.T.reshape(q.shape[1], d, -1).contiguous()
        cores[k - 1] = torch.einsum("isj,kj->isk", cores[k - 1], r)
    cores[0] = (cores[0] / cores[0].norm()).contiguous()
    return cores


def _field_train(L, d, chi, g):
    """A random-phase field on a periodic grid, digits interleaved (coarsest first), compressed to bond chi."""
    dims, base = {2: (1, 2), 3: (1, 3), 4: (2, 2), 8: (3, 2)}[d]
    n = base ** L
    cut = {1: 0.5 * chi, 2: 0.7 * chi ** 0.5, 3: 0.5 * chi ** (1.0 / 3.0)}[dims]  # a cut-off that the bond resolves
    k1 = torch.fft.fftfreq(n, d=1.0 / n, device=_device(), dtype=torch.float64)
    k = torch.sqrt(sum(x ** 2 for x in torch.meshgrid(*([k1] * dims), indexing="ij")))
    amp = torch.where(k > 0, k.clamp(min=1.0) ** (-5.0 / 6.0 - 0.5 * (dims - 1)), torch.zeros_like(k)) * torch.exp(-k / cut)
    hat = amp * torch.fft.fftn(_normal(g, *([n] * dims)))
    x = torch.fft.ifftn(hat).real
    x = x / x.square().mean().sqrt()
    x = x.reshape([base] * (L * dims)).permute([a * L + i for i in range(L) for a in range(dims)]).reshape(1, -1)
    D, cores = _bonds(L, d, chi), []
    for i in range(L - 1):
        m = x.reshape(D[i] * d, -1)
        _, u = torch.linalg.eigh(m @ m.T)
        u = u[:, u.shape[1] - D[i + 1]:].flip(1)
        cores.append(u.reshape(D[i], d, D[i + 1]).contiguous())
        x = u.T @ m
    cores.append(x.reshape(D[L - 1], d, 1).contiguous())
    return cores


_TRAINS = {"random": _random_train, "spectral": _spectral_train, "field": _field_train}


def _unit(T):
    T[-1] = T[-1] / T[-1].norm()
    return T


def _inputs(case, seed):
    g = _generator(seed)
    op = case["op"]
    if op == "multiply":
        make = _TRAINS[case["kind"]]
        return [make(case["L"], case["d"], case["chiA"], g), make(case["L"], case["d"], case["chiB"], g)]
    if op == "batch":
        # the bonds are the case's, the values the seed's: a program that batches knows its shapes
        return [[_random_train(case["L"], case["d"], c, g) for c in pair] for pair in _batch_bonds(case)]
    if op == "inner":
        return [_unit(_random_train(case["L"], case["d"], c, g)) for c in (case["chiA"], case["chiB"])]
    if op == "grad":
        T = [_unit(_random_train(case["L"], case["d"], c, g)) for c in (case["chiA"], case["chiB"], case["chiW"])]
        if case["loss"] == "sqdist":  # a target of the size of the product, d^(-L/2) for unit trains
            T[2][-1] = T[2][-1] * case["d"] ** (-case["L"] / 2)
        return T
    return [_normal(g, case["M"], case["K"]), _normal(g, case["K"], case["N"])]


def _batch_bonds(case):
    """Uneven bonds spread over [chi_lo, chi_hi]."""
    n, lo, hi = case["n"], case["chi_lo"], case["chi_hi"]
    return [(lo + (hi - lo) * i // max(1, n - 1), lo + (hi - lo) * ((5 * i + 2) % n) // max(1, n - 1)) for i in range(n)]


def prepare(case, seed):
    """Inputs on the GPU and a handle on the current stream, as a program keeps them."""
    return {"case": case, "in": _inputs(case, seed), "handle": ttm.Handle(0)}


# ---------------------------------------------------------------- one pass

def _dense(cores):
    """The tensor of a train, contracted from both ends to the middle."""
    L = len(cores)
    mid = (L + 1) // 2
    left = cores[0].reshape(cores[0].shape[1], -1)
    for c in cores[1:mid]:
        left = (left @ c.reshape(c.shape[0], -1)).reshape(-1, c.shape[2])
    if mid == L:
        return left.reshape(-1)
    right = cores[-1].reshape(cores[-1].shape[0], -1)
    for c in reversed(cores[mid:-1]):
        right = (c.reshape(-1, c.shape[2]) @ right).reshape(c.shape[0], -1)
    return (left @ right).reshape(-1)


def run(state):
    case, x, h = state["case"], state["in"], state["handle"]
    op = case["op"]
    if op == "multiply":
        cores, _ = ttm.ttm_multiply(h, x[0], x[1], eps=case["eps"], chi_max=case["chi_max"], chi_out=case["chi_out"],
                                    prec=case["prec"], use_graph=case["graph"])
        return {"field": _dense(cores)}
    if op == "batch":
        outs, _ = ttm.ttm_multiply_batched(h, x, eps=case["eps"], chi_max=case["chi_max"], chi_out=case["chi_out"],
                                           prec=case["prec"])
        return {"fields": [_dense(c) for c in outs]}
    if op == "inner":
        return {"value": np.float64(ttm.ttm_inner(h, x[0], x[1]))}
    if op == "grad":
        value, gA, gB = ttm.ttm_backward(h, case["loss"], x[0], x[1], x[2])
        return {"value": np.float64(value), "gA": gA, "gB": gB}
    return {"C": ttm.ttm_gemm(h, x[0], x[1], prec=case["prec"])}


# ---------------------------------------------------------------- what a pass cannot do without

def _train_elements(bonds, d):
    return sum(bonds[k] * d * bonds[k + 1] for k in range(len(bonds) - 1))


def _product_flops(a, b, d, cap):
    """Factorisations and contractions of the swap-and-contract sweep with every bond at its bound:
    a QR and the merge of R per gauge move, the two-site tensor and the two factors of its truncated
    SVD per Swap (counted as a Gram matrix and one basis change: 2 m n^2 + 2 m n k), and the joins."""
    L, fl = len(a) - 1, 0.0

    def qr(dl, dr, nxt):
        m, n = d * dl, dr
        k, p = min(m, n), max(m, n)
        return k, 2.0 * p * k * k - 2.0 / 3.0 * k ** 3 + 2.0 * m * k * k - 2.0 / 3.0 * k ** 3 + 2.0 * k * n * d * nxt

    a, b = list(a), list(b)
    for t in (a, b):
        for k in range(L - 1):
            t[k + 1], f = qr(t[k], t[k + 1], t[k + 2])
            fl += f
    left, right = [0] * (L + 2), [0] * (L + 2)
    left[L], right[L] = a[L - 1], b[L - 1]
    fl += 2.0 * d * a[L - 1] * b[L - 1]
    for i in range(L - 1, 0, -1):
        mv = b[i - 1]
        for j in range(i + 1, L + 1):
            right[j], f = qr(left[j], right[j], right[j + 1] if j < L else mv)
            fl += f
            if j < L:
                left[j + 1] = right[j]
        for j in range(L, i, -1):
            m, n = d * left[j], d * mv
            k = min(m, n, cap) if cap else min(m, n)
            fl += 2.0 * m * n * right[j] + 2.0 * m * n * min(m, n) + 2.0 * m * n * k
            left[j], right[j], mv = k, mv, k
        fl += 2.0 * d * a[i - 1] * a[i] * mv
        left[i], right[i] = a[i - 1], mv
    return fl


def _product_work(case, ca, cb):
    L, d = case["L"], case["d"]
    a, b = _bonds(L, d, ca), _bonds(L, d, cb)
    cap = case["chi_out"] or case["chi_max"] or d ** L
    out = [min(x * y, d ** i, d ** (L - i), cap) for i, (x, y) in enumerate(zip(a, b))]
    return {"bytes": 8.0 * (_train_elements(a, d) + _train_elements(b, d) + _train_elements(out, d)),
            "flops": _product_flops(a, b, d, case["chi_max"])}


def work(case):
    op = case["op"]
    if op == "multiply":
        return _product_work(case, case["chiA"], case["chiB"])
    if op == "batch":
        each = [_product_work(case, ca, cb) for ca, cb in _batch_bonds(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    if op == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 8.0 * (M * K + K * N + M * N), "flops": 2.0 * M * N * K}
    L, d = case["L"], case["d"]
    a, b = _bonds(L, d, case["chiA"]), _bonds(L, d, case["chiB"])
    el = _train_elements(a, d) + _train_elements(b, d)
    if op == "inner":
        fl = sum(2.0 * d * (a[k] * b[k] * b[k + 1] + a[k] * a[k + 1] * b[k + 1]) for k in range(L))
        return {"bytes": 8.0 * (el + 1), "flops": fl}
    w = _bonds(L, d, case["chiW"])
    fl = 0.0
    for k in range(L):  # one left and one right environment step, and the adjoint of both cores
        three = (w[k] * a[k] * b[k] * b[k + 1] + w[k] * a[k] * a[k + 1] * b[k + 1] + w[k] * w[k + 1] * a[k + 1] * b[k + 1])
        fl += 2.0 * d * 4 * three
        if case["loss"] == "sqdist":
            fl += 2.0 * d * 4 * (a[k] ** 2 * b[k] ** 2 * b[k + 1] + a[k] ** 2 * b[k] * b[k + 1] ** 2
                                 + a[k] ** 2 * a[k + 1] * b[k + 1] ** 2 + a[k] * a[k + 1] ** 2 * b[k + 1] ** 2)
    return {"bytes": 8.0 * (2 * el + _train_elements(w, d)), "flops": fl}


# ---------------------------------------------------------------- the results in 64 bits

def _overlap(*trains):
    """sum over the grid of the product of the trains, by environments."""
    letters = "abc"[: len(trains)]
    E = torch.ones([1] * len(trains), dtype=torch.float64, device=trains[0][0].device)
    for cores in zip(*trains):
        T = E.unsqueeze(-1).expand(*E.shape, cores[0].shape[1])  # the shared physical index last
        for i, c in enumerate(cores):
            done, rest = letters[:i].upper(), letters[i:]
            T = torch.einsum("%s%ss,%ss%s->%s%ss" % (done, rest, rest[0], rest[0].upper(), done + rest[0].upper(), rest[1:]), T, c)
        E = T.sum(-1)
    return E.reshape(())


def exact(case, seed):
    """run()'s outputs by plain torch in float64. None for truncated random and spectral products:
    their truncation error is of the size of the product, so no closed value stands for them."""
    op = case["op"]
    if op == "batch" or (op == "multiply" and case["kind"] != "field" and (case["chi_max"] or case["chi_out"])):
        return None
    x = _inputs(case, seed)
    if op == "multiply":
        return {"field": _dense(x[0]) * _dense(x[1])}
    if op == "inner":
        return {"value": np.float64(_overlap(x[0], x[1]).item())}
    if op == "grad":
        A, B, W = x
        for c in A + B:
            c.requires_grad_(True)
        if case["loss"] == "inner":
            f = _overlap(W, A, B)
        else:
            f = (_dense(A) * _dense(B) - _dense(W)).square().sum()
        g = torch.autograd.grad(f, A + B)
        return {"value": np.float64(f.item()), "gA": list(g[: len(A)]), "gB": list(g[len(A):])}
    return {"C": x[0] @ x[1]}
