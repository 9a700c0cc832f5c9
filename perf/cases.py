"""What a user of this library has it do, as measurable cases.

Each case is one call of a public entry point on inputs that are resident on
the GPU: the forward Gauss sum in its data types (single clouds, one cloud
against itself, few and many channels, batches), the squared MMD, the
gradient step of a particle flow and the vector-Jacobian product of a
training step.  ``listed`` names twelve of them from the smallest to the
largest calls, ``draw`` gives others of the same ranges.
"""
from __future__ import annotations

import math

import torch

import paper_2609_04910_gb300 as gs

_DTYPES = {"fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}


def _case(op, dtype, M, N, D, C=1, B=1, points="normal", values="normal", same=False):
    return {"op": op, "dtype": dtype, "M": M, "N": N, "D": D, "C": C, "B": B, "points": points,
            "values": values, "same": same}


def listed():
    named = {
        # A kernel mean of a minibatch: the smallest calls, one after another
        # inside a training loop, where launches are what a caller waits for.
        "sum_small": _case("sum", "fp16", 1024, 1024, 64),
        # The same latency regime in single precision, at the size of the
        # repository's fp32 workload.
        "sum_fp32": _case("sum", "fp32", 4096, 4096, 16),
        # Kernel regression or density estimation on single-precision features
        # whose width keeps them off the reduced-precision formats.
        "sum_fp32_wide": _case("sum", "fp32", 16384, 16384, 64),
        # The benchmark workload: the witness function of two samples, queries
        # drawn apart from the keys.
        "sum_mmd": _case("sum", "fp16", 65536, 65536, 64, values="signed_halves"),
        # One cloud against itself with arbitrary weights (kernel density or a
        # matrix-vector product of an iterative solver), at sizes that are no
        # multiple of anything.
        "sum_self": _case("sum", "fp16", 50021, 50021, 50, same=True),
        # Many channels at once: smoothing of 64 features over a point cloud.
        "sum_multi": _case("sum", "bf16", 65536, 65536, 128, C=64, points="half_normal"),
        # Wide embeddings with a common offset against a long list of keys: the
        # largest call, keys beyond the L2 cache.
        "sum_offset": _case("sum", "fp16", 16384, 1048576, 256, C=4, points="offset",
                            values="uniform"),
        # Independent clouds of the paper's benchmark in one batched call.
        "batched": _case("batched", "fp16", 4096, 4096, 64, B=64),
        # A squared MMD per element of a batch, as a loss or a two-sample test.
        "mmd2": _case("mmd2", "bf16", 2000, 2000, 32, B=64, values="signed_halves", same=True),
        # One step of a particle flow with a few thousand particles of ragged
        # count and width: many short steps follow one another.
        "grad_small": _case("grad", "fp16", 3001, 3001, 20, points="gmm", values="signed_halves",
                            same=True),
        # One step of a large MMD / SVGD flow: the sum and its gradient.
        "grad_svgd": _case("grad", "fp16", 131072, 131072, 32, points="gmm",
                           values="signed_halves", same=True),
        # The backward pass of a multi-channel sum inside a training step.
        "vjp": _case("vjp", "fp16", 65536, 65536, 64, C=4),
    }
    return [dict(c, name=n) for n, c in named.items()]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    """A point dimension: a usual one, or any."""
    usual = [d for d in (16, 32, 64, 128) if lo <= d <= hi]
    return rng.choice(usual) if usual and rng.random() < 0.5 else _log_int(rng, lo, hi)


def draw(rng):
    kind = rng.choice(["sum", "sum", "sum", "sum_fp32", "sum_fp32", "sum_multi", "sum_offset",
                       "batched", "mmd2", "grad", "grad", "vjp"])
    half = rng.choice(["fp16", "fp16", "bf16"])
    if kind == "sum":
        N = _log_int(rng, 1024, 65536)
        same = rng.random() < 0.4
        M = N if same else _log_int(rng, 1024, 65536)
        return _case("sum", half, M, N, _width(rng, 2, 100), C=rng.choice([1, 1, 1, 2, 3, 4]),
                     values=rng.choice(["normal", "signed_halves"]), same=same)
    if kind == "sum_fp32":
        D = _width(rng, 2, 64)
        top = min(32768, int(math.sqrt(2 ** 34 / D)))
        return _case("sum", "fp32", _log_int(rng, 1024, top), _log_int(rng, 1024, top), D,
                     C=rng.choice([1, 1, 2]))
    if kind == "sum_multi":
        return _case("sum", half, _log_int(rng, 4096, 65536), _log_int(rng, 4096, 65536),
                     _width(rng, 16, 128), C=_log_int(rng, 5, 64), points="half_normal")
    if kind == "sum_offset":
        M = _log_int(rng, 1024, 16384)
        return _case("sum", half, M, _log_int(rng, 65536, 1048576), _log_int(rng, 130, 256),
                     C=rng.randint(1, 4), points="offset", values="uniform")
    if kind in ("batched", "mmd2"):
        B = _log_int(rng, 8, 256)
        N = _log_int(rng, 512, int(math.sqrt(2 ** 30 / B)))
        return _case(kind, half, N, N, _width(rng, 2, 64), B=B, same=kind == "mmd2",
                     values="signed_halves" if kind == "mmd2" else "normal")
    if kind == "grad":
        N = _log_int(rng, 1024, 131072)
        return _case("grad", half, N, N, _width(rng, 2, 64), points="gmm",
                     values="signed_halves", same=True)
    return _case("vjp", half, _log_int(rng, 2048, 65536), _log_int(rng, 2048, 65536),
                 _width(rng, 8, 64), C=rng.randint(1, 4))


def _points(case, rows, gen, shared):
    """Point clouds as the repository's workloads draw them."""
    D, B = case["D"], case["B"]
    x = torch.randn(B * rows, D, generator=gen, device="cuda")
    if case["points"] == "half_normal":
        x *= 0.5
    elif case["points"] == "gmm":
        label = torch.randint(0, 4, (B * rows,), generator=gen, device="cuda")
        x += shared[label]
    elif case["points"] == "offset":
        x = x.mul_(0.1).add_(shared)
    x = x.to(_DTYPES[case["dtype"]])
    return x.view(B, rows, D) if case["op"] in ("batched", "mmd2") else x


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    M, N, D, C, B = (case[n] for n in "MNDCB")
    shared = None
    if case["points"] == "gmm":
        shared = 2.0 * torch.randn(4, D, generator=gen, device="cuda")
    elif case["points"] == "offset":
        shared = torch.randn(D, generator=gen, device="cuda")
        shared *= 50.0 / shared.norm()
    k = _points(case, N, gen, shared)
    q = k if case["same"] else _points(case, M, gen, shared)
    if case["values"] == "signed_halves":
        v = torch.full((N,), 1.0 / N, device="cuda")
        v[N // 2:] = -1.0 / N
        v = v.view(1, N, 1).expand(B, N, C)
    elif case["values"] == "uniform":
        v = 2.0 * torch.rand(B, N, C, generator=gen, device="cuda") - 1.0
    else:
        v = torch.randn(B, N, C, generator=gen, device="cuda")
    v = v.to(_DTYPES[case["dtype"]]).contiguous()
    if case["op"] == "mmd2":
        v = v.view(B, N)
    elif case["op"] != "batched":
        v = v.view(N, C)
    g = None
    if case["op"] == "vjp":
        g = torch.randn(M, C, generator=gen, device="cuda")
    tau = (10.0 if case["points"] == "offset" else 2.0 if case["points"] == "half_normal" else 1.0) / D
    return q, k, v, g, tau


def prepare(case, seed):
    q, k, v, g, tau = _inputs(case, seed)
    return {"op": case["op"], "q": q, "k": k, "v": v, "g": g, "tau": tau}


def run(state):
    q, k, v, tau = state["q"], state["k"], state["v"], state["tau"]
    if state["op"] == "sum":
        return gs.gauss_sum(q, k, v, tau)
    if state["op"] == "batched":
        return gs.gauss_sum_batched(q, k, v, tau)
    if state["op"] == "mmd2":
        return gs.gauss_sum_mmd2(k, v, tau)
    if state["op"] == "grad":
        return gs.gauss_sum_grad_q(q, k, v, tau)
    return gs.gauss_sum_vjp(q, k, v, state["g"], tau)


def work(case):
    """Inputs read once and outputs written once; per pair of points one
    distance (2 D flops; an unordered pair of one cloud has one distance) and
    one exponential, and 2 flops per channel summed over."""
    M, N, D, C, B = (case[n] for n in "MNDCB")
    eb = 4 if case["dtype"] == "fp32" else 2
    points = N * D if case["same"] else (M + N) * D
    distances = N * (N + 1) // 2 if case["same"] else M * N
    bytes_in = (points + N * C) * eb
    flops = distances * (2 * D + 1)
    if case["op"] in ("sum", "batched"):
        bytes_out = 4 * M * C
        flops += 2 * M * N * C
    elif case["op"] == "mmd2":
        bytes_out = 4
        flops += 2 * distances
    elif case["op"] == "grad":
        bytes_out = 4 * M * (D + 1)
        flops += 2 * M * N * (D + 1)
    else:
        bytes_in += 4 * M * C
        bytes_out = 4 * (M * D + N * D + N * C)
        # pair weights g_m . v_n, then the three contractions
        flops += 2 * M * N * (C + 2 * (D + 1) + C)
    return {"bytes": B * (bytes_in + bytes_out), "flops": B * flops}


_PAIRS = 1 << 27     # pairs per block of rows


def _phi(q, k, k2, tau):
    d2 = (q * q).sum(1, keepdim=True) + k2 - 2.0 * (q @ k.T)
    return d2.clamp_(min=0.0).mul_(-0.5 * tau).exp_()


def exact(case, seed):
    M, N, D, C = (case[n] for n in "MNDC")
    q, k, v, g, tau = _inputs(case, seed)
    same = q is k
    q, k, v = (t.double() for t in (q, k, v))
    if case["op"] in ("batched", "mmd2"):
        out = []
        for b in range(case["B"]):
            kb, vb = k[b], v[b].reshape(N, -1)
            mu = kb.mean(0)
            kb = kb - mu
            qb = kb if same else q[b] - mu
            s = _phi(qb, kb, (kb * kb).sum(1), tau) @ vb
            out.append((vb * s).sum() if case["op"] == "mmd2" else s)
        return torch.stack(out)
    mu = k.mean(0)
    k = k - mu
    q = k if same else q - mu
    k2 = (k * k).sum(1)
    rows = max(1, _PAIRS // N)
    if case["op"] == "sum":
        return torch.cat([_phi(q[r:r + rows], k, k2, tau) @ v for r in range(0, M, rows)])
    if case["op"] == "grad":
        grad, s = [], []
        w = torch.cat([k * v, v], dim=1)
        for r in range(0, M, rows):
            qr = q[r:r + rows]
            a = _phi(qr, k, k2, tau) @ w
            grad.append(tau * (a[:, :D] - qr * a[:, D:]))
            s.append(a[:, D])
        return torch.cat(grad), torch.cat(s)
    g = g.double()
    gq = []
    gk, gv = torch.zeros_like(k), torch.zeros_like(v)
    for r in range(0, M, rows):
        qr, gr = q[r:r + rows], g[r:r + rows]
        p = _phi(qr, k, k2, tau)
        gv += p.T @ gr
        p *= gr @ v.T
        gq.append(tau * (p @ k - qr * p.sum(1, keepdim=True)))
        gk += tau * (p.T @ qr - k * p.sum(0)[:, None])
    return torch.cat(gq), gk, gv
