"""Timed cases: the work a program gives this library, through its public entry points.

A case is a dict of plain values.  ``kind`` says which calls one pass makes:

  map       set_conductances + factor + solve: a new conductance map and its batch of input vectors
  solve     solve alone, with both node-voltage fields, on a factorization that is kept
  tiles     Batch.run: the factor and solve of many uneven tiles in one call
  transfer  set_conductances + factor + transfer_matrix + solve_transfer (currents only)
  predict   Surrogate.predict: the learned estimate of the currents of a new map
  grad      Surrogate.grad: loss and gradient of one minibatch of surrogate training

Conductances are log-uniform in [1e-6, 1e-4] S and voltages uniform in [0, v_max], as in the
package's own input generators.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2410_19993_gb300 import xbar

G_LO, G_HI = 1e-6, 1e-4
HIDDEN = 256        # width of the surrogate's hidden layers
LOSS_LAMBDA = 0.1   # weight of the surrogate's error head in its loss
LOSS_EPS = 1e-6


# ------------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest: a 16 x 16 crossbar with 64 input vectors in FP64; launches and latency count
        _map("map16_fp64_b64", 16, 16, 64, "fp64"),
        # an ordinary FP64 map: the 64 x 64 sweep over wire resistances, 1024 vectors a map
        _map("map64_fp64_b1024", 64, 64, 1024, "fp64", rw=2.5),
        # one input vector of an unpartitioned 256 x 256 crossbar in FP64 (the paper's largest)
        _map("map256_fp64_b1", 256, 256, 1, "fp64", rs=5.0, rw=5.0, rsense=5.0),
        # a tall crossbar, more word lines than bit lines: FP64 blocks over the rows
        _map("tall256x32_fp64_b1", 256, 32, 1, "fp64", rs=5.0, rw=5.0, rsense=5.0),
        # exact labels of a 128 x 128 map for the surrogate: mixed precision, 1000 vectors
        _map("map128_mixed_b1000", 128, 128, 1000, "fp32_ir", rw=2.5),
        # the headline workload: 256 x 256, mixed precision, 8192 vectors
        _map("map256_mixed_b8192", 256, 256, 8192, "fp32_ir"),
        # one vector of a 256 x 256 map in mixed precision, with cyclic reduction as few vectors want it
        _map("cr256_mixed_b1", 256, 256, 1, "fp32_ir", algorithm="cr"),
        # node voltages of a ragged crossbar, an odd batch, on a kept mixed-precision factorization
        {"name": "volt100x37_mixed_b77", "kind": "solve", "M": 100, "N": 37, "B": 77, "precision": "fp32_ir",
         "algorithm": "thomas", "rs": 1.0, "rw": 1.0, "rsense": 10.0, "v_max": 0.5},
        # a 784 -> 256 -> 10 network on ragged 128 x 128 tiles, 4096 vectors a tile, in one call
        {"name": "tiles_fc784_mixed", "kind": "tiles", "n0": 784, "n1": 256, "n2": 10, "tile": 128, "B": 4096,
         "precision": "fp32_ir", "rs": 1.0, "rw": 2.5, "rsense": 10.0, "v_max": 0.3},
        # currents only of a large batch: the transfer matrix of a new map and one product
        {"name": "transfer256_mixed_b8192", "kind": "transfer", "M": 256, "N": 256, "B": 8192,
         "precision": "fp32_ir", "algorithm": "thomas", "rs": 1.0, "rw": 1.0, "rsense": 10.0, "v_max": 0.5},
        # the surrogate's estimate for a held-out 128 x 128 map with 1000 vectors
        {"name": "predict128_b1000", "kind": "predict", "M": 128, "N": 128, "B": 1000, "passes": 2,
         "rs": 1.0, "rw": 2.5, "rsense": 10.0, "v_max": 0.5},
        # one minibatch of the surrogate's training: forward and backward
        {"name": "grad128_r4096", "kind": "grad", "M": 128, "N": 128, "rows": 4096},
    ]


def _map(name, M, N, B, precision, rs=1.0, rw=1.0, rsense=10.0, algorithm="thomas", v_max=0.5):
    return {"name": name, "kind": "map", "M": M, "N": N, "B": B, "precision": precision, "algorithm": algorithm,
            "rs": rs, "rw": rw, "rsense": rsense, "v_max": v_max}


def _log(rng: random.Random, lo: int, hi: int) -> int:
    """A whole number spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _circuit(rng: random.Random):
    rw = rng.choice([0.5, 1.0, 2.5, 5.0, 10.0])
    return {"rs": rng.choice([1.0, rw]), "rw": rw, "rsense": rng.choice([10.0, rw])}


def draw(rng: random.Random):
    kind = rng.choice(["fp64", "fp64", "tall", "mixed", "mixed", "mixed", "solve", "tiles", "transfer", "predict",
                       "grad"])
    c = {"v_max": rng.choice([0.3, 0.5])}
    if kind == "fp64":      # FP64 maps from the smallest to 192 x 192, one vector to a thousand
        c.update(kind="map", M=_log(rng, 8, 192), N=_log(rng, 8, 192), B=_log(rng, 1, 1024), precision="fp64",
                 algorithm="thomas", **_circuit(rng))
    elif kind == "tall":    # many word lines, few bit lines
        N = _log(rng, 8, 64)
        c.update(kind="map", M=_log(rng, 2 * N, 1024), N=N, B=_log(rng, 1, 256), precision="fp64",
                 algorithm="thomas", **_circuit(rng))
    elif kind == "mixed":   # mixed-precision maps; cyclic reduction where a map has few vectors
        B = _log(rng, 1, 8192)
        c.update(kind="map", M=_log(rng, 16, 256), N=_log(rng, 16, 256), B=B, precision="fp32_ir",
                 algorithm=rng.choice(["thomas", "cr"]) if B <= 64 else "thomas", **_circuit(rng))
    elif kind == "solve":
        c.update(kind="solve", M=_log(rng, 8, 200), N=_log(rng, 8, 200), B=_log(rng, 1, 256),
                 precision=rng.choice(["fp64", "fp32_ir"]), algorithm="thomas", **_circuit(rng))
    elif kind == "tiles":   # layers mapped onto tiles of other sizes
        c.update(kind="tiles", n0=_log(rng, 64, 784), n1=_log(rng, 32, 256), n2=_log(rng, 8, 32),
                 tile=rng.choice([64, 100, 128]), B=_log(rng, 64, 4096), precision="fp32_ir", **_circuit(rng))
    elif kind == "transfer":
        c.update(kind="transfer", M=_log(rng, 32, 256), N=_log(rng, 32, 256), B=_log(rng, 256, 8192),
                 precision="fp32_ir", algorithm="thomas", **_circuit(rng))
    elif kind == "predict":
        c.update(kind="predict", M=_log(rng, 32, 160), N=_log(rng, 32, 160), B=_log(rng, 16, 2000),
                 passes=rng.choice([1, 2, 3]), **_circuit(rng))
    else:
        c = {"kind": "grad", "M": _log(rng, 32, 160), "N": _log(rng, 32, 160), "rows": _log(rng, 128, 8192)}
    return c


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _gen(seed: int):
    return torch.Generator(device="cuda").manual_seed(seed)


def _uniform(g, shape, lo, hi):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _conductances(g, M, N):
    return torch.exp(_uniform(g, (M, N), math.log(G_LO), math.log(G_HI)))


def _resistances(case):
    return case["rs"], case["rw"], case["rw"], case["rsense"]


def _map_inputs(case, seed):
    g = _gen(seed)
    G = _conductances(g, case["M"], case["N"])
    V = _uniform(g, (case["B"], case["M"]), 0.0, case["v_max"])
    return G, V


def _tile_inputs(case, seed):
    """Layers n0 -> n1 -> n2 with weights N(0, 0.05), each weight a (positive, negative) pair of
    neighbouring columns, cut into tiles of at most tile x tile; every tile has its own voltages."""
    g = _gen(seed)
    out = []
    for a, b in ((case["n0"], case["n1"]), (case["n1"], case["n2"])):
        w = 0.05 * torch.randn((a, b), generator=g, device="cuda", dtype=torch.float64)
        top = w.abs().max()
        pair = torch.stack([w.clamp(min=0.0), (-w).clamp(min=0.0)], dim=2).reshape(a, 2 * b)
        layer = G_LO + (G_HI - G_LO) * pair / top
        t = case["tile"]
        for r in range(0, a, t):
            for c in range(0, 2 * b, t):
                G = layer[r:r + t, c:c + t].contiguous()
                out.append((G, _uniform(g, (case["B"], G.shape[0]), 0.0, case["v_max"])))
    return out


def _padded_features(M):
    return (3 * M + 127) // 128 * 128


def _network(M, seed):
    """He-scaled network parameters in the surrogate's flat order (FP32)."""
    rng = np.random.default_rng([seed, 1])
    F, Fp = 3 * M, _padded_features(M)
    W1 = np.zeros((HIDDEN, Fp))
    W1[:, :F] = rng.normal(0.0, math.sqrt(2.0 / F), (HIDDEN, F))
    parts = [W1.ravel(), rng.normal(0.0, 0.05, HIDDEN),
             rng.normal(0.0, math.sqrt(2.0 / HIDDEN), HIDDEN * HIDDEN), rng.normal(0.0, 0.05, HIDDEN),
             rng.normal(0.0, math.sqrt(1.0 / HIDDEN), 2 * HIDDEN), rng.normal(0.0, 0.1, 2)]
    return np.concatenate(parts).astype(np.float32)


def _minibatch(case, seed):
    """Feature rows as the training set has them (conductances, voltages and remaining row sums, all
    scaled to about one) and standardised targets."""
    rng = np.random.default_rng([seed, 2])
    R, M = case["rows"], case["M"]
    X = np.empty((R, 3 * M), dtype=np.float32)
    X[:, :M] = np.exp(rng.uniform(math.log(G_LO / G_HI), 0.0, (R, M)))
    X[:, M:2 * M] = rng.uniform(0.0, 1.0, (R, M))
    X[:, 2 * M:] = 0.215 * rng.uniform(0.0, 1.0, (R, 1)) * rng.uniform(0.8, 1.2, (R, M))
    y = rng.normal(0.0, 1.0, R).astype(np.float32)
    return X, y


# ------------------------------------------------------------------------------------------------
# prepare and run
# ------------------------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("map", "solve", "transfer"):
        G, V = _map_inputs(case, seed)
        I = torch.zeros((case["B"], case["N"]), dtype=torch.float64, device="cuda")
        # the handle a program keeps while it goes from map to map
        h = xbar.Crossbar.assemble(G, *_resistances(case))
        if case["algorithm"] == "cr":
            h.set_option("algorithm", "cr")
        s = {"kind": kind, "h": h, "G": G, "V": V, "I": I, "precision": case["precision"]}
        if kind == "solve":
            h.factor(case["precision"])
            s["vWL"] = torch.zeros((case["B"], case["M"], case["N"]), dtype=torch.float64, device="cuda")
            s["vBL"] = torch.zeros_like(s["vWL"])
        return s
    if kind == "tiles":
        tiles = _tile_inputs(case, seed)
        b = xbar.Batch([(G, *_resistances(case)) for G, _ in tiles])
        Is = [torch.zeros((V.shape[0], G.shape[1]), dtype=torch.float64, device="cuda") for G, V in tiles]
        return {"kind": kind, "b": b, "Vs": [V for _, V in tiles], "Is": Is, "precision": case["precision"]}
    if kind == "predict":
        G, V = _map_inputs(case, seed)
        s = xbar.Surrogate(case["M"], case["N"], _resistances(case), passes=case["passes"], g_scale=G_HI,
                           v_scale=case["v_max"], seed=0)
        s.set_params(_network(case["M"], seed))
        s.scaling(mu=0.0, sigma=0.01, c=2.0)
        I = torch.zeros((case["B"], case["N"]), dtype=torch.float64, device="cuda")
        return {"kind": kind, "s": s, "G": G, "V": V, "I": I, "err": torch.zeros_like(I)}
    X, y = _minibatch(case, seed)
    s = xbar.Surrogate(case["M"], case["N"], (1.0, 2.5, 2.5, 10.0), passes=2, g_scale=G_HI, v_scale=0.5, seed=0)
    s.set_params(_network(case["M"], seed))
    return {"kind": kind, "s": s, "X": X, "y": y}


def run(state):
    kind = state["kind"]
    if kind == "map":
        h = state["h"]
        h.set_conductances(state["G"])
        h.factor(state["precision"])
        h.solve(state["V"], state["I"], tol=1e-8, max_iter=10)
        return {"I": state["I"]}
    if kind == "solve":
        state["h"].solve(state["V"], state["I"], vWL=state["vWL"], vBL=state["vBL"], tol=1e-8, max_iter=10)
        return {"I": state["I"], "vWL": state["vWL"], "vBL": state["vBL"]}
    if kind == "tiles":
        state["b"].run(state["precision"], state["Vs"], state["Is"], tol=1e-8, max_iter=6)
        return {"I": state["Is"]}
    if kind == "transfer":
        h = state["h"]
        h.set_conductances(state["G"])
        h.factor(state["precision"])
        h.transfer_matrix(tol=1e-9, max_iter=10)
        h.solve_transfer(state["V"], state["I"])
        return {"I": state["I"]}
    if kind == "predict":
        state["s"].predict(state["G"], state["V"], state["I"], err_est=state["err"])
        return {"I": state["I"], "err": state["err"]}
    loss, grad = state["s"].grad(state["X"], state["y"])
    return {"loss": loss, "grad": grad}


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------------
def _nodal_flops(M, N, B):
    """One direct decomposition of the nodal system in its smaller blocks and B substitutions."""
    k, n = min(M, N), max(M, N)
    return 2.0 * n * k ** 3 + 4.0 * n * k * k * B


def work(case):
    kind = case["kind"]
    if kind in ("map", "solve"):
        M, N, B = case["M"], case["N"], case["B"]
        if kind == "map":
            return {"bytes": 8.0 * (M * N + B * (M + N)), "flops": _nodal_flops(M, N, B)}
        k, n = min(M, N), max(M, N)
        return {"bytes": 8.0 * (n * k * k + B * (M + N + 2 * M * N)), "flops": 4.0 * n * k * k * B}
    if kind == "tiles":
        by = fl = 0.0
        for a, b in ((case["n0"], 2 * case["n1"]), (case["n1"], 2 * case["n2"])):
            t = case["tile"]
            for r in range(0, a, t):
                for c in range(0, b, t):
                    M, N = min(t, a - r), min(t, b - c)
                    by += 8.0 * (M * N + case["B"] * (M + N))
                    fl += _nodal_flops(M, N, case["B"])
        return {"bytes": by, "flops": fl}
    if kind == "transfer":
        M, N, B = case["M"], case["N"], case["B"]
        return {"bytes": 8.0 * (M * N + B * (M + N)), "flops": _nodal_flops(M, N, min(M, N)) + 2.0 * M * N * B}
    if kind == "predict":
        M, N, B = case["M"], case["N"], case["B"]
        mlp = 2.0 * HIDDEN * (2 * M * N + M * B) + 2.0 * B * N * (HIDDEN * HIDDEN + 2 * HIDDEN)
        line = 8.0 * case["passes"] * M * M * N
        return {"bytes": 8.0 * (M * N + B * (M + 2 * N)) + 2.0 * HIDDEN * (3 * M + HIDDEN),
                "flops": mlp + line + 4.0 * B * M * N}
    R, M = case["rows"], case["M"]
    n_par = HIDDEN * (_padded_features(M) + HIDDEN + 4) + 2
    return {"bytes": 4.0 * (R * (3 * M + 1) + n_par) + 2.0 * n_par,
            "flops": 2.0 * R * HIDDEN * (2 * 3 * M + 3 * HIDDEN + 4)}


# ------------------------------------------------------------------------------------------------
# the same results in plain 64-bit torch
# ------------------------------------------------------------------------------------------------
class _Nodal:
    """Maps of one shape (leading dimension t): direct solves of the nodal equations, block
    elimination over the columns, with residuals of the whole system as sums of branch currents."""

    def __init__(self, G, rs, rw, rb, rsense):
        self.G = G                                             # t x M x N
        t, M, N = G.shape
        self.gs, self.gw, self.gb, self.go = 1.0 / rs, 1.0 / rw, 1.0 / rb, 1.0 / rsense
        self.Gc = G.transpose(1, 2).contiguous()               # t x N x M
        d = self.Gc.clone()
        d[:, :, 1:] += self.gb
        d[:, :, :-1] += self.gb
        d[:, :, -1] += self.go
        T = torch.diag_embed(d)
        if M > 1:
            i = torch.arange(M - 1, device=G.device)
            T[:, :, i, i + 1] = -self.gb
            T[:, :, i + 1, i] = -self.gb
        self.Tinv = torch.linalg.inv(T)                        # t x N x M x M
        dW = self.Gc.clone()
        dW[:, 0] += self.gs
        dW[:, 1:] += self.gw
        dW[:, :-1] += self.gw
        self.X = []
        Z = None
        for j in range(N):
            g = self.Gc[:, j]
            C = torch.diag_embed(dW[:, j]) - g[:, :, None] * self.Tinv[:, j] * g[:, None, :]
            Z = C if j == 0 else C - self.gw ** 2 * self.X[-1]
            self.X.append(torch.linalg.inv(Z))

    def direct(self, rw, ru):
        """w, u (t x N x M x k) of right-hand sides on the word-line and bit-line nodes."""
        N = self.Gc.shape[1]
        g = self.Gc[..., None]
        y = rw + g * (self.Tinv @ ru) if ru is not None else rw.clone()
        for j in range(1, N):
            y[:, j] += self.gw * (self.X[j - 1] @ y[:, j - 1])
        w = torch.empty_like(y)
        for j in range(N - 1, -1, -1):
            w[:, j] = self.X[j] @ (y[:, j] + self.gw * w[:, j + 1] if j + 1 < N else y[:, j])
        u = self.Tinv @ (g * w + ru if ru is not None else g * w)
        return w, u

    def solve(self, V):
        """V: t x k x M -> (w, u), each t x N x M x k, refined twice."""
        t, k, M = V.shape
        N = self.Gc.shape[1]
        src = V.transpose(1, 2)                                # t x M x k
        rw = torch.zeros((t, N, M, k), dtype=torch.float64, device=V.device)
        rw[:, 0] = self.gs * src
        w, u = self.direct(rw, None)
        for _ in range(2):
            br = self.Gc[..., None] * (u - w)
            rw = br.clone()
            rw[:, 0] += self.gs * (src - w[:, 0])
            dw = self.gw * (w[:, 1:] - w[:, :-1])
            rw[:, :-1] += dw
            rw[:, 1:] -= dw
            ru = -br
            du = self.gb * (u[:, :, 1:] - u[:, :, :-1])
            ru[:, :, :-1] += du
            ru[:, :, 1:] -= du
            ru[:, :, -1] -= self.go * u[:, :, -1]
            cw, cu = self.direct(rw, ru)
            w = w + cw
            u = u + cu
        return w, u

    def currents(self, V):
        """t x k x N bit-line currents, through the transfer matrix where that is smaller."""
        t, k, M = V.shape
        if k <= M:
            return self.go * self.solve(V)[1][:, :, -1].transpose(1, 2)
        eye = torch.eye(M, dtype=torch.float64, device=V.device).expand(t, M, M)
        return V @ (self.go * self.solve(eye)[1][:, :, -1].transpose(1, 2))


def _exact_tiles(case, seed):
    tiles = _tile_inputs(case, seed)
    out = [None] * len(tiles)
    shapes = {}
    for n, (G, _) in enumerate(tiles):
        shapes.setdefault(tuple(G.shape), []).append(n)
    for idx in shapes.values():
        sys_ = _Nodal(torch.stack([tiles[n][0] for n in idx]), *_resistances(case))
        I = sys_.currents(torch.stack([tiles[n][1] for n in idx]))
        for k, n in enumerate(idx):
            out[n] = I[k].contiguous()
    return out


def _unpack(P, M):
    P = torch.from_numpy(P).cuda().double()
    Fp = _padded_features(M)
    sizes = [HIDDEN * Fp, HIDDEN, HIDDEN * HIDDEN, HIDDEN, 2 * HIDDEN, 2]
    W1, b1, W2, b2, W3, b3 = torch.split(P, sizes)
    return W1.view(HIDDEN, Fp), b1, W2.view(HIDDEN, HIDDEN), b2, W3.view(2, HIDDEN), b3


def _chain_inverse(G, end, link, first):
    """Dense inverses of single lines: rows of G (lines x nodes) as device conductances to a fixed
    node, `link` between neighbours, `end` to ground at the first or the last node."""
    L, n = G.shape
    d = G.clone()
    d[:, 1:] += link
    d[:, :-1] += link
    d[:, 0 if first else -1] += end
    A = torch.diag_embed(d)
    if n > 1:
        i = torch.arange(n - 1, device=G.device)
        A[:, i, i + 1] = -link
        A[:, i + 1, i] = -link
    return torch.linalg.inv(A)


def _line_transfer(G, rs, rw, rb, rsense, passes):
    """The line model's transfer matrix: lines solved alone in turn, `passes` times."""
    M, N = G.shape
    gs, gw, gb, go = 1.0 / rs, 1.0 / rw, 1.0 / rb, 1.0 / rsense
    Wi = _chain_inverse(G, gs, gw, True)                       # M x N x N
    Bi = _chain_inverse(G.T.contiguous(), go, gb, False)       # N x M x M
    u = torch.zeros((M, M, N), dtype=torch.float64, device=G.device)  # unit input k, row i, column j
    k = torch.arange(M, device=G.device)
    for _ in range(passes):
        r = G * u
        r[k, k, 0] += gs
        w = torch.einsum("iab,kib->kia", Wi, r)
        u = torch.einsum("jab,kbj->kaj", Bi, G * w)
    return go * u[:, M - 1]


def _exact_predict(case, seed):
    G, V = _map_inputs(case, seed)
    M, N = G.shape
    W1, b1, W2, b2, W3, b3 = _unpack(_network(M, seed), M)
    S = torch.flip(torch.cumsum(torch.flip(G, [1]), 1), [1])
    per_col = (G.T / G_HI) @ W1[:, :M].T + (S.T / (N * G_HI)) @ W1[:, 2 * M:3 * M].T
    per_vec = (V / case["v_max"]) @ W1[:, M:2 * M].T + b1
    ideal, line = V @ G, V @ _line_transfer(G, *_resistances(case), case["passes"])
    n = torch.empty((V.shape[0], N, 2), dtype=torch.float64, device="cuda")
    for a in range(0, V.shape[0], 64):
        h1 = torch.relu(per_vec[a:a + 64, None] + per_col[None])
        n[a:a + 64] = torch.relu(h1 @ W2.T + b2) @ W3.T + b3
    I = line + ideal * (0.01 * n[..., 0])
    return {"I": I, "err": 2.0 * 0.01 * torch.exp(n[..., 1]) * ideal.abs() / I.abs()}


def _exact_grad(case, seed):
    M = case["M"]
    X, y = _minibatch(case, seed)
    par = [p.clone().requires_grad_(True) for p in _unpack(_network(M, seed), M)]
    W1, b1, W2, b2, W3, b3 = par
    X = torch.from_numpy(X).cuda().double()
    y = torch.from_numpy(y).cuda().double()
    n = torch.relu(torch.relu(X @ W1[:, :3 * M].T + b1) @ W2.T + b2) @ W3.T + b3
    e = n[:, 0] - y
    l0 = (e ** 2).mean()
    l1 = ((n[:, 1] - torch.log(e.detach().abs() + LOSS_EPS)) ** 2).mean()
    (l0 + LOSS_LAMBDA * l1).backward()
    return {"loss": torch.stack([l0, l1]).detach(), "grad": torch.cat([p.grad.reshape(-1) for p in par])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "tiles":
        return {"I": _exact_tiles(case, seed)}
    if kind == "predict":
        return _exact_predict(case, seed)
    if kind == "grad":
        return _exact_grad(case, seed)
    G, V = _map_inputs(case, seed)
    nodal = _Nodal(G[None], *_resistances(case))
    if kind == "solve":
        w, u = nodal.solve(V[None])
        return {"I": nodal.go * u[0, :, -1].T.contiguous(), "vWL": w[0].permute(2, 1, 0).contiguous(),
                "vBL": u[0].permute(2, 1, 0).contiguous()}
    return {"I": nodal.currents(V[None])[0].contiguous()}
