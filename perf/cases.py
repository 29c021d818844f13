"""The work a program has this library do, as cases that can be timed and checked.

Every case goes through the package's public calls.  The kinds:

  gram     C = alpha op(A)^T B + beta C    tsmttsm: inner products of two block vectors
  apply    B = alpha A C + beta B          tsmm: a block vector times a small matrix
  project  C = A^H B, B -= A C             gs_step: one block Gram-Schmidt projection
  split    gram on the tensor cores        split.tsmttsm_split, 4 to 6 slices
  batch    many uneven products at once    batched.Batch (plan made once, run per pass)
  model    the cost model's network        mlp.Mlp: forward, or loss and gradient

Sizes: widths 1..64, 10^3 to 2^24 rows, real and complex, rows with and
without padding.
"""

import math

import numpy as np
import torch

import paper_1905_03136_gb300 as tsm
from paper_1905_03136_gb300 import batched, mlp, split

DEV = "cuda"
# A drawn case stays below the largest listed ones: multiply-adds count as 2
# (real) or 8 (complex) operations per entry and row.
FLOPS_MAX = 6.8e10
SPLIT_FLOPS_MAX = 1.3e11
BYTES_MAX = 8.5e9


def listed():
    return [
        # the smallest call: a few short vectors, as in a block solver on a coarse grid
        {"name": "gram_r64_4x4_10k", "kind": "gram", "cplx": False, "M": 4, "N": 4, "K": 10000, "op": "T",
         "pad": 0, "alpha": 1.0, "beta": 0.0},
        # a block of eight complex vectors of moderate length (block eigensolver on one GPU's share)
        {"name": "gram_c64_8x8_100k", "kind": "gram", "cplx": True, "M": 8, "N": 8, "K": 100000, "op": "C",
         "pad": 0, "alpha": 1.0, "beta": 0.0},
        # odd widths inside wider arrays, accumulated into an existing small matrix
        {"name": "gram_r64_37x53_ragged", "kind": "gram", "cplx": False, "M": 37, "N": 53, "K": 300007, "op": "T",
         "pad": 3, "alpha": -0.5, "beta": 0.25},
        # the widest product, complex, long: the Gram matrix of a full search space
        {"name": "gram_c64_64x64_2m", "kind": "gram", "cplx": True, "M": 64, "N": 64, "K": 1 << 21, "op": "C",
         "pad": 0, "alpha": 1.0, "beta": 0.0},
        # two long vectors rotated by a 2 x 2 matrix: memory traffic
        {"name": "apply_r64_2x2_16m", "kind": "apply", "cplx": False, "M": 2, "N": 2, "K": 1 << 24, "pad": 0,
         "alpha": 1.0, "beta": 0.0},
        # a subspace update with an odd, non-square coefficient matrix
        {"name": "apply_c64_23x11_update", "kind": "apply", "cplx": True, "M": 23, "N": 11, "K": 200003, "pad": 0,
         "alpha": -1.0, "beta": 1.0},
        # orthogonalisation of a short block: both products, latency counts
        {"name": "project_c64_16x16_10k", "kind": "project", "cplx": True, "M": 16, "N": 16, "K": 10000, "pad": 0},
        # orthogonalisation of long vectors
        {"name": "project_r64_8x8_4m", "kind": "project", "cplx": False, "M": 8, "N": 8, "K": 1 << 22, "pad": 0},
        # the widest product on the tensor cores, default precision
        {"name": "split_c64_64x64_4m", "kind": "split", "cplx": True, "M": 64, "N": 64, "K": 1 << 22, "op": "C",
         "pad": 0, "slices": 6, "dist": "uniform"},
        # a ragged product of medium width with fewer slices
        {"name": "split_r64_24x40_s5", "kind": "split", "cplx": False, "M": 24, "N": 40, "K": 1000003, "op": "T",
         "pad": 1, "slices": 5, "dist": "normal"},
        # a solver step's mixed bag of products, launched as one
        {"name": "batch_32_mixed", "kind": "batch", "count": 32, "lg_lo": 14, "lg_hi": 18, "mix": 7},
        # one training step of the cost model on the shipped timing log's size
        {"name": "model_gradient_6126", "kind": "model", "way": "gradient", "n": 6126, "D": 17, "H": 64},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _rows(rng, cplx, M, N, flops_max):
    c = 2 if cplx else 1
    top = min(1 << 24, flops_max / (2 * M * N * c * c), BYTES_MAX / (8 * c * (M + 2 * N)))
    return _log(rng, 1000, top)


def draw(rng):
    kind = rng.choice(["gram", "gram", "gram", "apply", "apply", "project", "project", "split", "split", "batch",
                       "model"])
    if kind == "batch":
        lo = rng.randint(10, 15)
        return {"kind": kind, "count": rng.randint(4, 64), "lg_lo": lo, "lg_hi": lo + rng.randint(1, 3),
                "mix": rng.randint(0, 1 << 20)}
    if kind == "model":
        return {"kind": kind, "way": rng.choice(["gradient", "gradient", "forward"]), "n": _log(rng, 256, 16384),
                "D": rng.randint(4, 32), "H": rng.randint(8, 64)}
    cplx = rng.random() < 0.5
    M, N = _log(rng, 1, 64), _log(rng, 1, 64)
    if rng.random() < 0.4:
        N = M
    c = {"kind": kind, "cplx": cplx, "M": M, "N": N,
         "K": _rows(rng, cplx, M, N, SPLIT_FLOPS_MAX if kind == "split" else FLOPS_MAX),
         "pad": rng.choice([0, 0, 0, 1, 2, 5])}
    if kind in ("gram", "split"):
        c["op"] = "C" if cplx and rng.random() < 0.75 else "T"
    if kind == "gram":
        c["alpha"], c["beta"] = rng.choice([(1.0, 0.0), (1.0, 0.0), (-1.0, 0.5), (0.75, 0.25)])
    if kind == "apply":
        c["alpha"], c["beta"] = rng.choice([(1.0, 0.0), (1.0, 0.0), (-1.0, 1.0), (0.5, -0.75)])
    if kind == "split":
        c["slices"] = rng.choice([4, 5, 6, 6, 6])
        c["dist"] = rng.choice(["uniform", "normal", "loguniform"])
    return c


# ------------------------------------------------------------------ inputs


def _gen(seed, what):
    return torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + what)


def _block(g, rows, width, pad, cplx, dist="normal"):
    """A row-major rows x width view of a rows x (width + pad) array."""
    shape = (rows, (width + pad) * (2 if cplx else 1))
    if dist == "normal":
        x = torch.randn(shape, generator=g, device=DEV, dtype=torch.float64)
    else:
        x = torch.rand(shape, generator=g, device=DEV, dtype=torch.float64).mul_(2.0).sub_(1.0)
        if dist == "loguniform":  # magnitudes over 2^-20 .. 2^20
            x.mul_(torch.exp2(torch.rand(shape, generator=g, device=DEV, dtype=torch.float64).mul_(40.0).sub_(20.0)))
    if cplx:
        x = torch.view_as_complex(x.view(rows, width + pad, 2))
    return x[:, :width]


def _batch_shapes(case):
    """Kind, type, widths and rows of every product of a batch."""
    rng = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["count"]):
        kind, cplx = int(rng.integers(2)), bool(rng.integers(2))
        M, N = int(rng.integers(1, 65)), int(rng.integers(1, 65))
        K = int(2.0 ** rng.uniform(case["lg_lo"], case["lg_hi"]))
        out.append((kind, cplx, M, N, K))
    return out


def _batch_inputs(case, seed):
    g = _gen(seed, 1)
    out = []
    for kind, cplx, M, N, K in _batch_shapes(case):
        A = _block(g, K, M, 0, cplx)
        if kind == batched.TSMTTSM:
            out.append((kind, A, _block(g, K, N, 0, cplx)))
        else:
            out.append((kind, A, _block(g, M, N, 0, cplx)))
    return out


def _params(case, seed):
    D, H = case["D"], case["H"]
    rng = np.random.default_rng(int(seed))
    sizes = [(H * D, D), (H, D), (H * H, H), (H, H), (H, H), (1, H)]
    return np.concatenate([rng.uniform(-1, 1, n) / math.sqrt(f) for n, f in sizes]).astype(np.float32)


def _samples(case, seed):
    g = _gen(seed, 2)
    X = torch.rand((case["n"], case["D"]), generator=g, device=DEV).mul_(2.0).sub_(1.0)
    return X, torch.randn(case["n"], generator=g, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "batch":
        s["in"] = _batch_inputs(case, seed)
        s["out"], descs = [], []
        for kd, A, B in s["in"]:
            rows = A.shape[1] if kd == batched.TSMTTSM else A.shape[0]
            out = torch.zeros((rows, B.shape[1]), dtype=A.dtype, device=DEV)
            op = None if kd == batched.TSMM else ("C" if A.is_complex() else "T")
            descs.append(batched.desc(kd, A, B, out, op=op))
            s["out"].append(out)
        s["plan"] = batched.Batch(descs)
        return s
    if kind == "model":
        s["net"] = mlp.Mlp(case["D"], case["H"], max_batch=case["n"])
        s["net"].set_params(_params(case, seed))
        s["X"], s["t"] = _samples(case, seed)
        return s
    cplx, M, N, K, pad = case["cplx"], case["M"], case["N"], case["K"], case["pad"]
    dt = torch.complex128 if cplx else torch.float64
    g = _gen(seed, 0)
    dist = case.get("dist", "normal")
    s["A"] = _block(g, K, M, pad, cplx, dist)
    if kind == "project":
        # orthogonal columns; of norm sqrt(2), so that the step reflects B and
        # B keeps its size however often the step is run (of norm 1, a second
        # step on the same B would find nothing but rounding errors in C)
        _orthonormal(s["A"])
        s["A"].mul_(math.sqrt(2.0))
    if kind == "apply":
        s["C"] = _block(g, M, N, 0, cplx)
        s["B"] = _block(g, K, N, pad, cplx)
        return s
    s["B"] = _block(g, K, N, pad, cplx, dist)
    s["C"] = torch.zeros((M, N), dtype=dt, device=DEV)
    if case.get("beta"):
        s["C"] = _block(g, M, N, 0, cplx) * math.sqrt(K)
    return s


def _orthonormal(A):
    """Columns made orthonormal in place (two Cholesky passes)."""
    for _ in range(2):
        G = _gram(A, A, True)
        R = torch.linalg.cholesky(G).mH
        A.copy_(A @ torch.linalg.inv(R))


# --------------------------------------------------------------- one pass


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "gram":
        return tsm.tsmttsm(s["A"], s["B"], s["C"], c["alpha"], c["beta"], op=c["op"])
    if kind == "apply":
        return tsm.tsmm(s["A"], s["C"], s["B"], c["alpha"], c["beta"])
    if kind == "project":
        return [tsm.gs_step(s["A"], s["B"], s["C"]), s["B"]]
    if kind == "split":
        return split.tsmttsm_split(s["A"], s["B"], s["C"], op=c["op"], slices=c["slices"])
    if kind == "batch":
        s["plan"].run()
        return s["out"]
    if c["way"] == "forward":
        return s["net"].forward(s["X"])
    return [s["net"].backward(s["X"], s["t"]), s["net"].grads()]


# ------------------------------------------------------- work and values


def _product_work(kind, cplx, M, N, K, beta):
    c = 2 if cplx else 1
    by = 8 * c * (M * K + N * K + M * N + (N * K if kind == "apply" and beta else 0))
    return by, 2 * M * N * K * c * c


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [_product_work("apply" if kd == batched.TSMM else "gram", cplx, M, N, K, 0.0)
             for kd, cplx, M, N, K in _batch_shapes(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    if kind == "model":
        n, D, H = case["n"], case["D"], case["H"]
        weights = H * D + H * H + H
        if case["way"] == "forward":
            return {"bytes": 4 * (n * (D + 1) + weights), "flops": 2 * n * weights}
        return {"bytes": 4 * (n * (D + 1) + 2 * weights), "flops": 2 * n * (2 * weights + H * H + H)}
    cplx, M, N, K = case["cplx"], case["M"], case["N"], case["K"]
    if kind == "project":  # A and B read, B and C written; both products
        c = 2 if cplx else 1
        return {"bytes": 8 * c * (M * K + 2 * N * K + M * N), "flops": 4 * M * N * K * c * c}
    by, fl = _product_work(kind, cplx, M, N, K, case.get("beta", 0.0))
    return {"bytes": by, "flops": fl}


def _gram(A, B, conj):
    """op(A)^T B in 64 bits: blocks of 512 rows, their products summed pairwise."""
    parts = []
    for k in range(0, A.shape[0], 1 << 18):
        a, b = A[k : k + (1 << 18)], B[k : k + (1 << 18)]
        n = a.shape[0] // 512 * 512
        at = (lambda t: t.mH) if conj else (lambda t: t.mT)
        if n:
            p = torch.matmul(at(a[:n].reshape(-1, 512, a.shape[1])), b[:n].reshape(-1, 512, b.shape[1]))
            parts.append(_pairwise(p))
        if n < a.shape[0]:
            parts.append(at(a[n:]) @ b[n:])
    return _pairwise(torch.stack(parts))


def _pairwise(p):
    while p.shape[0] > 1:
        h = (p.shape[0] + 1) // 2
        q = p[:h].clone()
        q[: p.shape[0] - h] += p[h:]
        p = q
    return p[0]


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for kd, A, B in _batch_inputs(case, seed):
            out.append(_gram(A, B, A.is_complex()) if kd == batched.TSMTTSM else A @ B)
        return out
    if kind == "model":
        D, H, n = case["D"], case["H"], case["n"]
        p = torch.from_numpy(_params(case, seed).astype(np.float64)).to(DEV).requires_grad_(True)
        X, t = (v.double() for v in _samples(case, seed))
        W1, b1, W2, b2, w3, b3 = torch.split(p, [H * D, H, H * H, H, H, 1])
        h = torch.tanh(X @ W1.view(H, D).mT + b1)
        h = torch.tanh(h @ W2.view(H, H).mT + b2)
        y = h @ w3 + b3
        if case["way"] == "forward":
            return y.detach()
        loss = (y - t).square().sum() / n
        loss.backward()
        return [loss.detach().reshape(1), p.grad.detach().cpu().numpy()]
    s = prepare(case, seed)
    if kind in ("gram", "split"):
        G = _gram(s["A"], s["B"], case["op"] == "C")
        if kind == "split":
            return G
        return case["alpha"] * G + (case["beta"] * s["C"] if case["beta"] else 0.0)
    if kind == "apply":
        out = case["alpha"] * (s["A"] @ s["C"])
        return out + case["beta"] * s["B"] if case["beta"] else out
    C = _gram(s["A"], s["B"], True)
    return [C, s["B"] - s["A"] @ C]

