"""Performance cases: the products a user of the library runs, through its
Python entry points (paper_2606_20863_gb300), with the plan, workspace and
result buffers that a program keeps between calls.

A case is a dict with a "kind":
  gemm         C = op(A) op(B) with a kept plan and workspace; mode "plain" (FP64
               pieces), "ozaki" (slices on the tensor cores, the default form) or
               "crt" (residues on the tensor cores);
  autograd     MWGemm forward and backward, which plan every product themselves;
  batch        independent products of uneven sizes in one call;
  dot          inner products of the rows of two matrices;
  series       products of truncated power series;
  elementwise  add, mul or div entry by entry.
Inputs are m-doubles on the GPU: leading word U[-1, 1) ("spread" 0) or
+-2^U[-spread, spread), every lower word the one above x 2^-53 U[-1, 1).
"""
import math
import random

import numpy as np
import torch

import paper_2606_20863_gb300 as mw


def listed():
    return [
        # a small dense product on the FP64 pipe: the smallest call of the library
        dict(name="gemm_plain_dd_64", kind="gemm", mode="plain", m=2, M=64, N=64, K=64,
             ta=False, tb=False, spread=0),
        # the same operands through the default form: latency and launches
        dict(name="gemm_ozaki_dd_64", kind="gemm", mode="ozaki", m=2, M=64, N=64, K=64,
             ta=False, tb=False, spread=0),
        # an ordinary quad-double product in the default form
        dict(name="gemm_ozaki_qd_1024", kind="gemm", mode="ozaki", m=4, M=1024, N=1024, K=1024,
             ta=False, tb=False, spread=8),
        # ragged sizes and a transposed operand: a block of a larger factorisation
        dict(name="gemm_crt_qd_ragged", kind="gemm", mode="crt", m=4, M=777, N=1300, K=905,
             ta=True, tb=False, spread=8),
        # large products, magnitudes over 40 binades: the library's headline
        dict(name="gemm_crt_dd_4096", kind="gemm", mode="crt", m=2, M=4096, N=4096, K=4096,
             ta=False, tb=False, spread=20),
        dict(name="gemm_crt_qd_4096", kind="gemm", mode="crt", m=4, M=4096, N=4096, K=4096,
             ta=False, tb=False, spread=20),
        # a training step through the autograd function: forward, dA and dB
        dict(name="autograd_dd", kind="autograd", m=2, M=2048, N=2048, K=1024, spread=0),
        # many small octo-double products of uneven sizes (power series methods)
        dict(name="batch_od", kind="batch", m=8, count=2000, lo=8, hi=128, shapes=3, square=True,
             spread=0),
        # inner products of length 6,144, short and long m-doubles
        dict(name="dot_dd", kind="dot", m=2, count=1024, K=6144, spread=0),
        dict(name="dot_od", kind="dot", m=8, count=1024, K=6144, spread=0),
        # octo-double power series of degree 127
        dict(name="series_od", kind="series", m=8, count=2000, n=128, spread=0),
        # quad-double multiplication entry by entry
        dict(name="elementwise_mul_qd", kind="elementwise", op="mul", m=4, n=1 << 22, spread=20),
    ]


def _log_int(rng, lo, hi):
    """An integer between lo and hi, uniform in its logarithm."""
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["gemm", "gemm", "gemm", "autograd", "batch", "dot", "series", "elementwise"])
    if kind == "gemm":
        mode = rng.choice(["plain", "ozaki", "crt", "crt"])
        m = rng.choice({"plain": [2, 4], "ozaki": [2, 4, 8], "crt": [2, 4]}[mode])
        top = {"plain": 384 // m, "ozaki": 4096 // m, "crt": 3600}[mode]
        return dict(kind=kind, mode=mode, m=m, M=_log_int(rng, 24, top), N=_log_int(rng, 24, top),
                    K=_log_int(rng, 24, top), ta=rng.random() < 0.3, tb=rng.random() < 0.3,
                    spread=rng.choice([0, 8, 20]))
    if kind == "autograd":
        return dict(kind=kind, m=rng.choice([2, 4]), M=_log_int(rng, 32, 1500),
                    N=_log_int(rng, 32, 1500), K=_log_int(rng, 32, 1500), spread=0)
    if kind == "batch":
        m = rng.choice([2, 4, 8])
        return dict(kind=kind, m=m, count=_log_int(rng, 16, 1600), lo=rng.randint(4, 24),
                    hi=rng.randint(40, 128), shapes=rng.randrange(1 << 20),
                    square=rng.random() < 0.5, spread=rng.choice([0, 4]))
    if kind == "dot":
        return dict(kind=kind, m=rng.choice([2, 4, 8, 16]), count=_log_int(rng, 16, 1024),
                    K=_log_int(rng, 64, 6144), spread=rng.choice([0, 8]))
    if kind == "series":
        n = _log_int(rng, 8, 400)
        return dict(kind=kind, m=rng.choice([2, 4, 8]), n=n,
                    count=_log_int(rng, 4, max(5, 200000 // n)), spread=0)
    op, m = rng.choice(["add", "mul", "div"]), rng.choice([2, 4, 8])
    top = 1 << ({2: 22, 4: 21, 8: 18}[m] - (3 if op == "div" else 0))
    return dict(kind=kind, op=op, m=m, n=_log_int(rng, 1000, top), spread=rng.choice([0, 20]))


def _shapes(case):
    """(count, 3) sizes M, N, K of a batch's products, largest first."""
    rng = random.Random(case["shapes"])
    out = []
    for _ in range(case["count"]):
        M = rng.randint(case["lo"], case["hi"])
        out.append((M, M, M) if case["square"] else
                   (M, rng.randint(case["lo"], case["hi"]), rng.randint(case["lo"], case["hi"])))
    return sorted(out, key=lambda s: -s[0] * s[1] * s[2])


def _mdouble(gen, m, shape, spread, device):
    """m planes of random m-doubles of the given shape."""
    def sym():
        return torch.rand(shape, dtype=torch.float64, device=device, generator=gen) * 2 - 1
    X = torch.empty((m,) + tuple(shape), dtype=torch.float64, device=device)
    if spread:
        sign = torch.where(sym() < 0, -1.0, 1.0).to(torch.float64)
        X[0] = torch.exp2(sym() * spread) * sign
    else:
        X[0] = sym()
    for j in range(1, m):
        X[j] = X[j - 1] * sym() * 2.0 ** -53
    return X


def _inputs(case, seed, device):
    gen = torch.Generator(device=device)
    gen.manual_seed(seed)
    kind, m, sp = case["kind"], case["m"], case["spread"]
    if kind == "gemm":
        a = (case["K"], case["M"]) if case["ta"] else (case["M"], case["K"])
        b = (case["N"], case["K"]) if case["tb"] else (case["K"], case["N"])
        return _mdouble(gen, m, a, sp, device), _mdouble(gen, m, b, sp, device)
    if kind == "autograd":
        A = _mdouble(gen, m, (case["M"], case["K"]), sp, device)
        B = _mdouble(gen, m, (case["K"], case["N"]), sp, device)
        G = torch.zeros((m, case["M"], case["N"]), dtype=torch.float64, device=device)
        G[0] = torch.rand(G.shape[1:], dtype=torch.float64, device=device, generator=gen) * 2 - 1
        return A, B, G
    if kind == "batch":
        s = np.array(_shapes(case), dtype=np.int64)
        return (_mdouble(gen, m, (int((s[:, 0] * s[:, 2]).sum()),), sp, device),
                _mdouble(gen, m, (int((s[:, 2] * s[:, 1]).sum()),), sp, device))
    if kind == "elementwise":
        shape = (case["n"],)
    else:
        shape = (case["count"], case["K"] if kind == "dot" else case["n"])
    return _mdouble(gen, m, shape, sp, device), _mdouble(gen, m, shape, sp, device)


def prepare(case, seed):
    dev = torch.device("cuda")
    X = _inputs(case, seed, dev)
    kind, m = case["kind"], case["m"]
    s = dict(case=case, X=X)
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        s["plan"] = mw.plan_for(X[0], X[1], case["mode"], case["ta"], case["tb"])
        s["ws"] = torch.empty(mw.workspace_size(s["plan"], M, N, K), dtype=torch.uint8, device=dev)
        s["C"] = torch.empty((m, M, N), dtype=torch.float64, device=dev)
    elif kind == "autograd":
        X[0].requires_grad_(True)
        X[1].requires_grad_(True)
    elif kind == "batch":
        shapes = np.array(_shapes(case), dtype=np.int64)
        M, N, K = shapes.T
        starts = [np.concatenate([[0], np.cumsum(n)[:-1]]) for n in (M * K, K * N, M * N)]
        C = torch.empty((m, int((M * N).sum())), dtype=torch.float64, device=dev)
        s["batch"] = mw.Batch.packed(X[0], X[1], C, shapes, np.stack(starts, axis=1))
    elif kind == "dot":
        s["plan"] = mw.plan_dot(*X)
        s["C"] = torch.empty((m, case["count"]), dtype=torch.float64, device=dev)
    elif kind == "series":
        s["plan"] = mw.plan_convolve(*X)
        s["C"] = torch.empty((m, case["count"], case["n"]), dtype=torch.float64, device=dev)
    else:
        s["C"] = torch.empty_like(X[0])
    return s


def run(state):
    case, X = state["case"], state["X"]
    kind = case["kind"]
    if kind == "gemm":
        return mw.mw_gemm(X[0], X[1], state["plan"], transA=case["ta"], transB=case["tb"],
                          C=state["C"], ws=state["ws"], check=False)
    if kind == "autograd":
        A, B, G = X
        C = mw.MWGemm.apply(A, B)
        dA, dB = torch.autograd.grad(C, (A, B), G)
        return {"C": C.detach(), "dA": dA, "dB": dB}
    if kind == "batch":
        return state["batch"].run()
    if kind == "dot":
        return mw.mw_dot_batched(X[0], X[1], state["plan"], C=state["C"], check=False)
    if kind == "series":
        return mw.mw_convolve_batched(X[0], X[1], state["plan"], C=state["C"], check=False)
    return mw.mw_elementwise(case["op"], X[0], X[1], C=state["C"])


# operations of one double per m-double operation, as the paper counts them
_TABLE1 = {"add": {2: 20, 4: 89, 8: 269}, "mul": {2: 23, 4: 336, 8: 1742},
           "div": {2: 70, 4: 893, 8: 5126}}


def work(case):
    """Bytes: every input word read and every output word written once.  Flops of
    the sums of products: a product of two m-doubles has 104 m significant bits
    and one multiply-add of residues or digits that bfloat16 holds makes at most
    8 of them, so 13 m multiply-adds a term."""
    kind, m = case["kind"], case["m"]
    if kind in ("gemm", "autograd"):
        M, N, K = case["M"], case["N"], case["K"]
        n = M * K + K * N + M * N
        if kind == "gemm":
            return {"bytes": 8 * m * n, "flops": 2 * 13 * m * M * N * K}
        # reads A, B and dL/dC, writes C, dA and dB; three products
        return {"bytes": 8 * m * 2 * n, "flops": 3 * 2 * 13 * m * M * N * K}
    if kind == "batch":
        b = f = 0
        for M, N, K in _shapes(case):
            b += M * K + K * N + M * N
            f += M * N * K
        return {"bytes": 8 * m * b, "flops": 2 * 13 * m * f}
    if kind == "dot":
        return {"bytes": 8 * m * case["count"] * (2 * case["K"] + 1),
                "flops": 2 * 13 * m * case["count"] * case["K"]}
    if kind == "series":
        n = case["n"]
        return {"bytes": 8 * m * 3 * case["count"] * n,
                "flops": 13 * m * case["count"] * n * (n + 1)}
    return {"bytes": 8 * m * 3 * case["n"], "flops": _TABLE1[case["op"]][m] * case["n"]}


# ---- exact results, in Python's integers ---------------------------------------

_UNIT = 1300   # every word is an integer multiple of 2^-_UNIT


def _integers(X):
    """Entries of the m planes X as exact integers in units of 2^-_UNIT."""
    X = X.detach().cpu().numpy()
    total = np.zeros(X.shape[1:], dtype=object)
    for plane in X:
        mant, e = np.frexp(plane)
        shift = np.where(plane == 0, 0, e.astype(np.int64) - 53 + _UNIT)
        total = total + np.left_shift((mant * 2.0 ** 53).astype(np.int64).astype(object),
                                      shift.astype(object))
    return total


def _words(values, unit, m):
    """m planes of doubles, each the rest of value 2^-unit rounded to nearest."""
    flat = values.reshape(-1)
    out = np.zeros((m, flat.size))
    for i, x in enumerate(flat):
        for j in range(m):
            if x == 0:
                break
            sh = max(abs(x).bit_length() - 64, 0)
            q = abs(x) >> sh
            if sh and abs(x) & ((1 << sh) - 1):
                q |= 1
            w = float(q) if x > 0 else -float(q)
            out[j, i] = math.ldexp(w, sh - unit)
            x -= int(w) << sh
    return torch.from_numpy(out.reshape((m,) + values.shape))


_MOST_TERMS = 6_000_000   # multiplications that Python's integers do in a few seconds
_MOST_WORDS = 400_000     # and words of the result


def exact(case, seed):
    kind, m = case["kind"], case["m"]
    if kind == "gemm":
        terms, outs = case["M"] * case["N"] * case["K"], case["M"] * case["N"]
    elif kind == "autograd":
        terms = 3 * case["M"] * case["N"] * case["K"]
        outs = case["M"] * case["N"] + case["M"] * case["K"] + case["K"] * case["N"]
    elif kind == "batch":
        terms = sum(M * N * K for M, N, K in _shapes(case))
        outs = sum(M * N for M, N, K in _shapes(case))
    elif kind == "dot":
        terms, outs = 4 * case["count"] * case["K"] * m, case["count"]
    elif kind == "series":
        terms, outs = case["count"] * case["n"] ** 2, case["count"] * case["n"]
    else:
        terms = outs = case["n"]
    if terms > _MOST_TERMS or m * outs > _MOST_WORDS:
        return None
    X = _inputs(case, seed, torch.device("cuda"))
    if kind == "batch":
        A, B = _integers(X[0]), _integers(X[1])
        parts, a, b = [], 0, 0
        for M, N, K in _shapes(case):
            P = A[a:a + M * K].reshape(M, K).dot(B[b:b + K * N].reshape(K, N))
            parts.append(P.reshape(-1))
            a, b = a + M * K, b + K * N
        return _words(np.concatenate(parts), 2 * _UNIT, m)
    I = [_integers(x) for x in X]
    if kind == "gemm":
        A = I[0].T if case["ta"] else I[0]
        B = I[1].T if case["tb"] else I[1]
        return _words(A.dot(B), 2 * _UNIT, m)
    if kind == "autograd":
        A, B, G = I
        return {"C": _words(A.dot(B), 2 * _UNIT, m), "dA": _words(G.dot(B.T), 2 * _UNIT, m),
                "dB": _words(A.T.dot(G), 2 * _UNIT, m)}
    if kind == "dot":
        return _words((I[0] * I[1]).sum(axis=1), 2 * _UNIT, m)
    if kind == "series":
        n = case["n"]
        C = np.zeros((case["count"], n), dtype=object)
        for k in range(n):
            C[:, k:] = C[:, k:] + I[0][:, k:k + 1] * I[1][:, :n - k]
        return _words(C, 2 * _UNIT, m)
    if case["op"] == "add":
        return _words(I[0] + I[1], _UNIT, m)
    if case["op"] == "mul":
        return _words(I[0] * I[1], 2 * _UNIT, m)
    Q = np.array([(abs(a) << _UNIT) // abs(b) * (1 if (a < 0) == (b < 0) else -1)
                  for a, b in zip(I[0], I[1])], dtype=object)
    return _words(Q, _UNIT, m)
