"""The calls whose speed is measured, each through the package's public entry points.

A case is a dict of plain values.  ``prepare`` makes what a program holds before
the call, ``run`` is one call (or one training step), ``work`` counts what no
implementation can do without, and ``exact`` forms the same outputs in 64 bits
with plain torch.  The sizes are those of the test and benchmark configurations,
and generic ones between them.
"""
from __future__ import annotations

import math

import torch

import paper_1511_05690_gb300 as pn

DEV = "cuda"


def listed():
    return [
        # A single small product in the accurate format: the configuration that the
        # tests hold to 1e-5.  Latency and launches.
        {"name": "product f32 256", "kind": "product", "M": 256, "N": 256, "K": 256,
         "compute": "f32", "n_p": 8, "data": "uniform", "estimator": 0, "correction": 0,
         "aux": True},
        # An ordinary product with the default options and odd sizes, whose rows
        # are not 16-byte aligned.
        {"name": "product bf16 ragged", "kind": "product", "M": 1021, "N": 2047, "K": 1531,
         "compute": "bf16", "n_p": 7, "data": "uniform", "estimator": 0, "correction": 0,
         "aux": True},
        # The large product: the benchmark's default configuration.
        {"name": "product bf16 16384", "kind": "product", "M": 16384, "N": 16384, "K": 16384,
         "compute": "bf16", "n_p": 7, "data": "wide", "estimator": 0, "correction": 0,
         "aux": False},
        # The fastest format with the bias removed by an affine fit to 1024 exact entries.
        {"name": "product e4m3 8192 affine", "kind": "product", "M": 8192, "N": 8192,
         "K": 8192, "compute": "e4m3", "n_p": 7, "data": "wide", "estimator": 0,
         "correction": 2, "aux": False},
        # The experiments' estimator (projection onto two values) on a medium product.
        {"name": "product bf16 4096 r=2", "kind": "product", "M": 4096, "N": 4096, "K": 4096,
         "compute": "bf16", "n_p": 7, "data": "wide", "estimator": 2, "correction": 0,
         "aux": False},
        # Many uneven products planned once and run together: square sizes
        # log-uniform in [16, 1024].
        {"name": "grouped bf16 64", "kind": "grouped", "count": 64, "lo": 16, "hi": 1024,
         "compute": "bf16"},
        # Shortest paths of a small graph whose distances spread over several p levels.
        {"name": "apsp 512", "kind": "apsp", "n": 512, "lo": 1.0, "hi": 10.0},
        # Shortest paths of a large graph.
        {"name": "apsp 4096", "kind": "apsp", "n": 4096, "lo": 0.2, "hi": 1.0},
        # One training step: the product and its adjoint, P = {1..64}.
        {"name": "train f32 2048", "kind": "train", "M": 2048, "N": 2048, "K": 2048,
         "compute": "f32", "n_p": 7},
        # A batch of max-convolutions, one problem per row.
        {"name": "maxconv 1024 x 4096", "kind": "maxconv", "batch": 1024, "nx": 4096,
         "ny": 4096},
        # One long max-convolution.
        {"name": "maxconv long 2^21", "kind": "maxconv", "batch": 1, "nx": 1 << 21,
         "ny": 1 << 21},
        # The top 1024 of x_i y_j and their indices, for a batch of vector pairs.
        {"name": "topk 256 x 4096", "kind": "topk", "batch": 256, "n": 4096, "k": 1024},
    ]


def _log(rng, lo, hi):
    """A whole number in [lo, hi], spread over its logarithm: odd ones come as often as even ones."""
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["product"] * 4 + ["grouped", "apsp", "train", "maxconv", "long", "topk"])
    if kind == "product":
        M, N, K = (_log(rng, 128, 8192) for _ in range(3))
        if rng.random() < 0.5:  # half of them with aligned rows
            N, K = (N + 15) // 16 * 16, (K + 15) // 16 * 16
        compute = rng.choice(["f32", "tf32", "bf16", "bf16", "f16", "e4m3"])
        estimator = rng.choice([0, 0, 0, 1, 2])
        correction = rng.choice([0, 0, 1, 2]) if estimator == 0 else 0
        return {"kind": "product", "M": M, "N": N, "K": K, "compute": compute, "n_p": 7,
                "data": "wide" if estimator or compute == "e4m3" else
                rng.choice(["uniform", "wide"]),
                "estimator": estimator, "correction": correction, "aux": rng.random() < 0.5}
    if kind == "grouped":
        return {"kind": "grouped", "count": _log(rng, 6, 64), "lo": _log(rng, 8, 64),
                "hi": _log(rng, 128, 1200), "compute": rng.choice(["bf16", "f32", "e4m3"])}
    if kind == "apsp":
        lo, hi = rng.choice([(1.0, 10.0), (0.2, 1.0)])
        return {"kind": "apsp", "n": _log(rng, 200, 3000), "lo": lo, "hi": hi}
    if kind == "train":
        return {"kind": "train", "M": _log(rng, 200, 3000), "N": _log(rng, 200, 3000),
                "K": _log(rng, 200, 3000), "compute": rng.choice(["f32", "f32", "bf16"]),
                "n_p": 7}
    if kind == "maxconv":
        return {"kind": "maxconv", "batch": _log(rng, 16, 1024), "nx": _log(rng, 64, 4096),
                "ny": _log(rng, 64, 4096)}
    if kind == "long":
        return {"kind": "maxconv", "batch": _log(rng, 1, 3), "nx": _log(rng, 8192, 1 << 21),
                "ny": _log(rng, 8192, 1 << 21)}
    n = _log(rng, 200, 4096)
    return {"kind": "topk", "batch": _log(rng, 8, 256), "n": n, "k": _log(rng, 16, 1024)}


# ---------------------------------------------------------------- inputs ---
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + 1511)
    return g


def _values(shape, data, g):
    """(0, 1]: uniform, or U^(1/4) = exp(-Exponential(4))."""
    x = 1.0 - torch.rand(shape, generator=g, device=DEV)
    return x.sqrt_().sqrt_() if data == "wide" else x


def _pair(case, g):
    return (_values((case["M"], case["K"]), case.get("data", "uniform"), g),
            _values((case["K"], case["N"]), case.get("data", "uniform"), g))


def _sizes(case, seed):
    """Square sizes log-uniform in [lo, hi], a fixed spread of them jittered by the seed."""
    g = torch.Generator().manual_seed(int(seed) * 7919 + 3)
    u = (torch.arange(case["count"], dtype=torch.float64)
         + torch.rand(case["count"], generator=g, dtype=torch.float64)) / case["count"]
    u = u[torch.randperm(case["count"], generator=g)]
    return [int(round(case["lo"] * (case["hi"] / case["lo"]) ** float(v))) for v in u]


def _inputs(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind in ("product", "train"):
        A, B = _pair(case, g)
        if kind == "train":  # and the gradient that comes from the rest of the model
            G = torch.randn((case["M"], case["N"]), generator=g, device=DEV)
            return {"A": A, "B": B, "G": G}
        s = {"A": A, "B": B}
        if case["correction"] == 2:
            for name, size in (("fit_i", "M"), ("fit_j", "N")):
                s[name] = torch.randint(0, case[size], (1024,), generator=g, device=DEV,
                                        dtype=torch.int32)
        return s
    if kind == "grouped":
        sizes = _sizes(case, 0)  # one shape table: the values are the seed's
        return {"As": [_values((n, n), "uniform", g) for n in sizes],
                "Bs": [_values((n, n), "uniform", g) for n in sizes]}
    if kind == "apsp":
        n = case["n"]
        W = torch.rand((n, n), generator=g, device=DEV) * (case["hi"] - case["lo"]) + case["lo"]
        W[torch.rand((n, n), generator=g, device=DEV) >= 0.1] = math.inf
        W.fill_diagonal_(0.0)
        return {"W": W}
    if kind == "maxconv":
        return {"x": _values((case["batch"], case["nx"]), "wide", g),
                "y": _values((case["batch"], case["ny"]), "wide", g)}
    return {"x": torch.rand((case["batch"], case["n"]), generator=g, device=DEV),
            "y": torch.rand((case["batch"], case["n"]), generator=g, device=DEV)}


def prepare(case, seed):
    s = _inputs(case, seed)
    if case["kind"] == "grouped":  # the plan a program makes once
        s["plan"] = pn.GroupedProduct(s["As"], s["Bs"], compute=case["compute"])
    s["case"] = case
    return s


# --------------------------------------------------------------- the call ---
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "product":
        C, psel, ssel = pn.maxprod_pnorm(
            state["A"], state["B"], p_log2=range(case["n_p"]), compute=case["compute"],
            estimator=case["estimator"], correction=case["correction"],
            fit_i=state.get("fit_i"), fit_j=state.get("fit_j"), want_psel=case["aux"],
            want_ssel=case["aux"], check=False)
        return {"C": C, "p_sel": psel, "S_sel": ssel}
    if kind == "grouped":
        return state["plan"].run()
    if kind == "apsp":
        return {"D": pn.apsp_pnorm(state["W"], check=False)}
    if kind == "train":
        opts = dict(p_log2=range(case["n_p"]), compute=case["compute"], check=False)
        C, psel, ssel = pn.maxprod_pnorm(state["A"], state["B"], **opts)
        dA, dB = pn.maxprod_pnorm_backward(state["A"], state["B"], C, ssel, psel, state["G"],
                                           **opts)
        return {"C": C, "p_sel": psel, "S_sel": ssel, "dA": dA, "dB": dB}
    if kind == "maxconv":
        z, psel = pn.maxconv_pnorm(state["x"], state["y"], check=False)
        return {"z": z, "p_sel": psel}
    vals, i, j = pn.topk_xy(state["x"], state["y"], case["k"], check=False)
    return {"vals": vals, "i": i, "j": j}


# ------------------------------------------------------------------- work ---
def work(case):
    """Inputs read once and outputs written once; the ring products at the
    smallest number of p levels the estimator needs (three tensor products
    each in the 3xTF32 format); for convolutions the three real transforms."""
    kind = case["kind"]
    three = 3 if case.get("compute") == "f32" or kind == "apsp" else 1
    if kind in ("product", "train"):
        M, N, K = case["M"], case["N"], case["K"]
        ring = 2.0 * M * N * K * three
        if kind == "train":
            return {"bytes": 8.0 * (M * K + K * N) + 13.0 * M * N, "flops": 3 * ring}
        return {"bytes": 4.0 * (M * K + K * N) + (9.0 if case["aux"] else 4.0) * M * N,
                "flops": ring * (1, 2, 4)[case["estimator"]]}
    if kind == "grouped":
        sizes = _sizes(case, 0)
        return {"bytes": 12.0 * sum(n * n for n in sizes),
                "flops": 2.0 * three * sum(n ** 3 for n in sizes)}
    if kind == "apsp":
        n = case["n"]
        return {"bytes": 8.0 * n * n, "flops": 2.0 * three * n ** 3 * math.ceil(math.log2(n))}
    if kind == "maxconv":
        b, nx, ny = case["batch"], case["nx"], case["ny"]
        N = 2 ** math.ceil(math.log2(nx + ny - 1))
        return {"bytes": b * (4.0 * (nx + ny) + 5.0 * (nx + ny - 1)),
                "flops": b * 3 * 2.5 * N * math.log2(N)}
    b, n, k = case["batch"], case["n"], case["k"]
    N = 2 ** math.ceil(math.log2(2 * n - 1))
    # 13 p-sums of every diagonal from transforms, then k pops of 13 p-sums each
    return {"bytes": b * (8.0 * n + 12.0 * k),
            "flops": b * (13 * 3 * 2.5 * N * math.log2(N) + 2.0 * k * 13)}


# --------------------------------------------------------- 64-bit outputs ---
def _tau(K, compute):
    e = {"f32": -105, "tf32": -116, "bf16": -119, "f16": -19, "e4m3": -11}[compute]
    return max(K, 1) * 2.0 ** e


def _scale(x, dim):
    """2^ceil(log2 max) per row or column, 1 where the maximum is 0."""
    m, e = torch.frexp(x.amax(dim, keepdim=True).double())
    s = torch.ldexp(torch.ones_like(m), e - (m == 0.5).to(e.dtype))
    return torch.where(m > 0, s, torch.ones_like(s))


def _pow2(x, q):
    """x^(2^q)."""
    for _ in range(q):
        x = x * x
    return x


def _levels(As, Bs, n_p, tau):
    """p* (its log2) and S^(p*) of every entry of the scaled operands' product."""
    S = q_sel = None
    for q in range(n_p - 1, -1, -1):
        s = _pow2(As, q) @ _pow2(Bs, q)
        if S is None:
            S, q_sel, open_ = s, torch.full_like(s, q, dtype=torch.int32), s < tau
        else:
            S = torch.where(open_, s, S)
            q_sel = torch.where(open_, q, q_sel)
            open_ = open_ & (s < tau)
        if not bool(open_.any()):
            break
    return S, q_sel


def _root(S, q):
    return S ** torch.exp2(-q.double())


def _exact_product(case, s):
    A, B = s["A"].double(), s["B"].double()
    r, c = _scale(s["A"], 1), _scale(s["B"], 0)
    A /= r
    B /= c
    tau, n_p = _tau(case["K"], case["compute"]), case["n_p"]
    S, q = _levels(A, B, n_p, tau)
    x = _root(S, q)
    if case["correction"] == 1:
        x = x / float(case["K"]) ** torch.exp2(-q.double())
    elif case["correction"] == 2:
        i, j = s["fit_i"].long(), s["fit_j"].long()
        best = torch.cat([(A[u] * B[:, v].t()).amax(1)
                          for u, v in zip(i.split(256), j.split(256))])
        est, cls, y = x[i, j], q[i, j], x.clone()
        for t in range(n_p):
            at = cls == t
            n = int(at.sum())
            if n == 0:
                continue
            e, b = est[at], best[at]
            sxx = (e * e).sum() - e.sum() ** 2 / n
            if n == 1 or float(sxx) <= 1e-12 * float((e * e).sum()):
                a, b0 = b.sum() / e.sum(), torch.zeros((), device=DEV, dtype=torch.float64)
            else:
                a = ((e * b).sum() - e.sum() * b.sum() / n) / sxx
                b0 = (b.sum() - a * e.sum()) / n
            y = torch.where(q == t, a * x + b0, y)
        x = y
    if case["estimator"]:
        top = n_p - 1
        if not bool((q == top).all()) or n_p < 3:
            return {"C": None, "p_sel": None, "S_sel": S if case["aux"] else None}
        half = _pow2(A, top - 1) @ _pow2(B, top - 1)
        if case["estimator"] == 1:
            x = (S / half) ** (2.0 / 2 ** top)
        else:
            s1 = _pow2(A, top - 2) @ _pow2(B, top - 2)
            s2, s4 = half, S
            a, b = _pow2(A, top - 2), _pow2(B, top - 2)
            s3 = (a * a * a) @ (b * b * b)
            g0, g1, g2 = s2 * s4 - s3 * s3, s2 * s3 - s1 * s4, s1 * s3 - s2 * s2
            u = {"f32": 2.0 ** -21, "bf16": 2.0 ** -8, "e4m3": 2.0 ** -4}.get(case["compute"],
                                                                             2.0 ** -11)
            root = (-g1 + torch.sqrt((g1 * g1 - 4 * g0 * g2).clamp(min=0))) / (2 * g2)
            one = s2 / s1
            two = torch.minimum(torch.maximum(root, one), s4 ** 0.25)
            two = torch.where(g2 <= 32 * u * s2 * s2, s4 / s2, two * two)
            x = two ** (2.0 / 2 ** top)
    x *= r
    x *= c
    return {"C": x, "p_sel": None, "S_sel": S if case["aux"] else None}


def _exact_apsp(case, s):
    n = case["n"]
    tau = _tau(n, "f32")
    X = torch.exp(-s["W"].double())
    X.fill_diagonal_(1.0)
    for _ in range(math.ceil(math.log2(n))):
        r, c = _scale(X.float(), 1), _scale(X.float(), 0)
        S, q = _levels(X / r, X / c, 7, tau)
        X = (_root(S, q) * r * c).clamp(max=1.0)
        X.fill_diagonal_(1.0)
    return {"D": -torch.log(X)}


def _exact_train(case, s):
    A, B, G = s["A"].double(), s["B"].double(), s["G"].double()
    r, c = _scale(s["A"], 1), _scale(s["B"], 0)
    A, B = A / r, B / c
    S, q = _levels(A, B, case["n_p"], _tau(case["K"], case["compute"]))
    C = _root(S, q) * r * c
    dA, dB = torch.zeros_like(A), torch.zeros_like(B)
    W = G * C / S
    for t in range(case["n_p"]):
        at = q == t
        if not bool(at.any()):
            continue
        w, a, b = torch.where(at, W, 0.0), _pow2(A, t), _pow2(B, t)
        dA += (w @ b.t()) * (a / A) / r
        dB += (a.t() @ w) * (b / B) / c
    return {"C": C, "p_sel": None, "S_sel": S, "dA": dA, "dB": dB}


def _conv(x, y):
    """Linear convolution of the rows in 64 bits; the first and last sums, whose
    few terms a transform would drown in its rounding, are summed directly."""
    nx, ny = x.shape[1], y.shape[1]
    nz = nx + ny - 1
    N = 2 ** math.ceil(math.log2(nz))
    z = torch.fft.irfft(torch.fft.rfft(x, N) * torch.fft.rfft(y, N), N)[:, :nz]
    m = min(256, nx, ny)
    at = torch.arange(m, device=DEV)
    k = at[:, None] - at[None, :]

    def edge(u, v):  # sum_i u_i v_(m-i) for the first m outputs
        out = [torch.einsum("bi,bmi->bm", a, torch.where(k >= 0, b[:, k.clamp(min=0)], 0.0))
               for a, b in zip(u.split(64), v.split(64))]
        return torch.cat(out)
    z[:, :m] = edge(x[:, :m], y[:, :m])
    z[:, nz - m:] = edge(x.flip(1)[:, :m], y.flip(1)[:, :m]).flip(1)
    return z


def _exact_maxconv(case, s):
    sx, sy = (s[k].double().amax(1, keepdim=True) for k in ("x", "y"))
    x, y = s["x"].double() / sx, s["y"].double() / sy
    S = None
    for q in range(6, -1, -1):
        t = _conv(_pow2(x, q), _pow2(y, q))
        if S is None:
            S, sel, open_ = t, torch.full_like(t, q, dtype=torch.int32), t < 1e-12
        else:
            S = torch.where(open_, t, S)
            sel = torch.where(open_, q, sel)
            open_ = open_ & (t < 1e-12)
        if not bool(open_.any()):
            break
    return {"z": _root(S, sel) * sx * sy, "p_sel": None}


def exact(case, seed):
    kind = case["kind"]
    if kind == "topk":
        # the pops are a sequential approximation: after a near-tie equally
        # valid sequences part, so no 64-bit run gives the values to compare
        return None
    s = _inputs(case, seed)
    if kind == "product":
        return _exact_product(case, s)
    if kind == "apsp":
        return _exact_apsp(case, s)
    if kind == "train":
        return _exact_train(case, s)
    if kind == "maxconv":
        return _exact_maxconv(case, s)
    tau = {n: _tau(n, case["compute"]) for n in {a.shape[0] for a in s["As"]}}
    out = []
    for A, B in zip(s["As"], s["Bs"]):
        r, c = _scale(A, 1), _scale(B, 0)
        S, q = _levels(A.double() / r, B.double() / c, 7, tau[A.shape[0]])
        out.append(_root(S, q) * r * c)
    return out
