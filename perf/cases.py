"""The workloads that the performance of this library is measured on.

Each case is one pass of a user's program through the public entry points
(``fl.Plan``, ``fl.BatchedPlan``, ``fl.XiPlan``, ``fl.LaplacePlan`` and the
autograd module): the plan is built once per node set, as such programs do, and
a pass executes it.  Node sets and coefficients are those of the repository's
own workloads (``paper_1606_03255_gb300/workloads.py``), drawn on the GPU from
the seed: "disk" (uniform in the unit disk), "circle" (half on |z| = 1, half
with 1 - |z| = 10^(-6U)) and "section5" (x ~ U[0, 1), y ~ U[0, (2q - 1) ln 2], q = 12).

kind: "forward"  f = C c (``Plan.execute``)
      "solve"    f = C c and C^* f, the two products of one step of an iterative
                 least-squares solver on a fixed node set
      "train"    loss sum |f - g|^2 through ``FourierLaplace``, with its backward
      "batched"  B transforms of different sizes in one plan
      "shared"   B coefficient vectors on one node set
      "xi"       real exponents, forward and transposed evaluation
      "laplace"  sum_k c_k kappa(s_j, t_k) (``LaplacePlan``)
"""
import math

import torch

from paper_1606_03255_gb300 import fl, workloads as W
from paper_1606_03255_gb300.autograd import FourierLaplace

TWO_PI = 2.0 * math.pi


def listed():
    return [
        # one small transform at double precision: a latency-bound call
        {"name": "forward 1024 fp64", "kind": "forward", "N": 1024, "M": 1024, "nodes": "disk",
         "precision": "fp64", "eps": 1e-10},
        # a small transform of odd size at single precision, nodes near the circle
        {"name": "forward 3001x2500 fp32", "kind": "forward", "N": 3001, "M": 2500, "nodes": "circle",
         "precision": "fp32", "eps": 1e-6},
        # the benchmark's headline transform
        {"name": "forward 2^20 fp32", "kind": "forward", "N": 1 << 20, "M": 1 << 20, "nodes": "circle",
         "precision": "fp32", "eps": 1e-6},
        # a full-accuracy transform in double arithmetic
        {"name": "forward 2^18 fp64", "kind": "forward", "N": 1 << 18, "M": 1 << 18, "nodes": "circle",
         "precision": "fp64", "eps": 1e-12},
        # a step of an iterative solver, ragged sizes
        {"name": "solve 300007x250001 fp32", "kind": "solve", "N": 300007, "M": 250001,
         "nodes": "circle", "precision": "fp32", "eps": 1e-6},
        # fitting coefficients and nodes by gradients, single precision
        {"name": "train 2^18 fp32", "kind": "train", "N": 1 << 18, "M": 1 << 18, "nodes": "disk",
         "precision": "fp32", "eps": 1e-7},
        # the same at the accuracy of doubles, from float pairs
        {"name": "train 2^18 fp64ff", "kind": "train", "N": 1 << 18, "M": 1 << 18, "nodes": "disk",
         "precision": "fp64ff", "eps": 1e-12},
        # many transforms of log-uniform sizes in one plan
        {"name": "batched 512 fp32", "kind": "batched", "B": 512, "lo": 8.0, "hi": 16.0, "sizes": 0,
         "nodes": "disk", "precision": "fp32", "eps": 1e-6},
        # generalised polynomials: real exponents, both directions
        {"name": "xi 200003x150001 fp32", "kind": "xi", "N": 200003, "M": 150001, "nodes": "circle",
         "precision": "fp32", "eps": 1e-6},
        # the real discrete Laplace transform of the paper's Section 3
        {"name": "laplace 2^16 fp64", "kind": "laplace", "N": 1 << 16, "M": 1 << 16,
         "kernel": "laplace", "precision": "fp64", "eps": 1e-6},
        # a large one in the single-precision form, ragged sizes
        {"name": "laplace 1000003x700001 fp32", "kind": "laplace", "N": 1000003, "M": 700001,
         "kernel": "laplace", "precision": "fp32", "eps": 1e-6},
        # the asymptotically smooth kernel K_1/2 by the generalised algorithm
        {"name": "bessel_half 2^16 fp64", "kind": "laplace", "N": 1 << 16, "M": 1 << 16,
         "kernel": "bessel_half", "precision": "fp64", "eps": 1e-6},
    ]


def _size(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]; a power of two one time in four."""
    v = 2.0 ** rng.uniform(math.log2(lo), math.log2(hi))
    return 1 << round(math.log2(v)) if rng.random() < 0.25 else max(1, round(v))


def draw(rng):
    kind = rng.choice(["forward", "forward", "solve", "train", "batched", "shared", "xi", "laplace"])
    nodes = rng.choice(["disk", "circle", "circle", "section5"])
    if kind == "laplace":
        kernel = rng.choice(["laplace", "laplace", "exp", "bessel_half"])
        hi = 1000000 if kernel == "laplace" else 1 << 16
        return {"kind": kind, "N": _size(rng, 1000, hi), "M": _size(rng, 1000, min(hi, 700000)),
                "kernel": kernel, "precision": rng.choice(["fp32", "fp64"]),
                "eps": rng.choice([1e-4, 1e-6, 1e-8])}
    if kind == "xi":
        return {"kind": kind, "N": _size(rng, 1000, 200000), "M": _size(rng, 1000, 150000),
                "nodes": rng.choice(["disk", "circle"]), "precision": "fp32",
                "eps": rng.choice([1e-4, 1e-5, 1e-6])}
    if kind == "batched":
        hi = rng.uniform(11.0, 15.0)
        return {"kind": kind, "B": rng.randint(8, 256), "lo": 8.0, "hi": hi, "sizes": rng.randint(1, 999),
                "nodes": nodes, "precision": "fp32", "eps": rng.choice([1e-4, 1e-5, 1e-6])}
    if kind == "shared":
        n = _size(rng, 1 << 10, 1 << 16)
        return {"kind": kind, "B": rng.randint(4, 64), "N": n, "M": _size(rng, 1 << 10, 1 << 16),
                "nodes": nodes, "precision": "fp32", "eps": rng.choice([1e-4, 1e-5, 1e-6])}
    precision = rng.choice(["fp32", "fp32", "fp64", "fp64ff"])
    if precision == "fp32":
        eps, hi = rng.choice([1e-4, 1e-5, 1e-6, 1e-7]), 1 << (20 if kind == "forward" else 18)
    else:
        eps = rng.choice([1e-8, 1e-10, 1e-12]) if precision == "fp64" else rng.choice([1e-10, 1e-12])
        hi = 1 << (17 if kind == "forward" else 15)
    return {"kind": kind, "N": _size(rng, 256, hi), "M": _size(rng, 256, hi), "nodes": nodes,
            "precision": precision, "eps": eps}


# ---------------------------------------------------------------------------
# Inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 13)


def _uniform(n, g):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _normal(n, g, dtype):
    return torch.randn(n, generator=g, device="cuda", dtype=dtype)


def _nodes(kind, M, g):
    """(M, 2) float64 (Re w, Im w), the recipes of workloads.py."""
    x = _uniform(M, g)
    if kind == "disk":
        v = -0.5 * torch.log(1.0 - _uniform(M, g)) / TWO_PI
    elif kind == "circle":
        delta = 10.0 ** (-6.0 * _uniform(M, g))
        v = torch.clamp(-torch.log1p(-delta) / TWO_PI, max=40.0)
        on = torch.randperm(M, generator=g, device="cuda")[: M // 2]
        v[on] = 0.0
    else:
        v = _uniform(M, g) * (2 * 12 - 1) * math.log(2.0) / TWO_PI
    return torch.stack([x, v], dim=-1)


def _cdtype(case):
    return torch.complex64 if case["precision"] == "fp32" else torch.complex128


def _rdtype(case):
    return torch.float32 if case["precision"] == "fp32" else torch.float64


def _degrees(case):
    return [int(n) for n in W.batched_degrees(case["B"], seed=case["sizes"], lo=case["lo"], hi=case["hi"])]


def _inputs(case, seed):
    """The tensors of a case, from the seed alone."""
    g, kind = _gen(seed), case["kind"]
    if kind == "laplace":
        # t_k ~ U(0, 1], s_j ~ U(0, 2N] (positive, as K_1/2 wants them)
        return {"t": 1.0 - _uniform(case["N"], g), "s": (1.0 - _uniform(case["M"], g)) * 2.0 * case["N"],
                "c": _normal(case["N"], g, _rdtype(case))}
    if kind == "batched":
        Ns = _degrees(case)
        return {"Ns": Ns, "w": _nodes(case["nodes"], sum(Ns), g), "c": _normal(sum(Ns), g, _cdtype(case))}
    N, M = case["N"], case["M"]
    d = {"w": _nodes(case["nodes"], M, g)}
    d["c"] = _normal(N * (case["B"] if kind == "shared" else 1), g, _cdtype(case))
    if kind == "train":
        d["g"] = _normal(M, g, _cdtype(case))
    if kind == "xi":
        d["w"][:, 0] -= 0.5
        d["xi"] = 1.0 + _uniform(N, g) * (N - 1)
        d["h"] = _normal(M, g, _cdtype(case))
    return d


def prepare(case, seed):
    fl.load()
    kind, d = case["kind"], _inputs(case, seed)
    d["kind"] = kind
    if kind in ("forward", "solve"):
        d["plan"] = fl.Plan(case["N"], d["w"], case["eps"], precision=case["precision"])
    elif kind == "train":
        d["op"] = FourierLaplace(case["N"], eps=case["eps"], precision=case["precision"])
        d["c"].requires_grad_(True)
        d["w"].requires_grad_(True)
        d["op"].plan_for(d["w"])
    elif kind == "batched":
        d["plan"] = fl.BatchedPlan(d["Ns"], d["Ns"], d["w"], case["eps"], precision=case["precision"])
    elif kind == "shared":
        d["plan"] = fl.BatchedPlan([case["N"]] * case["B"], None, d["w"], case["eps"],
                                   precision=case["precision"], shared_nodes=True)
    elif kind == "xi":
        d["plan"] = fl.XiPlan(d["xi"], d["w"], case["eps"], precision=case["precision"])
    else:
        d["plan"] = fl.LaplacePlan(d["t"], d["s"], case["eps"], precision=case["precision"],
                                   kernel=case["kernel"])
    return d


def run(state):
    kind = state["kind"]
    if kind == "solve":
        f = state["plan"].execute(state["c"])
        return {"f": f, "r": state["plan"].adjoint(f)}
    if kind == "train":
        c, w = state["c"], state["w"]
        c.grad = w.grad = None
        f = state["op"](c, w)
        loss = torch.sum(torch.abs(f - state["g"]) ** 2)
        loss.backward()
        return {"f": f.detach(), "c": c.grad, "w": w.grad}
    if kind == "xi":
        return {"f": state["plan"].execute(state["c"]), "g": state["plan"].transposed(state["h"])}
    return {"f": state["plan"].execute(state["c"])}


# ---------------------------------------------------------------------------
# What a pass cannot do without

def work(case):
    """Bytes: coefficients and nodes read once, results written once.  Operations: one
    FFT of N points (5 N log2 N) and one complex multiply-add per coefficient and
    per node for each of the transforms of a pass (Laplace: a multiply-add per
    element and rank, and one per value)."""
    kind = case["kind"]
    cs = 8.0 if case["precision"] == "fp32" else 16.0
    if kind == "laplace":
        rank = math.ceil(0.5 + math.log(1.0 / case["eps"]) / math.log(4.0))
        n = float(case["N"] + case["M"])
        return {"bytes": n * (8.0 + cs / 2), "flops": 2.0 * rank * n}

    def flops(N, M):
        return 5.0 * N * math.log2(max(2, N)) + 8.0 * (N + M)

    if kind == "batched":
        Ns = _degrees(case)
        return {"bytes": sum(Ns) * (2 * cs + 16.0), "flops": sum(flops(n, n) for n in Ns)}
    N, M = float(case["N"]), float(case["M"])
    if kind == "shared":
        B = case["B"]
        return {"bytes": B * (N + M) * cs + 16.0 * M, "flops": B * flops(N, M)}
    if kind == "forward":
        return {"bytes": N * cs + M * (16.0 + cs), "flops": flops(N, M)}
    if kind == "solve":      # c, w in; f, C^* f out
        return {"bytes": 2 * N * cs + M * (16.0 + cs), "flops": 2 * flops(N, M)}
    if kind == "train":      # c, w, g in; f and the two gradients out
        return {"bytes": 2 * N * cs + M * (32.0 + 2 * cs), "flops": 3 * flops(N, M)}
    return {"bytes": 2 * N * cs + 8.0 * N + M * (16.0 + 2 * cs), "flops": 2 * flops(N, M)}


# ---------------------------------------------------------------------------
# The same sums in 64 bits

def _frac_product(k, x):
    """k x mod 1 for |k| < 2^26: x split so that the leading product is exact."""
    hi = torch.round(x * 67108864.0) / 67108864.0
    p = k * hi
    return (p - torch.round(p)) + k * (x - hi)


def _powers(w, k):
    """z_j^k as an (nodes, exponents) complex128 matrix."""
    ph = _frac_product(k[None, :], w[:, :1]) * TWO_PI
    return torch.polar(torch.exp(-TWO_PI * w[:, 1:] * k[None, :]), ph)


def _blocks(N):
    a = max(1, 1 << max(0, (N - 1).bit_length() // 2))      # frequencies k = a i + b, b < a
    return a, -(-N // a)


def _flt(c, w):
    """sum_k c_k z_j^k, by k = a i + b: z^(a i) and z^b as two matrices."""
    N, M = c.numel(), w.shape[0]
    a, n = _blocks(N)
    cc = torch.zeros(n * a, dtype=torch.complex128, device=c.device)
    cc[:N] = c.to(torch.complex128)
    cc = cc.reshape(n, a).T.contiguous()
    lo = torch.arange(a, device=c.device, dtype=torch.float64)
    hi = torch.arange(n, device=c.device, dtype=torch.float64) * a
    step = max(1, min(M, (1 << 24) // max(a, n)))
    return torch.cat([((_powers(w[j:j + step], lo) @ cc) * _powers(w[j:j + step], hi)).sum(1)
                      for j in range(0, M, step)]) if M else cc.new_zeros(0)


def _flt_adjoint(r, w, N):
    """sum_j conj(z_j)^k r_j for k < N."""
    M = w.shape[0]
    a, n = _blocks(N)
    lo = torch.arange(a, device=r.device, dtype=torch.float64)
    hi = torch.arange(n, device=r.device, dtype=torch.float64) * a
    out = torch.zeros(n, a, dtype=torch.complex128, device=r.device)
    step = max(1, min(M, (1 << 24) // max(a, n)))
    for j in range(0, M, step):
        wj, rj = w[j:j + step], r[j:j + step].to(torch.complex128)
        out += (_powers(wj, hi).conj() * rj[:, None]).T @ _powers(wj, lo).conj()
    return out.reshape(-1)[:N].contiguous()


def exact(case, seed):
    kind = case["kind"]
    d = _inputs(case, seed)
    if kind == "laplace":
        N, M = case["N"], case["M"]
        if float(N) * M > 2.0e10:
            return None
        c, out = d["c"].to(torch.float64), []
        step = max(1, (1 << 26) // N)
        for j in range(0, M, step):
            x = d["s"][j:j + step, None] * d["t"][None, :]
            k = torch.exp(-x)
            if case["kernel"] == "bessel_half":
                k = k * torch.sqrt(0.5 * math.pi / x)
            out.append(k @ c)
        return {"f": torch.cat(out)}
    if kind == "batched":
        out, o = [], 0
        for n in d["Ns"]:
            out.append(_flt(d["c"][o:o + n], d["w"][o:o + n]))
            o += n
        return {"f": torch.cat(out)}
    N, w, c = case["N"], d["w"], d["c"].to(torch.complex128)
    if kind == "shared":
        return {"f": torch.cat([_flt(c[b * N:(b + 1) * N], w) for b in range(case["B"])])}
    if kind == "xi":
        if float(N) * case["M"] > 3.5e10:
            return None
        h, g, f = d["h"].to(torch.complex128), torch.zeros_like(c), []
        step = max(1, (1 << 25) // N)
        for j in range(0, case["M"], step):
            P = _powers(w[j:j + step], d["xi"])
            f.append(P @ c)
            g += h[j:j + step] @ P
        return {"f": torch.cat(f), "g": g}
    f = _flt(c, w)
    if kind == "forward":
        return {"f": f}
    if kind == "solve":
        return {"f": f, "r": _flt_adjoint(f, w, N)}
    G = 2.0 * (f - d["g"].to(torch.complex128))
    k = torch.arange(N, device=c.device, dtype=torch.float64)
    gw = G * torch.conj(_flt(c * (TWO_PI * 1j * k), w))
    return {"f": f, "c": _flt_adjoint(G, w, N), "w": torch.view_as_real(gw)}
