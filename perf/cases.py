"""Timed calls of libmpjacobi: what its users have it do, through mpj's entry points.

A case is a dict of plain values; ``family`` says which call it is:

solve      one symmetric eigenproblem, mixed method with the default options
           (``mpj.syev``, or ``mpj.syev_ex`` on a kept workspace)
two_pass   the same with ``precond_passes = 2``
plain      the plain FP64 Jacobi from the identity (``method = "plain"``)
cyclic     the mixed method with the paper's cyclic-by-row FP64 sweeps
eigh       differentiable solve and its gradient (``mpj.eigh`` + autograd)
backward   the eigen-adjoint of a batch of equal sizes (``mpj.syev_backward``)
batched    many small matrices of uneven sizes (``mpj.BatchedSolver``)
product    FP64-accurate matrix product on the tensor cores (``mpj.dgemm_tc``)

Spectra are separated enough that every eigenvector is determined to far
better than single precision.  An eigenvector's sign is not determined by the
problem, so the calls that return vectors fix it as a program that stores or
compares them does: the components of each vector sum to a non-negative value.
"""
import math

import torch

from paper_2509_00495_gb300 import mpj

_F64 = torch.float64


def listed():
    return [
        # one small matrix, the paper's lower range: latency of a whole call
        {"name": "solve_96", "family": "solve", "n": 96, "spectrum": "geo", "kappa": 1e3, "workspace": False},
        # an odd size just above a multiple of every tile, random dense matrix
        {"name": "solve_257", "family": "solve", "n": 257, "spectrum": "goe", "kappa": 0.0, "workspace": False},
        # ordinary size, eigenvalues spread evenly over [-1, 1]
        {"name": "solve_1024", "family": "solve", "n": 1024, "spectrum": "linear", "kappa": 0.0, "workspace": False},
        # the large single matrix, solved repeatedly on a kept workspace
        {"name": "solve_4096", "family": "solve", "n": 4096, "spectrum": "geo", "kappa": 1e2, "workspace": True},
        # second preconditioning pass, the faster option for large matrices
        {"name": "two_pass_2048", "family": "two_pass", "n": 2048, "spectrum": "geo", "kappa": 1e2, "workspace": True},
        # the plain method on the paper's random dense matrix, ragged size
        {"name": "plain_1500", "family": "plain", "n": 1500, "spectrum": "goe", "kappa": 0.0, "workspace": False},
        # the paper's own ordering at one of its timed sizes (kappa = 500)
        {"name": "cyclic_300", "family": "cyclic", "n": 300, "spectrum": "geo", "kappa": 5e2, "workspace": False},
        # forward and backward of one matrix inside a differentiable program
        {"name": "eigh_512", "family": "eigh", "n": 512, "gap": 1e-3},
        # the adjoint of a batch, the differentiation workload
        {"name": "backward_64x512", "family": "backward", "batch": 64, "n": 512, "gap": 1e-3},
        # the batched workload: sizes uniform in [8, 256]
        {"name": "batched_2048", "family": "batched", "count": 2048, "lo": 8, "hi": 256},
        # a small batch of small matrices
        {"name": "batched_200_small", "family": "batched", "count": 200, "lo": 8, "hi": 48},
        # one rectangular ragged product, first operand transposed
        {"name": "product_3000", "family": "product", "m": 3000, "n": 1777, "k": 2050, "ta": "T", "tb": "N"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["solve", "solve", "solve", "two_pass", "plain", "cyclic", "eigh", "backward", "batched",
                         "batched", "product"])
    if family in ("solve", "two_pass", "plain", "cyclic"):
        lo, hi = {"solve": (17, 4096), "two_pass": (64, 2048), "plain": (48, 1500), "cyclic": (33, 400)}[family]
        n = _log_int(rng, lo, hi)
        spectrum = rng.choice(["geo", "linear", "goe"])
        # condition numbers of the paper's tests, smaller ones for larger n so
        # that the closest eigenvalues stay about 1e-5 apart
        kappa = rng.choice([1e2, 5e2, 1e3] if n <= 512 else [1e2]) if spectrum == "geo" else 0.0
        return {"family": family, "n": n, "spectrum": spectrum, "kappa": kappa, "workspace": rng.random() < 0.5}
    if family == "eigh":
        return {"family": family, "n": _log_int(rng, 32, 700), "gap": 1e-3}
    if family == "backward":
        return {"family": family, "batch": rng.randint(1, 64), "n": _log_int(rng, 48, 512), "gap": 1e-3}
    if family == "batched":
        return {"family": family, "count": _log_int(rng, 32, 2048), "lo": 8, "hi": rng.randint(24, 256)}
    return {"family": family, "m": _log_int(rng, 100, 4096), "n": _log_int(rng, 100, 4096),
            "k": _log_int(rng, 100, 4096), "ta": rng.choice("NT"), "tb": rng.choice("NT")}


# ------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _haar(n, g, batch=None):
    shape = (n, n) if batch is None else (batch, n, n)
    q, r = torch.linalg.qr(torch.randn(shape, dtype=_F64, device="cuda", generator=g))
    d = torch.diagonal(r, dim1=-2, dim2=-1)
    return q * torch.where(d < 0, -1.0, 1.0).unsqueeze(-2)


def _symmetric(a):
    return (a + a.transpose(-2, -1)) / 2


def _matrix(case, seed):
    n, g = case["n"], _generator(seed)
    if case["spectrum"] == "goe":
        return _symmetric(torch.randn(n, n, dtype=_F64, device="cuda", generator=g))
    q = _haar(n, g)
    if case["spectrum"] == "linear":
        lam = torch.linspace(-1.0, 1.0, n, dtype=_F64, device="cuda")
    else:
        e = torch.linspace(-math.log(case["kappa"]), 0.0, n, dtype=_F64, device="cuda")
        sign = torch.where(torch.rand(n, device="cuda", generator=g) < 0.5, -1.0, 1.0)
        lam = torch.exp(e) * sign
    return _symmetric((q * lam) @ q.T)


def _gapped(n, gap, g, batch):
    s = torch.rand(batch, n, dtype=_F64, device="cuda", generator=g).sort(dim=-1).values
    return -1.0 + (2.0 - (n - 1) * gap) * s + torch.arange(n, dtype=_F64, device="cuda") * gap


def _batch_matrices(case, seed):
    # the sizes belong to the case, as in the seeded workload; the values to the seed
    gs = torch.Generator()
    gs.manual_seed(case["count"])
    sizes = torch.randint(case["lo"], case["hi"] + 1, (case["count"],), generator=gs).tolist()
    g = _generator(seed)
    flat = torch.randn(sum(n * n for n in sizes), dtype=_F64, device="cuda", generator=g)
    mats, at = [], 0
    for n in sizes:
        mats.append(_symmetric(flat[at:at + n * n].view(n, n)) / math.sqrt(n))
        at += n * n
    return sizes, mats


def _product_operands(case, seed):
    g = _generator(seed)
    m, n, k = case["m"], case["n"], case["k"]
    a = torch.randn((k, m) if case["ta"] == "T" else (m, k), dtype=_F64, device="cuda", generator=g)
    b = torch.randn((n, k) if case["tb"] == "T" else (k, n), dtype=_F64, device="cuda", generator=g)
    return a, b


_OPTS = {"solve": {}, "two_pass": {"precond_passes": 2}, "plain": {"method": "plain"},
         "cyclic": {"ordering": "cyclic"}}


def prepare(case, seed):
    f = case["family"]
    s = {"case": case}
    if f in _OPTS:
        s["A"] = _matrix(case, seed)
        if case["workspace"]:
            s["work"] = torch.empty(mpj.syev_workspace(case["n"], **_OPTS[f]), dtype=torch.uint8, device="cuda")
    elif f in ("eigh", "backward"):
        n, g = case["n"], _generator(seed)
        batch = case.get("batch", 1)
        q = _haar(n, g, batch)
        w = _gapped(n, case["gap"], g, batch)
        dw = torch.randn(batch, n, dtype=_F64, device="cuda", generator=g)
        dq = torch.randn(batch, n, n, dtype=_F64, device="cuda", generator=g)
        if f == "eigh":
            s["A"] = _symmetric((q[0] * w[0]) @ q[0].T).requires_grad_()
            s["dW"], s["dQ"] = dw[0], dq[0]
        else:
            s["W"], s["Q"], s["dW"], s["dQ"] = w, q, dw, dq
    elif f == "batched":
        sizes, s["mats"] = _batch_matrices(case, seed)
        s["solver"] = mpj.BatchedSolver(sizes)
        s["rows"] = torch.tensor([n for n in sizes for _ in range(n)], device="cuda")
    else:
        s["A"], s["B"] = _product_operands(case, seed)
    return s


# ------------------------------------------------------------------ the calls
def _signs(sums):
    return torch.where(sums < 0, -1.0, 1.0).to(_F64)


def _fixed(q):
    return q * _signs(q.sum(0))


def run(s):
    case = s["case"]
    f = case["family"]
    if f in _OPTS:
        if f == "solve" and not case["workspace"]:
            w, q = mpj.syev(s["A"])
        else:
            r = mpj.syev_ex(s["A"], workspace=s.get("work"), **_OPTS[f])
            w, q = r.W, r.Q
        return {"W": w, "Q": _fixed(q)}
    if f == "eigh":
        w, q = mpj.eigh(s["A"])
        q = q * _signs(q.detach().sum(0))
        dA, = torch.autograd.grad((w, q), s["A"], (s["dW"], s["dQ"]))
        return {"W": w.detach(), "Q": q.detach(), "dA": dA}
    if f == "backward":
        return {"dA": mpj.syev_backward(s["W"], s["Q"], s["dW"], s["dQ"])}
    if f == "batched":
        w, q, _, _ = s["solver"].solve(s["mats"])
        flat = torch.cat([x.T.reshape(-1) for x in q])  # one eigenvector after the other
        sign = _signs(torch.segment_reduce(flat, "sum", lengths=s["rows"], unsafe=True))
        return {"W": torch.cat(w), "Q": flat * torch.repeat_interleave(sign, s["rows"], output_size=flat.numel())}
    return {"C": mpj.dgemm_tc(case["ta"], case["tb"], 1.0, s["A"], s["B"])}


# ------------------------------------------------------------------ floors and 64-bit values
def work(case):
    """Algorithm 9 in nominal counts: 7 FP32 and 2 FP64 sweeps (plain: 10) of
    4 n^3 flops (both sides of a symmetric A, and V, one FMA an entry), two
    Newton-Schulz steps of 3 n^3 and a transform of 3 n^3 with the symmetric
    products' halves; the adjoint's three products 5 n^3."""
    f = case["family"]
    if f in _OPTS:
        n = case["n"]
        per = {"solve": 45, "cyclic": 45, "two_pass": 84, "plain": 40}[f]
        return {"bytes": 8 * (2 * n * n + n), "flops": per * n ** 3}
    if f == "eigh":
        n = case["n"]
        return {"bytes": 8 * (4 * n * n + 2 * n), "flops": 50 * n ** 3}
    if f == "backward":
        n = case["n"]
        return {"bytes": 8 * case["batch"] * (3 * n * n + 2 * n), "flops": 5 * case["batch"] * n ** 3}
    if f == "batched":
        lo, hi, c = case["lo"], case["hi"], case["count"]
        sizes = range(lo, hi + 1)
        n2 = sum(n * n for n in sizes) / len(sizes)
        n3 = sum(n ** 3 for n in sizes) / len(sizes)
        return {"bytes": 8 * c * (2 * n2 + (lo + hi) / 2), "flops": 45 * c * n3}
    m, n, k = case["m"], case["n"], case["k"]
    return {"bytes": 8 * (m * k + k * n + m * n), "flops": 2 * m * n * k}


def exact(case, seed):
    f = case["family"]
    if f in _OPTS:
        w, q = torch.linalg.eigh(_matrix(case, seed))
        return {"W": w, "Q": _fixed(q)}
    if f == "product":
        a, b = _product_operands(case, seed)
        return {"C": (a.T if case["ta"] == "T" else a) @ (b.T if case["tb"] == "T" else b)}
    if f == "batched":
        ws, qs = [], []
        for a in _batch_matrices(case, seed)[1]:
            w, q = torch.linalg.eigh(a.cpu())
            ws.append(w)
            qs.append((_fixed(q)).T.reshape(-1))
        return {"W": torch.cat(ws), "Q": torch.cat(qs)}
    s = prepare(case, seed)
    if f == "eigh":
        w, q = torch.linalg.eigh(s["A"].detach())
        w, q, dw, dq = w[None], _fixed(q)[None], s["dW"][None], s["dQ"][None]
    else:
        w, q, dw, dq = s["W"], s["Q"], s["dW"], s["dQ"]
    gap = w[:, None, :] - w[:, :, None]
    gap = gap + torch.eye(w.shape[1], dtype=_F64, device="cuda")
    g = (q.transpose(1, 2) @ dq) / gap
    g = g - torch.diag_embed(torch.diagonal(g, dim1=1, dim2=2)) + torch.diag_embed(dw)
    dA = _symmetric(q @ g @ q.transpose(1, 2))
    return {"dA": dA} if f == "backward" else {"W": w[0], "Q": q[0], "dA": dA[0]}
