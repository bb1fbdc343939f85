"""The workloads that the solver's speed is judged by, through its public calls.

Each case is what a program that uses the library has it do: a batch solved
with ``Solver.submit`` / ``wait``, many batches of different sizes submitted
and flushed together, host-buffer requests through the request server, and
the sensitivities of roots by ``nls_adjoint``.  Sizes follow the workloads of
``inputs.py`` and ``bench.py`` (cubic n = 3 and n = 8, the uneven 2..32 mix,
serving, Bratu n = 64..128) and the paper's ten-dimensional Rosenbrock batch,
with odd sizes between them.

A solve returns the roots and the per-instance statuses.  The other
per-instance outputs (pass counts, the last residual, which at a root is a
rounding residue below abstol) are optional diagnostics and stay unbound, as
in a program that wants the roots.
"""
from __future__ import annotations

import math
import random

import numpy as np  # noqa: F401
import torch

import paper_2403_16341_gb300 as nls

FAMILY = {"cubic": nls.NLS_CUBIC, "bratu": nls.NLS_BRATU, "square": nls.NLS_SQUARE,
          "rosenbrock": nls.NLS_ROSENBROCK}
ALG = {"newton": nls.NLS_NEWTON, "linesearch": nls.NLS_NEWTON_BACKTRACK,
       "trust": nls.NLS_TRUST_DOGLEG, "halley": nls.NLS_HALLEY}
ABSTOL = 1e-10
# Newton passes per instance that these problems need (an instance cannot do
# with fewer at abstol = 1e-10), for the operation counts of work()
PASSES = {"cubic": 5, "bratu": 4, "square": 6, "rosenbrock": 18}


# --------------------------------------------------------------------- cases

def listed():
    return [
        # The smallest real call: one small batch of three-dimensional systems
        # by plain Newton with the closed-form Jacobian; launch latency counts.
        _solve("cubic3_1k_newton", "cubic", 3, 1024, "newton", "fp64", jac="analytic"),
        # The paper's GPU example: 1024 ten-dimensional Rosenbrock systems from
        # random starts; long uneven iteration counts in a small batch.
        _solve("rosenbrock10_1k_trust", "rosenbrock", 10, 1024, "trust", "fp64"),
        # The headline batch, globalised Newton in FP64: one instance per thread.
        _solve("cubic8_1m_linesearch_fp64", "cubic", 8, 1 << 20, "linesearch", "fp64"),
        # The headline batch in mixed precision with the trust region.
        _solve("cubic8_1m_trust_mixed", "cubic", 8, 1 << 20, "trust", "mixed"),
        # A collocation-type sweep at an odd size and an odd count, full
        # precision: one instance per warp segment, FP64 LU.
        _solve("cubic27_20k_trust_fp64", "cubic", 27, 20011, "trust", "fp64"),
        # The largest size of the warp tiling in mixed precision.
        _solve("cubic32_64k_linesearch_mixed", "cubic", 32, 1 << 16, "linesearch", "mixed"),
        # An uneven mix, n log-uniform in 2..32, half cubic and half Bratu: 62
        # batches submitted one by one and flushed together.
        {"name": "uneven_256k_linesearch_mixed", "kind": "uneven", "count": 1 << 18, "n_lo": 2, "n_hi": 32,
         "alg": "linesearch", "precision": "mixed"},
        # Larger discretised boundary-value problems, n uniform in 64..128, one
        # instance per CTA: FP32 LU under an FP64 residual ...
        {"name": "bratu64_128_16k_trust_mixed", "kind": "spread", "count": 16384, "n_lo": 64, "n_hi": 128,
         "alg": "trust", "precision": "mixed"},
        # ... and with the FP64 LU (the largest case).
        {"name": "bratu64_128_16k_trust_fp64", "kind": "spread", "count": 16384, "n_lo": 64, "n_hi": 128,
         "alg": "trust", "precision": "fp64"},
        # Dense systems at an odd size, every FP32 Newton step refined.
        _solve("cubic100_2k_linesearch_refined", "cubic", 100, 2003, "linesearch", "refined"),
        # The backward direction: gradients of a loss of the roots with respect
        # to all parameters, at the roots of the largest warp-tiled size.
        {"name": "adjoint_cubic32_64k", "kind": "adjoint", "family": "cubic", "n": 32, "batch": 1 << 16},
        # A burst of serving requests on pinned host buffers (1..4096 instances
        # each, n in {3, 8, 16, 32}, both families), all admitted and waited for.
        {"name": "serve_burst_96", "kind": "serve", "requests": 96, "max_batch": 4096, "alg": "linesearch",
         "precision": "mixed"},
    ]


def _solve(name, family, n, batch, alg, precision, jac="dual"):
    return {"name": name, "kind": "solve", "family": family, "n": n, "batch": batch, "alg": alg,
            "precision": precision, "jac": jac}


def _log_uniform(rng, lo, hi):
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng: random.Random):
    kind = rng.choice(["solve"] * 6 + ["uneven", "spread", "adjoint", "serve"])
    if kind == "uneven":
        lo = rng.randint(2, 5)
        case = {"kind": kind, "count": _log_uniform(rng, 1 << 13, 1 << 18), "n_lo": lo,
                "n_hi": rng.randint(lo + 6, 32), "alg": rng.choice(["newton", "linesearch", "trust"]),
                "precision": rng.choice(["fp64", "mixed"])}
    elif kind == "spread":
        lo = rng.randint(33, 100)
        case = {"kind": kind, "count": _log_uniform(rng, 1 << 10, 1 << 14), "n_lo": lo,
                "n_hi": rng.randint(lo, min(128, lo + 50)), "alg": rng.choice(["newton", "linesearch", "trust"]),
                "precision": rng.choice(["fp64", "mixed", "refined"])}
    elif kind == "serve":
        case = {"kind": kind, "requests": _log_uniform(rng, 8, 128), "max_batch": _log_uniform(rng, 256, 4096),
                "alg": rng.choice(["linesearch", "trust"]), "precision": rng.choice(["fp64", "mixed"])}
    elif kind == "adjoint":
        family = rng.choice(["cubic", "cubic", "bratu"])
        n = _log_uniform(rng, 2, 128)
        case = {"kind": kind, "family": family, "n": n, "batch": _draw_batch(rng, family, n)}
    else:
        family = rng.choice(["cubic"] * 4 + ["bratu"] * 2 + ["square", "rosenbrock"])
        n = _log_uniform(rng, 2, 12 if family == "rosenbrock" else 128)
        alg = "trust" if family == "rosenbrock" else rng.choice(
            ["newton", "linesearch", "linesearch", "trust", "trust"] + (["halley"] if family == "cubic" else []))
        precision = rng.choice(["fp64", "mixed"] + (["refined"] if n > 32 and alg != "halley" else []))
        jac = rng.choice(["dual", "analytic"]) if n <= 8 and alg != "halley" else "dual"
        case = {"kind": kind, "family": family, "n": n, "batch": _draw_batch(rng, family, n), "alg": alg,
                "precision": precision, "jac": jac}
    # no drawn case costs more than the largest listed one
    largest = max(work(c)["flops"] for c in listed())
    while work(case)["flops"] > largest:
        key = "requests" if kind == "serve" else "count" if kind in ("uneven", "spread") else "batch"
        case[key] = max(1, case[key] // 2)
    return case


def _draw_batch(rng, family, n):
    # up to 2^20 small instances; the parameters and the LU work bound the rest
    most = min(1 << 20, int(6e8 / (8 * (_n_params(family, n) + 2 * n))), int(8e9 / n ** 3))
    return _log_uniform(rng, min(1000, most), most)


# --------------------------------------------------------------- the buckets

def _n_params(family, n):
    return {"cubic": n * n + n, "bratu": 1, "square": n, "rosenbrock": 0}[family]


def _alg(case):
    flags = {"fp64": 0, "mixed": nls.NLS_MIXED, "refined": nls.NLS_MIXED | nls.NLS_REFINE}[case["precision"]]
    if case.get("jac") == "analytic":
        flags |= nls.NLS_ANALYTIC_JAC
    return ALG[case["alg"]] | flags


def _buckets(case):
    """(family, n, batch) of every uniform batch of the case."""
    if case["kind"] in ("solve", "adjoint"):
        return [(case["family"], case["n"], case["batch"])]
    if case["kind"] == "uneven":  # the expected counts of n log-uniform in n_lo..n_hi
        lo, hi = case["n_lo"], case["n_hi"]
        span = math.log((hi + 1) / lo)
        return [(f, n, max(1, round(case["count"] / 2 * math.log((n + 1) / n) / span)))
                for f in ("cubic", "bratu") for n in range(lo, hi + 1)]
    if case["kind"] == "spread":  # n uniform in n_lo..n_hi
        sizes = range(case["n_lo"], case["n_hi"] + 1)
        per, more = divmod(case["count"], len(sizes))
        return [("bratu", n, per + (i < more)) for i, n in enumerate(sizes) if per + (i < more)]
    # serve: log-uniform request sizes in a fixed mixed order
    r, out = case["requests"], []
    for i in range(r):
        b = int(math.exp((i + 0.5) / r * math.log(case["max_batch"] + 1)))
        out.append((("cubic", "bratu")[i % 2], (3, 8, 16, 32)[(i // 2) % 4], max(1, min(b, case["max_batch"]))))
    random.Random(r).shuffle(out)
    return out


def _inputs(family, n, batch, gen):
    """params [E, batch] and u0 [n, batch]: A = 3 I + G with b ~ U[-w, w]^n
    (cubic), lambda ~ U[0.5, 3] (Bratu), p ~ U[0.25, 9]^n (square), random
    starts (Rosenbrock)."""
    dev = "cuda"
    u0 = torch.zeros(n, batch, dtype=torch.float64, device=dev)
    if family == "cubic":
        sigma = 0.3 if n <= 32 else 0.3 * math.sqrt(32.0 / n)
        p = torch.empty(n * n + n, batch, dtype=torch.float64, device=dev)
        p[: n * n].normal_(0.0, sigma, generator=gen)
        p[: n * n : n + 1] += 3.0
        w = 5.0 if n == 8 else 2.0
        p[n * n:].uniform_(-w, w, generator=gen)
    elif family == "bratu":
        p = torch.empty(1, batch, dtype=torch.float64, device=dev).uniform_(0.5, 3.0, generator=gen)
    elif family == "square":
        p = torch.empty(n, batch, dtype=torch.float64, device=dev).uniform_(0.25, 9.0, generator=gen)
        u0.fill_(1.0)
    else:
        p = torch.empty(0, batch, dtype=torch.float64, device=dev)
        u0.uniform_(0.0, 1.0, generator=gen)
    return p, u0


def _all_inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return [(f, n, b) + _inputs(f, n, b, gen) for f, n, b in _buckets(case)], gen


def _adjoint_inputs(case, seed):
    """params, roots and cotangents: roots drawn first, b from F(u) = 0."""
    (f, n, b, p, _), = _all_inputs(case, seed)[0]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 1)
    u = torch.empty(n, b, dtype=torch.float64, device="cuda").uniform_(-0.7, 0.7, generator=gen)
    if f == "cubic":
        p[n * n:] = torch.einsum("ijb,jb->ib", p[: n * n].view(n, n, b), u) + u ** 3
    w = torch.empty(n, b, dtype=torch.float64, device="cuda").normal_(generator=gen)
    return f, n, b, p, u, w


class _Server:
    """A request server and the end of its life."""

    def __init__(self):
        self.s = nls.nls_server_create(0, 1 << 30, 4)

    def __del__(self):
        if self.s:
            nls.nls_server_destroy(self.s)
            self.s = None


# ---------------------------------------------------------------- run and co

def prepare(case, seed):
    if case["kind"] == "adjoint":
        f, n, b, p, u, w = _adjoint_inputs(case, seed)
        return {"kind": "adjoint", "solver": nls.Solver(0), "family": FAMILY[f], "n": n, "batch": b, "params": p,
                "u": u, "w": w, "grad": torch.empty_like(p),
                "status": torch.empty(b, dtype=torch.int32, device="cuda")}
    data, _ = _all_inputs(case, seed)
    rows, total = sum(n * b for _, n, b, _, _ in data), sum(b for _, _, b, _, _ in data)
    host = case["kind"] == "serve"
    kw = {"pin_memory": True} if host else {"device": "cuda"}
    # the roots of all batches lie in one array, their statuses in another
    u0 = torch.cat([x.reshape(-1) for *_, x in data])
    u = torch.empty(rows, dtype=torch.float64, **kw)
    status = torch.empty(total, dtype=torch.int32, **kw)
    if host:
        u0 = u0.cpu()
        flat = torch.empty(sum(p.numel() for *_, p, _ in data), dtype=torch.float64, pin_memory=True)
    batches, iu, ib, ip = [], 0, 0, 0
    for f, n, b, p, _ in data:
        if host:
            q = flat[ip: ip + p.numel()].view(p.shape)
            q.copy_(p)
            ip += p.numel()
            p = q
        batches.append((FAMILY[f], p, u[iu: iu + n * b].view(n, b), status[ib: ib + b]))
        iu, ib = iu + n * b, ib + b
    state = {"kind": case["kind"], "alg": _alg(case), "batches": batches, "u0": u0, "u": u, "status": status,
             "maxiters": 300 if case.get("family") == "rosenbrock" else 50}
    if host:
        torch.cuda.synchronize()
        state["server"] = _Server()
    else:
        state["solver"] = nls.Solver(0)
    return state


def run(state):
    if state["kind"] == "adjoint":
        s = state
        nls.nls_adjoint(s["solver"].h, s["family"], s["params"].data_ptr(), s["u"].data_ptr(), s["n"], s["batch"],
                        s["w"].data_ptr(), s["grad"].data_ptr(), s["status"].data_ptr())
        return {"grad": s["grad"], "status": s["status"]}
    state["u"].copy_(state["u0"])
    if state["kind"] == "serve":
        srv = state["server"].s
        tickets = [nls.nls_server_submit(srv, f, p.data_ptr(), u.data_ptr(), u.shape[0], u.shape[1], state["alg"],
                                         ABSTOL, state["maxiters"], st.data_ptr())
                   for f, p, u, st in state["batches"]]
        solved = sum(nls.nls_server_wait(srv, t)[0] for t in tickets)
    else:
        solver = state["solver"]
        reqs = [solver.submit(f, p, u, state["alg"], ABSTOL, state["maxiters"], (st, None, None, None))
                for f, p, u, st in state["batches"]]
        solver.flush()
        solved = sum(solver.wait(r) for r in reqs)
    return {"u": state["u"], "status": state["status"], "solved": solved}


def work(case):
    """Bytes: parameters and u0 read once, roots and statuses written once
    (adjoint: parameters, roots and cotangents read, gradients written).
    Operations: the FP64 residuals and, per pass, one dense LU with its two
    triangular solves (the trust region's and the line search's scalar work
    left out)."""
    nbytes = flops = 0
    for f, n, b in _buckets(case):
        e = _n_params(f, n)
        lu = 2 * n ** 3 / 3 + 2 * n * n
        residual = 2 * n * n + 3 * n if f == "cubic" else 8 * n
        if case["kind"] == "adjoint":
            nbytes += b * (8 * (2 * e + 2 * n) + 4)
            flops += b * (lu + e)
        else:
            nbytes += b * (8 * (e + 2 * n) + 4)
            flops += b * (PASSES[f] * (lu + residual) + residual)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------- 64 bits

def _residual_jacobian(family, n, p, u):
    """F [b, n] and J [b, n, n] at u [b, n]."""
    b = u.shape[0]
    if family == "cubic":
        a = p[: n * n].t().reshape(b, n, n)
        return (a @ u[..., None])[..., 0] + u ** 3 - p[n * n:].t(), a + torch.diag_embed(3 * u * u)
    if family == "bratu":
        h2, lam = float((n + 1) ** 2), p[0][:, None]
        z = torch.zeros(b, 1, dtype=u.dtype, device=u.device)
        v = torch.cat([z, u, z], 1)
        off = torch.full((b, n - 1), h2, dtype=u.dtype, device=u.device)
        j = torch.diag_embed(-2 * h2 + lam * u.exp()) + torch.diag_embed(off, 1) + torch.diag_embed(off, -1)
        return h2 * (v[:, :-2] - 2 * u + v[:, 2:]) + lam * u.exp(), j
    return u * u - p.t(), torch.diag_embed(2 * u)


def _root(family, n, p, u0):
    """The root by damped Newton to the end of what 64 bits give; [n, batch]."""
    if family == "rosenbrock":
        return torch.ones_like(u0)
    out = torch.empty_like(u0)
    step = max(1, int(2.5e8 / (n * n + 1)) // 4)
    for k in range(0, u0.shape[1], step):
        q, u = p[:, k: k + step], u0[:, k: k + step].t().contiguous()
        f, j = _residual_jacobian(family, n, q, u)
        for _ in range(14):
            d = torch.linalg.solve(j, f[..., None])[..., 0]
            alpha = torch.ones(u.shape[0], 1, dtype=u.dtype, device=u.device)
            for _ in range(6):
                worse = _residual_jacobian(family, n, q, u - alpha * d)[0].norm(dim=1) > 1.5 * f.norm(dim=1) + 1e-9
                if not worse.any():
                    break
                alpha[worse] *= 0.5
            u = u - alpha * d
            f, j = _residual_jacobian(family, n, q, u)
            if f.abs().max() < 1e-12 * (n + 1) ** (2 if family == "bratu" else 1):
                u = u - torch.linalg.solve(j, f[..., None])[..., 0]
                break
        out[:, k: k + step] = u.t()
    return out


def exact(case, seed):
    if case["kind"] == "adjoint":
        f, n, b, p, u, w = _adjoint_inputs(case, seed)
        grad = torch.empty_like(p)
        step = max(1, int(2.5e8 / (n * n)) // 4)
        for k in range(0, b, step):
            v = u[:, k: k + step].t().contiguous()
            _, j = _residual_jacobian(f, n, p[:, k: k + step], v)
            mu = torch.linalg.solve(j.transpose(1, 2), w[:, k: k + step].t()[..., None])[..., 0]
            if f == "cubic":
                grad[: n * n, k: k + step] = -(mu[:, :, None] * v[:, None, :]).reshape(v.shape[0], n * n).t()
                grad[n * n:, k: k + step] = mu.t()
            elif f == "bratu":
                grad[0, k: k + step] = -(mu * v.exp()).sum(1)
        return {"grad": grad, "status": None}
    data, _ = _all_inputs(case, seed)
    u = torch.cat([_root(f, n, p, u0).reshape(-1) for f, n, b, p, u0 in data])
    return {"u": u, "status": None, "solved": None}
