"""The work that programs have this library do, as cases that can be timed: which problems, how their inputs are
made, and the one call through the public binding (``paper_2603_09221_b200.lqr.LqrSolver``) that is a pass.

A case names an entry point (``op``) and its sizes:

  solve        time-invariant solve: ``K, P, x, u`` of every instance, or ``P_0`` and ``u_0`` (``first``)
  solve_tv     time-varying solve from operands in memory, ``P_0`` and ``u_0``
  grad         gradients of a loss of ``u_0`` with respect to every operand of the time-varying problem
  layer        contextualised Test-Time Control layer: ``u_1`` (and ``P_0``) from its coefficient vectors
  layer_grad   gradients of that layer with respect to every coefficient vector and both bases

``batch`` is sequences x heads x tokens.  A, B, R belong to the head (``per_instance``: to the instance); Q and x_0 to
the token.  Every pass writes into buffers that the program keeps, as a training or serving loop does.
"""
import math

import numpy as np
import torch

from paper_2603_09221_b200 import lqr

DEVICE = "cuda:0"


def _case(op, batch, n, H, m=None, dtype="f32", rho=0.9, first=False, per_instance=False, name=None, r=16, value=True):
    c = dict(op=op, seqs=batch[0], heads=batch[1], tokens=batch[2], n=n, m=n if m is None else m, H=H)
    if op == "solve":
        c.update(dtype=dtype, rho=rho, first=first, per_instance=per_instance)
    if op in ("layer", "layer_grad"):
        c.update(r=r)
    if op == "layer":
        c.update(value=value)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest call: one layer, one new token of one sequence, 16 heads (decoding).  Only the control is wanted.
        _case("layer", (1, 16, 1), 16, 32, value=False, name="layer_decode_d16"),
        # A bank of 64 small unrelated controllers, each with its own dynamics (configuration 0 of the benchmark).
        _case("solve", (1, 1, 64), 8, 8, per_instance=True, name="bank_n8"),
        # A short training batch at the layer's state dimension, dense dynamics per head (configuration 1).
        _case("solve", (4, 8, 128), 16, 16, name="batch_n16"),
        # A plant whose sizes are no power of two and fewer controls than states, a ragged number of tokens.
        _case("solve", (3, 5, 77), 40, 20, m=12, name="ragged_n40_m12"),
        # Few instances over a long planning horizon: the library takes the scan over the horizon here.
        _case("solve", (1, 16, 4), 16, 1024, rho=0.98, name="horizon_n16_H1024"),
        # Long horizon, many instances (configuration 3).
        _case("solve", (1, 16, 1024), 32, 64, rho=0.98, name="long_n32"),
        # Wide heads in bfloat16 with every result kept (configuration 2), and the largest call: prefill of wide heads
        # where the value and the first control are wanted (configuration 4).
        _case("solve", (4, 8, 2048), 64, 8, dtype="bf16", name="wide_n64_all"),
        _case("solve", (2, 16, 4096), 64, 16, dtype="bf16", first=True, name="wide_n64_first"),
        # One layer over the tokens of a training batch with its parameters from memory: forward, and the gradients.
        _case("solve_tv", (4, 16, 1024), 16, 32, name="tv_n16"),
        _case("grad", (4, 16, 1024), 16, 32, name="grad_n16"),
        # The same layer in its contextualised form: prefill, and the backward pass of training.
        _case("layer", (4, 16, 1024), 16, 32, name="layer_prefill_d16"),
        _case("layer_grad", (4, 16, 1024), 16, 32, name="layer_grad_d16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _batch(rng, lo, hi):
    """Sequences x heads x tokens with a total between about lo and hi, the number of tokens odd as often as not."""
    total = _log_int(rng, lo, hi)
    heads = rng.choice((1, 2, 3, 5, 8, 12, 16))
    while heads > total:
        heads //= 2
    heads = max(heads, 1)
    seqs = max(1, min(rng.choice((1, 1, 2, 3, 4)), total // heads))
    return seqs, heads, max(1, total // (seqs * heads))


def draw(rng):
    kind = rng.choice(("bank", "batch", "ragged", "horizon", "long", "wide_all", "wide_first", "tv", "grad", "layer",
                       "layer", "layer_grad"))
    if kind == "bank":                              # small plants, m <= n
        n = rng.randint(3, 16)
        return _case("solve", (1, 1, _log_int(rng, 16, 4096)), n, _log_int(rng, 4, 48), m=rng.randint(1, n),
                     per_instance=True, first=rng.random() < 0.25)
    if kind == "batch":
        return _case("solve", _batch(rng, 64, 32768), 16, _log_int(rng, 4, 64), first=rng.random() < 0.3,
                     dtype=rng.choice(("f32", "f32", "bf16")))
    if kind == "ragged":
        n = rng.randint(10, 60)
        return _case("solve", _batch(rng, 64, 2048), n, _log_int(rng, 4, 32), m=rng.randint(max(2, n // 6), n),
                     first=rng.random() < 0.3)
    if kind == "horizon":
        return _case("solve", _batch(rng, 4, 128), rng.choice((16, 32)), _log_int(rng, 256, 2048), rho=0.98,
                     first=rng.random() < 0.3)
    if kind == "long":
        return _case("solve", _batch(rng, 128, 16384), 32, _log_int(rng, 8, 64), rho=0.98, first=rng.random() < 0.3)
    if kind == "wide_all":
        return _case("solve", _batch(rng, 256, 65536), 64, rng.randint(2, 8), dtype="bf16")
    if kind == "wide_first":
        return _case("solve", _batch(rng, 256, 131072), 64, rng.randint(2, 16), dtype="bf16", first=True)
    n = rng.choice((16, 16, 16, 32))
    top = 65536 if n == 16 else 8192
    if kind == "tv":
        return _case("solve_tv", _batch(rng, 64, top), n, _log_int(rng, 8, 32))
    if kind == "grad":
        return _case("grad", _batch(rng, 64, top), n, _log_int(rng, 8, 32))
    if kind == "layer":
        N = _batch(rng, 16, top)
        T = _log_int(rng, 8, 128)
        while N[0] * N[1] * N[2] * T > top * 32:
            T //= 2
        return _case("layer", N, n, T, r=rng.choice((4, 8, 16, 16)), value=rng.random() < 0.5)
    return _case("layer_grad", _batch(rng, 64, top), n, _log_int(rng, 8, 32), r=rng.choice((4, 8, 16, 16)))


def _instances(c):
    return c["seqs"] * c["heads"] * c["tokens"]


def _gen(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    return g


def _sym(X):
    return 0.5 * (X + X.transpose(-1, -2))


def _psd(shape, n, gen, shift, chunk=4096):
    """L L'/n + shift I for Gaussian L, made a few thousand matrices at a time."""
    out = torch.empty(shape + (n, n), device=DEVICE)
    flat = out.view(-1, n, n)
    eye = shift * torch.eye(n, device=DEVICE)
    step = max(1, chunk * 4096 // (n * n))
    for i in range(0, flat.shape[0], step):
        L = torch.randn(flat[i:i + step].shape, generator=gen, device=DEVICE)
        flat[i:i + step] = _sym(L @ L.transpose(-1, -2) / n) + eye
    return out


def _prepare_solve(c, seed):
    n, m, N = c["n"], c["m"], _instances(c)
    batch = (c["seqs"], c["heads"], c["tokens"])
    sys_shape = batch if c["per_instance"] else (1, c["heads"], 1)
    rng = np.random.default_rng(seed)
    G = rng.standard_normal((int(np.prod(sys_shape)), n, n))
    A = G * (c["rho"] / np.abs(np.linalg.eigvals(G)).max(axis=1))[:, None, None]      # spectral radius rho
    gen = _gen(seed)
    s = dict(op="solve", H=c["H"])
    s["A"] = torch.from_numpy(A.astype(np.float32).reshape(sys_shape + (n, n))).to(DEVICE)
    s["B"] = torch.randn(sys_shape + (n, m), generator=gen, device=DEVICE) / n ** 0.5
    s["R"] = _psd(sys_shape, m, gen, 0.1)
    qdt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    if c["first"] and n == 64:                      # low rank plus diagonal, handed over densely
        Q = torch.empty((N, n, n), dtype=qdt, device=DEVICE)
        for i in range(0, N, 8192):
            U = torch.randn((min(8192, N - i), n, 8), generator=gen, device=DEVICE)
            d = 0.05 + 0.15 * torch.rand((U.shape[0], n), generator=gen, device=DEVICE)
            Q[i:i + 8192] = (_sym(U @ U.transpose(1, 2) / 8) + torch.diag_embed(d)).to(qdt)
        s["Q"] = Q.view(batch + (n, n))
    else:
        s["Q"] = _psd(batch, n, gen, 0.1).to(qdt)
    s["x0"] = torch.randn(batch + (n,), generator=gen, device=DEVICE).to(qdt)
    s["solver"] = lqr.LqrSolver(n, m, c["H"], batch)
    s["flags"] = lqr.TTC_OUT_FIRST_ONLY if c["first"] else 0
    s["out"] = lqr.alloc_outputs(n, m, c["H"], N, DEVICE, first_only=c["first"],
                                 want=("P", "u", "info") if c["first"] else ("K", "P", "x", "u", "info"))
    return s


def _prepare_tv(c, seed):
    n, m, H, N = c["n"], c["m"], c["H"], _instances(c)
    batch = (c["seqs"], c["heads"], c["tokens"])
    head = (1, c["heads"], 1, H)
    gen = _gen(seed)
    rn = lambda *shape: torch.randn(shape, generator=gen, device=DEVICE)
    s = dict(op=c["op"], H=H)
    s["A"] = torch.eye(n, device=DEVICE) + 0.1 * rn(*head, n, n) / n ** 0.5
    s["B"] = rn(*head, n, m) / n ** 0.5
    M = rn(*head, m, m)
    diag = torch.diag_embed(0.5 + torch.rand(head + (m,), generator=gen, device=DEVICE))
    s["R"] = _sym(diag + 0.05 * M @ M.transpose(-1, -2) / m).contiguous()
    s["Q"] = _psd(batch + (H,), n, gen, 0.05)
    s["Qf"] = _psd(batch, n, gen, 0.05)
    s["x0"] = rn(*batch, n)
    s["solver"] = lqr.LqrSolver(n, m, H, batch)
    e = lambda *shape: torch.empty(shape, device=DEVICE)
    if c["op"] == "grad":
        s["g"] = rn(N, m)
        s["out"] = dict(dA=e(N, H, n, n), dB=e(N, H, n, m), dQ=e(N, H, n, n), dQf=e(N, n, n), dR=e(N, H, m, m), dx0=e(N, n),
                        u0=e(N, m))
    else:
        s["out"] = dict(P=e(N, n, n), u=e(N, m))
    s["out"]["info"] = torch.empty((N,), dtype=torch.int32, device=DEVICE)
    return s


def _prepare_layer(c, seed):
    n, r, N = c["n"], c["r"], _instances(c)
    gen = _gen(seed)
    rn = lambda *shape: torch.randn(shape, generator=gen, device=DEVICE)
    sp = torch.nn.functional.softplus
    Qc = rn(r, n, n)
    s = dict(op=c["op"], H=c["H"])
    # what the coefficient projections of a layer hand over (here drawn), and the two bases that the layer keeps
    s["in"] = dict(s_a=0.3 * rn(N, n), s_gamma_a=sp(rn(N, n) - 2.0), s_gamma_b=sp(rn(N, n) - 2.0),
                   s_gamma_q=sp(rn(N, n) - 2.0), s_b=rn(N, r) / r ** 0.5, s_q=sp(rn(N, r)) / r, s_qf=sp(rn(N, r)) / r,
                   r_inv=sp(rn(N, n)) + 0.5, h0=rn(N, n), B_basis=rn(r, n, n) / n ** 0.5,
                   Q_basis=(Qc @ Qc.transpose(-1, -2) / n ** 0.5).contiguous())
    s["solver"] = lqr.LqrSolver(n, n, c["H"], (c["seqs"], c["heads"], c["tokens"]))
    s["out"] = dict(u1=torch.empty((N, n), device=DEVICE), info=torch.empty((N,), dtype=torch.int32, device=DEVICE))
    if c["op"] == "layer_grad":
        s["g"] = rn(N, n)
        s["grads"] = {k: torch.empty_like(v) for k, v in s["in"].items()}
    elif c["value"]:
        s["out"]["P0"] = torch.empty((N, n, n), device=DEVICE)
    return s


def prepare(case, seed):
    make = {"solve": _prepare_solve, "solve_tv": _prepare_tv, "grad": _prepare_tv, "layer": _prepare_layer,
            "layer_grad": _prepare_layer}
    return make[case["op"]](case, seed)


def run(s):
    op, H, solver, out = s["op"], s["H"], s["solver"], s["out"]
    if op == "solve":
        solver.solve(s["A"], s["B"], s["Q"], s["R"], s["x0"], H, flags=s["flags"], **out)
    elif op == "solve_tv":
        solver.solve_tv(s["A"], s["B"], s["Q"], s["R"], s["Qf"], s["x0"], H, flags=lqr.TTC_OUT_FIRST_ONLY, **out)
    elif op == "grad":
        solver.grad(s["A"], s["B"], s["Q"], s["R"], s["Qf"], s["x0"], s["g"], H, **out)
    elif op == "layer":
        solver.solve_layer(**s["in"], T=H, **out)
    else:
        solver.layer_grad(**s["in"], T=H, g=s["g"], grads=s["grads"], **out)
        return {**out, **s["grads"]}
    return out


def work(case):
    """Inputs read once, outputs written once; operations of the recursion with the symmetry of P, S and Z'Z used."""
    n, m, H, N = case["n"], case["m"], case["H"], _instances(case)
    op = case["op"]
    step = 3 * n ** 3 + 5 * n * n * m + 3 * n * m * m + m ** 3 / 3 + 2 * n * n + 4 * n * m
    if op == "solve":
        q = 2 if case["dtype"] == "bf16" else 4
        nsys = N if case["per_instance"] else case["heads"]
        size = 4 * nsys * (n * n + n * m + m * m) + N * q * (n * n + n)
        if case["first"]:
            size += 4 * N * (n * n + m + 1)
        else:
            size += 4 * N * (H * m * n + (H + 1) * n * n + (H + 1) * n + H * m + 1)
        return {"bytes": size, "flops": N * H * step}
    if op in ("solve_tv", "grad"):
        size = 4 * case["heads"] * H * (n * n + n * m + m * m) + 4 * N * ((H + 1) * n * n + n)
        if op == "solve_tv":
            return {"bytes": size + 4 * N * (n * n + m + 1), "flops": N * H * step}
        size += 4 * N * (m + H * (2 * n * n + n * m + m * m) + n * n + n + m + 1)
        outer = 3 * (2 * n * n + n * m + m * m) + 12 * n * n + 4 * n * m     # outer products; rollouts and co-states
        return {"bytes": size, "flops": N * H * (step + outer)}
    r = case["r"]
    # per step P B, B'(P B) and Z'Z with symmetry, the factorisation, the substitutions for Z; the parameters once
    flops = N * (H * (2 * n ** 3 + n ** 3 + n ** 3 + n ** 3 / 3 + n ** 3) + 6 * r * n * n)
    size = 4 * N * (6 * n + 3 * r) + 8 * r * n * n + 4 * N * (n + 1)
    if op == "layer":
        return {"bytes": size + (4 * N * n * n if case["value"] else 0), "flops": flops}
    # gains of every step, two rollouts and the co-states, the reductions onto coefficients and bases
    flops += N * (H * (n ** 3 + 16 * n * n) + 10 * r * n * n)
    return {"bytes": size + 4 * N * (7 * n + 3 * r) + 8 * r * n * n, "flops": flops}


def tolerance(case):
    # bfloat16 inputs run the tensor-core kernel in tf32 at n = 64; everything else is float32 arithmetic, whose
    # recursion, factorisation and substitutions leave a few units of 1e-6 in each result
    if case["op"] == "solve" and case["dtype"] == "bf16" and case["n"] == 64:
        return {"rel": 1e-2}
    return {"rel": 2e-5, "max": 1e-3}
