"""Workloads by which the speed of the coarsest-level solver is measured, through its public entry points.

A case is a dict of plain values.  ``kind`` names the entry point:

``apply``      ``CoarseOp.apply``: y = D_c x or D_c^H x, one or several columns, in one precision
``schur``      ``CoarseOp.schur``: the odd-even reduced operator, one column
``residual``   ``CoarseOp.residual``: FP64 residual and its norms, as refinement and its callers use it
``solve``      ``CoarseOp.solve``: GCRO-DR with the Leja polynomial inside FP64 refinement, to 1e-10
``batched``    ``solve_batched``: many operators of uneven size in lockstep
``grad``       ``CoarseSolve``: differentiable solve, forward and backward (adjoint solve, block gradients)

The operators are random ones with the structure of Galerkin coarse operators: sigma3-Hermitian self
blocks around a multiple of the identity, Gaussian forward hops, backward hops from the sigma3 relation.
The entries have the size of those that the generator in ``synthetic/`` produces, with hops strong enough
that a solve takes about as many Arnoldi steps as on its lattices.
"""
import math

import torch

import paper_2205_09104_gb300 as cg

PREC = {"fp64": cg.PREC_FP64, "fp32": cg.PREC_FP32, "bf16": cg.PREC_BF16}
# complex entries of one block, by precision
ENTRY_BYTES = {"fp64": 16, "fp32": 8, "bf16": 4}
VEC_BYTES = {"fp64": 16, "fp32": 8, "bf16": 8}

SELF_DIAG = 2.5      # mean diagonal of the self blocks
SELF_SPREAD = 0.4    # their random part: this over sqrt(n) per entry
HOP_RADIUS = 0.85    # spectral radius of the hops relative to the diagonal


def listed():
    return [
        # one column on the smallest lattice: launch and dependency latency
        {"name": "apply-fp32-4x4x4x4-n16", "kind": "apply", "dims": "4x4x4x4", "nv": 8, "mu": 0.0, "prec": "fp32",
         "nrhs": 1, "adjoint": False},
        # the stencil as a smoother or preconditioner calls it, mid-size lattice, adjoint product
        {"name": "apply-bf16-8x8x8x8-n32-adj", "kind": "apply", "dims": "8x8x8x8", "nv": 16, "mu": 0.0,
         "prec": "bf16", "nrhs": 1, "adjoint": True},
        # the twelve spin-colour columns of one propagator in single precision, unequal extents
        {"name": "apply-fp32-6x10x8x4-n32-c12", "kind": "apply", "dims": "6x10x8x4", "nv": 16, "mu": 0.0,
         "prec": "fp32", "nrhs": 12, "adjoint": False},
        # the same twelve columns through the BF16 tensor-core path, widest blocks
        {"name": "apply-bf16-8x8x8x8-n48-c12", "kind": "apply", "dims": "8x8x8x8", "nv": 24, "mu": 0.003,
         "prec": "bf16", "nrhs": 12, "adjoint": False},
        # odd extents, few columns, narrow blocks, adjoint
        {"name": "apply-bf16-7x6x9x5-n16-c5-adj", "kind": "apply", "dims": "7x6x9x5", "nv": 8, "mu": 0.003,
         "prec": "bf16", "nrhs": 5, "adjoint": True},
        # the true residual on the largest lattice: every refinement step computes one
        {"name": "residual-16x16x16x16-n48", "kind": "residual", "dims": "16x16x16x16", "nv": 24, "mu": 0.003},
        # the Krylov operator of odd-even solves: single precision, mid-size lattice
        {"name": "schur-fp32-8x8x8x8-n32", "kind": "schur", "dims": "8x8x8x8", "nv": 16, "mu": 0.0, "prec": "fp32"},
        # the polynomial chain's operator: BF16 blocks, unequal extents, widest blocks
        {"name": "schur-bf16-10x6x12x8-n48", "kind": "schur", "dims": "10x6x12x8", "nv": 24, "mu": 0.003,
         "prec": "bf16"},
        # one coarse solve of a Wilson-clover run
        {"name": "solve-8x8x8x8-n32", "kind": "solve", "dims": "8x8x8x8", "nv": 16, "mu": 0.0, "degree": 4, "k": 16},
        # one coarse solve of a twisted-mass run: the largest workload
        {"name": "solve-16x16x16x16-n48", "kind": "solve", "dims": "16x16x16x16", "nv": 24, "mu": 0.003, "degree": 8,
         "k": 32},
        # many operators of uneven size, one to twelve right-hand sides each
        {"name": "batched-12", "kind": "batched", "count": 12, "recipe": 4},
        # a training step through the solve: forward, adjoint solve, gradients of all nine blocks
        {"name": "grad-8x8x8x8-n32", "kind": "grad", "dims": "8x8x8x8", "nv": 16, "mu": 0.003, "degree": 4, "k": 16},
    ]


def _draw_dims(rng, low, high, even):
    """Four extents (2 .. 16) whose product lies near a volume spread over [low, high] on a log scale."""
    target = math.exp(rng.uniform(math.log(low), math.log(high)))
    best = None
    for _ in range(200):
        d = [2 * rng.randint(1, 8) for _ in range(4)] if even else [rng.randint(2, 16) for _ in range(4)]
        v = math.prod(d)
        if v <= high and (best is None or abs(math.log(v / target)) < abs(math.log(math.prod(best) / target))):
            best = d
    return "x".join(str(e) for e in best)


def draw(rng):
    kind = rng.choice(["apply"] * 5 + ["residual"] + ["schur"] * 2 + ["solve"] * 2 + ["batched", "grad"])
    nv = rng.choice([8, 16, 24])
    mu = rng.choice([0.0, 0.003])
    if kind == "apply":
        prec = rng.choice(["fp64", "fp32", "fp32", "bf16", "bf16"])
        nrhs = rng.choice([1, 1, rng.randint(2, 16)])
        top = 20000 if nrhs == 1 and prec != "fp64" else 4096
        return {"kind": kind, "dims": _draw_dims(rng, 64, top, False), "nv": nv, "mu": mu, "prec": prec, "nrhs": nrhs,
                "adjoint": rng.random() < 0.3}
    if kind == "residual":
        return {"kind": kind, "dims": _draw_dims(rng, 64, 20000, False), "nv": nv, "mu": mu}
    if kind == "schur":
        return {"kind": kind, "dims": _draw_dims(rng, 128, 20000, True), "nv": nv, "mu": mu,
                "prec": rng.choice(["fp32", "bf16"])}
    if kind == "batched":
        return {"kind": kind, "count": rng.randint(3, 12), "recipe": rng.randint(5, 10 ** 6)}
    degree, k = rng.choice([(4, 16), (8, 32), (4, 0)])
    return {"kind": kind, "dims": _draw_dims(rng, 256, 8000 if kind == "solve" else 4096, True), "nv": nv, "mu": mu,
            "degree": degree, "k": k}


# ------------------------------------------------------------------------------------------ inputs
def _dims(case):
    return tuple(int(v) for v in case["dims"].split("x"))


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _gauss(gen, *shape):
    return torch.randn(*shape, dtype=torch.complex128, device="cuda", generator=gen)


def _sigma3(n):
    s = torch.ones(n, dtype=torch.float64, device="cuda")
    s[n // 2:] = -1.0
    return s


def _blocks(gen, dims, nv):
    """Self blocks [V, n, n] and forward hops [V, 4, n, n] of a random coarse operator."""
    V, n = math.prod(dims), 2 * nv
    s = _sigma3(n)
    g = _gauss(gen, V, n, n).mul_(SELF_SPREAD / math.sqrt(2 * n))
    a = g + s[:, None] * g.mH * s
    a.diagonal(dim1=1, dim2=2).add_(SELF_DIAG)
    f = _gauss(gen, V, 4, n, n).mul_(SELF_DIAG * HOP_RADIUS / math.sqrt(8 * n))
    return a.contiguous(), f


def _roll(v, dims, mu, steps):
    """v[x] -> v[x - steps * mu] over sites (site index x0 + L0 (x1 + L1 (x2 + L2 x3)))."""
    w = v.reshape(*dims[::-1], *v.shape[1:])
    return torch.roll(w, steps, 3 - mu).reshape(v.shape)


def _hops64(f, dims, x):
    """Sum of the eight hops on x [V, n, R], in 64 bits."""
    s = _sigma3(x.shape[1])[:, None]
    y = torch.zeros_like(x)
    for mu in range(4):
        y += f[:, mu] @ _roll(x, dims, mu, -1)
        y += _roll(s * (f[:, mu].mH @ (s * x)), dims, mu, 1)
    return y


def _apply64(a, f, dims, x, mu):
    """D_c x for x [V, n, R], in 64 bits."""
    return a @ x + 1j * mu * _sigma3(x.shape[1])[:, None] * x + _hops64(f, dims, x)


def _adjoint64(a, f, dims, x, mu):
    s = _sigma3(x.shape[1])[:, None]
    return s * _apply64(a, f, dims, s * x, -mu)


def _columns(x):
    """[V, n, R] -> [R, V * n]"""
    return x.permute(2, 0, 1).reshape(x.shape[2], -1).contiguous()


def _sites(x, n):
    """[R, V * n] -> [V, n, R]"""
    return x.reshape(x.shape[0], -1, n).permute(1, 2, 0)


def _canonical_hops(f, dims):
    """All eight hops [V, 8, n, n] from the forward ones."""
    s = _sigma3(f.shape[-1])
    h = torch.empty(f.shape[0], 8, *f.shape[2:], dtype=f.dtype, device=f.device)
    h[:, :4] = f
    for mu in range(4):
        h[:, 4 + mu] = _roll(s[:, None] * f[:, mu].mH * s, dims, mu, 1)
    return h


def _even_sites(dims):
    i = torch.arange(math.prod(dims), device="cuda")
    p = torch.zeros_like(i)
    for e in dims:
        p += i % e
        i = i // e
    return p % 2 == 0


def _operator(a, f, dims, case, precisions, max_nrhs=1):
    return cg.CoarseOp(a, f, dims, case["nv"], mu=case["mu"], precisions=precisions, max_nrhs=max_nrhs,
                       assume_gamma5=True)


def _solve_params(case, extra=0):
    return cg.solve_params(m=50, max_restarts=100, tol=1e-10, poly_degree=case["degree"], defl_k=case["k"],
                           recycle_updates=10, precision=cg.PREC_FP32, inner_tol=2e-6, max_ir=20,
                           flags=cg.COARSE_ZERO_GUESS | cg.COARSE_POLY_BF16 | cg.COARSE_ODD_EVEN | extra)


def _setup_solves(op, case, gen, N, adjoint=False):
    """The solves of a multigrid setup: polynomial and recycle space, until the space is frozen."""
    full = cg.COARSE_RECYCLE_FULL_CYCLE if case["k"] else 0
    for i in range(12 if case["k"] else 1):
        _, info = op.solve(_gauss(gen, N), params=_solve_params(case, 0 if i else full), adjoint=adjoint)
        if info[0]["recycle_updates"] >= 10:
            break


def _recipe(case):
    """Uneven batch: extent, nv and right-hand sides per operator."""
    gen = torch.Generator().manual_seed(case["recipe"])
    pick = lambda top: int(torch.randint(top, (1,), generator=gen))  # noqa: E731
    return [((4, 6, 8)[pick(3)], (8, 16, 24)[pick(3)], 1 + pick(12)) for _ in range(case["count"])]


def _batched_params():
    return cg.solve_params(m=50, max_restarts=100, tol=1e-10, poly_degree=4, defl_k=16, recycle_updates=10,
                           precision=cg.PREC_FP32, inner_tol=1e-5, max_ir=20,
                           flags=cg.COARSE_ZERO_GUESS | cg.COARSE_POLY_BF16 | cg.COARSE_ODD_EVEN)


def prepare(case, seed):
    gen, kind = _generator(seed), case["kind"]
    if kind == "batched":
        ops, bs, xs = [], [], []
        for ext, nv, nrhs in _recipe(case):
            dims = (ext,) * 4
            a, f = _blocks(gen, dims, nv)
            ops.append(cg.CoarseOp(a, f, dims, nv, precisions=(cg.PREC_FP32, cg.PREC_BF16), max_nrhs=12,
                                   assume_gamma5=True))
            x = _gauss(gen, math.prod(dims), 2 * nv, nrhs)
            bs.append(_columns(_apply64(a, f, dims, x, 0.0)))
            xs.append(torch.zeros_like(bs[-1]))
        p = _batched_params()
        cg.solve_batched(ops, bs, xs, p)  # builds the polynomials and recycle spaces the operators then hold
        return {"kind": kind, "ops": ops, "bs": bs, "xs": xs, "params": p}
    dims, n = _dims(case), 2 * case["nv"]
    V = math.prod(dims)
    a, f = _blocks(gen, dims, case["nv"])
    if kind == "apply":
        prec = PREC[case["prec"]]
        op = _operator(a, f, dims, case, (prec,), max_nrhs=case["nrhs"])
        x = _columns(_gauss(gen, V, n, case["nrhs"]))
        x = x if case["prec"] == "fp64" else x.to(torch.complex64)
        return {"kind": kind, "op": op, "x": x, "prec": prec, "adjoint": case["adjoint"]}
    if kind == "schur":
        prec = PREC[case["prec"]]
        op = _operator(a, f, dims, case, (prec,))
        x = _gauss(gen, V // 2 * n).to(torch.complex64)
        op.schur(x, precision=prec)  # computes the diagonal blocks' inverses, which the operator keeps
        return {"kind": kind, "op": op, "x": x, "prec": prec}
    if kind == "residual":
        op = _operator(a, f, dims, case, ())
        return {"kind": kind, "op": op, "b": _gauss(gen, V * n), "x": _gauss(gen, V * n)}
    x = _gauss(gen, V, n, 1)
    b = _columns(_apply64(a, f, dims, x, case["mu"]))
    if kind == "solve":
        op = _operator(a, f, dims, case, (cg.PREC_FP32, cg.PREC_BF16))
        del a, f
        _setup_solves(op, case, gen, V * n)
        return {"kind": kind, "op": op, "b": b, "params": _solve_params(case)}
    c = _columns(_adjoint64(a, f, dims, _gauss(gen, V, n, 1), case["mu"]))
    op = _operator(a, f, dims, case, (cg.PREC_FP32, cg.PREC_BF16))
    _setup_solves(op, case, gen, V * n)
    if case["mu"]:
        _setup_solves(op, case, gen, V * n, adjoint=True)
    return {"kind": kind, "op": op, "b": b.requires_grad_(), "c": c, "self": a.requires_grad_(),
            "hops": _canonical_hops(f, dims).requires_grad_(), "params": _solve_params(case)}


def run(state):
    kind = state["kind"]
    if kind == "apply":
        return state["op"].apply(state["x"], precision=state["prec"], adjoint=state["adjoint"])
    if kind == "schur":
        return state["op"].schur(state["x"], precision=state["prec"])
    if kind == "residual":
        return state["op"].residual(state["b"], state["x"])
    if kind == "solve":
        return state["op"].solve(state["b"], params=state["params"])[0]
    if kind == "batched":
        cg.solve_batched(state["ops"], state["bs"], state["xs"], state["params"])
        return state["xs"]
    x = cg.CoarseSolve.apply(state["b"], state["self"], state["hops"], state["op"], state["params"])
    return [x, *torch.autograd.grad(x, (state["b"], state["self"], state["hops"]), state["c"])]


# ------------------------------------------------------------------------------ least work and 64 bits
def work(case):
    """Bytes: every stored block and vector once per pass.  Flops: one complex multiply-add is eight."""
    kind = case["kind"]
    if kind == "batched":
        nb = fl = 0.0
        for ext, nv, nrhs in _recipe(case):
            V, n = ext ** 4, 2 * nv
            nb += 5 * n * n * V * (16 + 8 + 4) + 2 * 16 * n * V * nrhs
            fl += 72.0 * n * n * V * nrhs
        return {"bytes": nb, "flops": fl}
    n, V = 2 * case["nv"], math.prod(_dims(case))
    if kind == "apply":
        p, r = case["prec"], case["nrhs"]
        return {"bytes": 5 * n * n * V * ENTRY_BYTES[p] + 2 * r * n * V * VEC_BYTES[p], "flops": 72.0 * n * n * V * r}
    if kind == "schur":
        # five blocks per site (the diagonal one as its inverse), half-length vectors
        return {"bytes": 5 * n * n * V * ENTRY_BYTES[case["prec"]] + n * V * 8, "flops": 72.0 * n * n * V}
    if kind == "residual":
        return {"bytes": 5 * n * n * V * 16 + 3 * n * V * 16, "flops": 72.0 * n * n * V}
    blocks = 5 * n * n * V * (16 + 8 + 4)
    if kind == "solve":
        return {"bytes": blocks + 2 * n * V * 16, "flops": 72.0 * n * n * V}
    return {"bytes": blocks + 9 * n * n * V * 16 + 5 * n * V * 16, "flops": 3 * 72.0 * n * n * V}


def exact(case, seed):
    gen, kind = _generator(seed), case["kind"]
    if kind == "batched":
        out = []
        for ext, nv, nrhs in _recipe(case):
            _blocks(gen, (ext,) * 4, nv)
            out.append(_columns(_gauss(gen, ext ** 4, 2 * nv, nrhs)))
        return out
    dims, n = _dims(case), 2 * case["nv"]
    V = math.prod(dims)
    a, f = _blocks(gen, dims, case["nv"])
    if kind == "apply":
        x = _columns(_gauss(gen, V, n, case["nrhs"]))
        x = x if case["prec"] == "fp64" else x.to(torch.complex64).to(torch.complex128)
        op64 = _adjoint64 if case["adjoint"] else _apply64
        return _columns(op64(a, f, dims, _sites(x, n), case["mu"]))
    if kind == "schur":
        v = _gauss(gen, V // 2 * n).to(torch.complex64).to(torch.complex128).reshape(-1, n, 1)
        even = _even_sites(dims)
        d = a + torch.diag(1j * case["mu"] * _sigma3(n))
        x = torch.zeros(V, n, 1, dtype=torch.complex128, device="cuda")
        x[even] = v
        t = torch.linalg.solve(d, _hops64(f, dims, x))
        t[even] = 0.0
        return (v - torch.linalg.solve(d, _hops64(f, dims, t))[even]).reshape(-1)
    if kind == "residual":
        b, x = _gauss(gen, V * n), _gauss(gen, V * n)
        r = b - _apply64(a, f, dims, x.reshape(V, n, 1), case["mu"]).reshape(-1)
        return r, float(torch.linalg.vector_norm(r)), float(torch.linalg.vector_norm(b))
    x = _gauss(gen, V, n, 1)
    if kind == "solve":
        return _columns(x)
    lam = _gauss(gen, V, n, 1)
    out = [_columns(x), _columns(lam), -lam @ x.mH, torch.empty(V, 8, n, n, dtype=x.dtype, device=x.device)]
    for mu in range(4):
        out[3][:, mu] = -lam @ _roll(x, dims, mu, -1).mH
        out[3][:, 4 + mu] = -lam @ _roll(x, dims, mu, 1).mH
    return out
