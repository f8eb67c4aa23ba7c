"""FP64 stencils with and without the digit copy of the blocks: which way an operator goes, and every FP64 entry point
on the FP64 pipe (fp64_pipe=True) against the oracle, alone and mixed with operators on digits in one batch.

Tolerances: the FP64 bounds of the other stencil tests (gpu_helpers.stencil_factor); solves reach the true residual
they were asked for, recomputed by the oracle.
"""
import numpy as np
import pytest
import torch

from gpu_helpers import abs_apply, assert_entrywise, stencil_factor
from oracle import coarse as ocoarse
from test_gpu_digits import blocks, canonical, columns

pytestmark = pytest.mark.gpu

UNDECIDED, DIGITS, ASKED = 0, 1, 2


def operator(s, f, dims, nv, mu, cols, pipe, precisions=(1, 2)):
    from paper_2205_09104_gb300 import CoarseOp
    return CoarseOp(torch.from_numpy(s).cuda(), torch.from_numpy(np.ascontiguousarray(f)).cuda(), dims, nv, mu=mu,
                    precisions=precisions, max_nrhs=cols, assume_gamma5=True, fp64_pipe=pipe)


def check_applies(dev, s, h, dims, X, mu, what):
    n = s.shape[1]
    for adjoint in (False, True):
        y = dev.apply(torch.from_numpy(X).cuda(), precision=0, adjoint=adjoint).cpu().numpy()
        ref_of = ocoarse.apply_adjoint if adjoint else ocoarse.apply
        for c in range(X.shape[0]):
            bound = stencil_factor(0, n) * abs_apply(s, h, dims, X[c], mu, adjoint=adjoint)
            assert_entrywise(y[c], ref_of(s, h, dims, X[c], mu), bound, f"{what} adjoint={adjoint} column {c}")


@pytest.mark.parametrize("dims,nv", [((2, 3, 2, 2), 8), ((2, 2, 2, 5), 16), ((4, 2, 2, 2), 24), ((4, 4, 8, 8), 8)])
@pytest.mark.parametrize("pipe", [False, True])
def test_apply_update_residual(dims, nv, pipe):
    s, f = blocks(dims, nv, 91)
    V, n = s.shape[0], 2 * nv
    X = columns(3, V * n, 92)
    dev = operator(s, f, dims, nv, 0.02, 3, pipe)
    dev.apply(torch.from_numpy(X[0]).cuda().to(torch.complex64), precision=1)
    dev.apply(torch.from_numpy(X).cuda().to(torch.complex64), precision=2)
    assert dev.fp64_path() == (ASKED if pipe else UNDECIDED)
    check_applies(dev, s, canonical(f, dims), dims, X[:1], 0.02, "one column")
    check_applies(dev, s, canonical(f, dims), dims, X, 0.02, "columns")
    assert dev.fp64_path() == (ASKED if pipe else DIGITS)
    s, f = blocks(dims, nv, 93)
    h = canonical(f, dims)
    dev.update(torch.from_numpy(s).cuda(), torch.from_numpy(h).cuda())
    check_applies(dev, s, h, dims, X[:1], 0.02, "updated")
    r, rn, bn = dev.residual(torch.from_numpy(X[1]).cuda(), torch.from_numpy(X[0]).cuda())
    ref = X[1] - ocoarse.apply(s, h, dims, X[0], 0.02)
    assert_entrywise(r.cpu().numpy(), ref, stencil_factor(0, n) * (abs_apply(s, h, dims, X[0], 0.02) + np.abs(X[1])),
                     "residual")
    assert abs(rn - np.linalg.norm(ref)) <= 1e-12 * rn and abs(bn - np.linalg.norm(X[1])) <= 1e-12 * bn
    dev.close()


@pytest.mark.parametrize("pipe", [False, True])
def test_captured_stencil_follows_updates(pipe):
    """A graph captured before the copy exists, and one captured after it, replayed on changed blocks."""
    dims, nv = (2, 3, 2, 2), 8
    s, f = blocks(dims, nv, 94)
    V, n = s.shape[0], 2 * nv
    x = torch.from_numpy(columns(1, V * n, 95)[0]).cuda()
    dev = operator(s, f, dims, nv, 0.0, 1, pipe)
    y = [torch.empty_like(x), torch.empty_like(x)]
    graphs = []
    for i in range(2):
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g):
            dev.apply(x, precision=0, out=y[i])
        assert dev.fp64_path() == (ASKED if pipe else (UNDECIDED if i == 0 else DIGITS))
        dev.apply(x, precision=0)
        graphs.append(g)
    s, f = blocks(dims, nv, 96)
    h = canonical(f, dims)
    dev.update(torch.from_numpy(s).cuda(), torch.from_numpy(h).cuda())
    ref = ocoarse.apply(s, h, dims, x.cpu().numpy(), 0.0)
    bound = stencil_factor(0, n) * abs_apply(s, h, dims, x.cpu().numpy(), 0.0)
    for i, g in enumerate(graphs):
        g.replay()
        torch.cuda.synchronize()
        assert_entrywise(y[i].cpu().numpy(), ref, bound, f"graph {i}")
    dev.close()


@pytest.mark.parametrize("prec,flags", [(0, 0), (1, 0), (1, 0x10 | 0x20), (2, 0)])
def test_solve_on_the_pipe(prec, flags):
    import paper_2205_09104_gb300 as cg
    dims, nv = (2, 4, 2, 2), 16
    s, f = blocks(dims, nv, 97)
    f *= 0.35
    h = canonical(f, dims)
    B = columns(2, s.shape[0] * 2 * nv, 98)
    p = cg.solve_params(m=30, tol=1e-10, poly_degree=3, defl_k=4, precision=prec, inner_tol=1e-2 if prec == 2 else 1e-5,
                        flags=cg.COARSE_ZERO_GUESS | flags)
    dev = operator(s, f, dims, nv, 0.01, 2, True)
    for adjoint in (False, True):
        x = dev.solve(torch.from_numpy(B).cuda(), params=p, adjoint=adjoint)[0].cpu().numpy()
        of = ocoarse.apply_adjoint if adjoint else ocoarse.apply
        for c in range(2):
            assert np.linalg.norm(B[c] - of(s, h, dims, x[c], 0.01)) <= 1.001e-10 * np.linalg.norm(B[c])
    assert dev.fp64_path() == ASKED
    dev.close()


@pytest.mark.parametrize("pipes", ["1", "101", "010", "0110"])
def test_batch_of_both_kinds(pipes):
    """Operators of one n with and without the copy, uneven columns, from a non-zero guess."""
    import paper_2205_09104_gb300 as cg
    p = cg.solve_params(m=30, tol=1e-10, poly_degree=3, defl_k=0, precision=cg.PREC_FP32, inner_tol=1e-5, flags=0)
    ops, bs, xs, ref = [], [], [], []
    for i, c in enumerate(pipes):
        dims, nv, cols = [((2, 4, 2, 2), 16, 3), ((2, 2, 2, 4), 16, 1), ((2, 2, 2, 2), 16, 4), ((4, 2, 2, 2), 8, 2)][i]
        s, f = blocks(dims, nv, 101 + i)
        f *= 0.35
        B = columns(cols, s.shape[0] * 2 * nv, 111 + i)
        ops.append(operator(s, f, dims, nv, 0.01, 1, c == "1"))
        bs.append(torch.from_numpy(B).cuda())
        xs.append(torch.from_numpy(0.1 * columns(cols, B.shape[1], 121 + i)).cuda())
        ref.append((s, canonical(f, dims), dims, B))
    cg.solve_batched(ops, bs, xs, p)
    for op, c, x, (s, h, dims, B) in zip(ops, pipes, xs, ref):
        assert op.fp64_path() == (ASKED if c == "1" else DIGITS)
        for q in range(B.shape[0]):
            r = B[q] - ocoarse.apply(s, h, dims, x[q].cpu().numpy(), 0.01)
            assert np.linalg.norm(r) <= 1.001e-10 * np.linalg.norm(B[q])
        op.close()


def test_first_use_while_another_stream_is_captured():
    """The copy is built on one stream in the middle of the capture of another."""
    dims, nv = (2, 3, 2, 2), 8
    s, f = blocks(dims, nv, 131)
    x = columns(1, s.shape[0] * 2 * nv, 132)[0]
    xd = torch.from_numpy(x).cuda()
    dev = operator(s, f, dims, nv, 0.0, 1, False)
    side = torch.cuda.Stream()
    y, a = torch.empty_like(xd), torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        a += 1
        dev.apply(xd, precision=0, stream=side, out=y)
        a += 1
    side.synchronize()
    assert dev.fp64_path() == DIGITS
    g.replay()
    torch.cuda.synchronize()
    assert (a == 2).all()
    h = canonical(f, dims)
    assert_entrywise(y.cpu().numpy(), ocoarse.apply(s, h, dims, x, 0.0), stencil_factor(0, 2 * nv) * abs_apply(s, h, dims, x),
                     "built beside a capture")
    dev.close()
