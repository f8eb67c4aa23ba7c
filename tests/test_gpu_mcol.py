"""Several columns of one operator at a time: the FP32 stencil's columns entry by entry against the oracle,
and the batched engine's column chunks against the single-operator solver.

Tolerances: the FP32 bound of the other stencil tests (gpu_helpers.stencil_factor); solves reach the true
residual they were asked for (recomputed by the oracle) in the single-operator solver's Arnoldi steps, one
more or less per cycle (the same Krylov process up to FP32 rounding).
"""
import numpy as np
import pytest
import torch

from gpu_helpers import abs_apply, assert_entrywise, stencil_factor
from oracle import coarse as ocoarse
from test_gpu_digits import blocks, canonical, columns

pytestmark = pytest.mark.gpu


def operator(s, f, dims, nv, mu, cols):
    from paper_2205_09104_gb300 import PREC_BF16, PREC_FP32, CoarseOp
    return CoarseOp(torch.from_numpy(s).cuda(), torch.from_numpy(np.ascontiguousarray(f)).cuda(), dims, nv, mu=mu,
                    precisions=(PREC_FP32, PREC_BF16), max_nrhs=cols, assume_gamma5=True)


@pytest.mark.parametrize("dims,nv,cols", [((2, 3, 2, 2), 8, 2), ((3, 2, 2, 5), 8, 13), ((2, 2, 3, 2), 16, 5),
                                          ((2, 2, 2, 3), 16, 12), ((3, 2, 2, 2), 24, 3), ((2, 2, 2, 2), 24, 25)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_fp32_columns_match_oracle(dims, nv, cols, adjoint):
    s, f = blocks(dims, nv, 41)
    h = canonical(f, dims)
    X = columns(cols, s.shape[0] * 2 * nv, 42)
    dev = operator(s, f, dims, nv, 0.02, cols)
    x = torch.from_numpy(X).cuda().to(torch.complex64)
    y = dev.apply(x, precision=1, adjoint=adjoint)
    odd = torch.empty(x.numel() + 1, dtype=x.dtype, device="cuda")[1:].reshape(x.shape)  # 8-byte aligned only
    odd.copy_(x)
    y8 = dev.apply(odd, precision=1, adjoint=adjoint).cpu().numpy()
    y = y.cpu().numpy()
    ref_of = ocoarse.apply_adjoint if adjoint else ocoarse.apply
    for c in range(cols):
        ref = ref_of(s, h, dims, X[c], 0.02)
        bound = stencil_factor(1, 2 * nv) * abs_apply(s, h, dims, X[c], 0.02, adjoint=adjoint)
        assert_entrywise(y[c], ref, bound, f"column {c}")
        assert_entrywise(y8[c], ref, bound, f"column {c}, unaligned")
    dev.close()


@pytest.mark.parametrize("flags", ["odd-even, BF16 chain", "odd-even", "full, BF16 chain", "full"])
def test_batched_chunks_match_single_solves(flags):
    import paper_2205_09104_gb300 as cg
    fl = cg.COARSE_ZERO_GUESS
    fl |= cg.COARSE_ODD_EVEN if "odd-even" in flags else 0
    fl |= cg.COARSE_POLY_BF16 if "BF16" in flags else 0
    p = cg.solve_params(m=30, tol=1e-10, poly_degree=3, defl_k=0, precision=cg.PREC_FP32, inner_tol=1e-5, flags=fl)
    ops, bs, xs, ref = [], [], [], []
    for i, (dims, nv, cols) in enumerate([((2, 4, 2, 2), 8, 13), ((2, 2, 2, 4), 16, 1), ((4, 2, 2, 2), 16, 6),
                                          ((2, 2, 2, 2), 24, 5), ((2, 2, 4, 2), 24, 12)]):
        s, f = blocks(dims, nv, 51 + i)
        f *= 0.5 if nv == 8 else 0.35
        h = canonical(f, dims)
        B = columns(cols, s.shape[0] * 2 * nv, 61 + i)
        ops.append(operator(s, f, dims, nv, 0.01, 1))
        bs.append(torch.from_numpy(B).cuda())
        xs.append(torch.zeros_like(bs[-1]))
        ref.append((s, h, dims, B))
    infos = cg.solve_batched(ops, bs, xs, p)
    at = 0
    for op, b, x, (s, h, dims, B) in zip(ops, bs, xs, ref):
        single = op.solve(b, params=p)[1]
        for c in range(b.shape[0]):
            xc = x[c].cpu().numpy()
            assert np.linalg.norm(B[c] - ocoarse.apply(s, h, dims, xc, 0.01)) <= 1.001e-10 * np.linalg.norm(B[c])
            assert abs(infos[at]["iterations"] - single[c]["iterations"]) <= single[c]["cycles"], (flags, dims, c)
            at += 1
        op.close()
