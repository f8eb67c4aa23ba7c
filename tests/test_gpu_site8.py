"""The layout of eight warps per site (csrc/site8.cuh), fixed through the autotuner: the full stencil (candidate 2)
and the odd-even half apply (candidate 7) against the oracle, entry by entry, on 16-byte aligned and on 8-byte
aligned vectors.

Tolerances: the bounds of the other stencil and reduced-system tests (gpu_helpers.stencil_factor, schur_factor).
"""
import numpy as np
import pytest
import torch

from gpu_helpers import abs_apply, assert_entrywise, bf16_operator, check_schur_entrywise, stencil_factor
from oracle import coarse as ocoarse
from test_gpu_digits import blocks, canonical, columns
from test_gpu_eo_configs import CASES, _run
from test_gpu_mcol import operator

pytestmark = pytest.mark.gpu

SIZES = [((2, 3, 2, 2), 8), ((2, 2, 2, 5), 16), ((4, 2, 2, 2), 24)]


class fixed:
    """The autotuner's decisions for FP32 and BF16 blocks of one lattice size, forgotten afterwards."""

    def __init__(self, family, n, V, choice):
        self.keys = [f"{family}/p{p}/n{n}/v{V.bit_length() - 1}" for p in (0, 1, 2)]
        self.choice = choice

    def __enter__(self):
        from paper_2205_09104_gb300 import autotune_set
        for k in self.keys:
            autotune_set(k, self.choice)

    def __exit__(self, *exc):
        from paper_2205_09104_gb300 import autotune_set
        for k in self.keys:
            autotune_set(k, -1)


def unaligned(x):
    """x in memory that is 8-byte aligned only."""
    y = torch.empty(x.numel() + 1, dtype=x.dtype, device="cuda")[1:].reshape(x.shape)
    return y.copy_(x)


@pytest.mark.parametrize("dims,nv", SIZES)
@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("adjoint", [False, True])
def test_stencil(dims, nv, prec, adjoint):
    s, f = blocks(dims, nv, 61)
    V, n = s.shape[0], 2 * nv
    x = columns(1, V * n, 62)[0]
    dev = operator(s, f, dims, nv, 0.02, 1)
    xd = torch.from_numpy(x).cuda().to(torch.complex64)
    with fixed("apply", n, V, 2):
        y = dev.apply(xd, precision=prec, adjoint=adjoint).cpu().numpy()
        y8 = dev.apply(unaligned(xd), precision=prec, adjoint=adjoint).cpu().numpy()
    dev.close()
    h = canonical(f, dims)
    ref_of = ocoarse.apply_adjoint if adjoint else ocoarse.apply
    if prec == 2:
        s, h = bf16_operator(s, h, dims)
    x32 = xd.cpu().numpy().astype(np.complex128)
    ref = ref_of(s, h, dims, x32, 0.02)
    bound = stencil_factor(prec, n, rounded_operands=prec == 2) * abs_apply(s, h, dims, x32, 0.02, adjoint=adjoint)
    assert_entrywise(y, ref, bound, f"prec {prec}")
    assert_entrywise(y8, ref, bound, f"prec {prec}, unaligned")


@pytest.mark.parametrize("dims,nv", [((2, 4, 2, 2), 8), ((2, 2, 2, 6), 16), ((4, 2, 2, 2), 24)])
def test_half_apply_vectors_8_byte_aligned(dims, nv):
    s, f = blocks(dims, nv, 63)
    V, n = s.shape[0], 2 * nv
    x = columns(1, V * n // 2, 64)[0]
    h = canonical(f, dims)
    dev = operator(s, f, dims, nv, 0.02, 1)
    with fixed("eo", n, V, 7):
        for prec in (0, 1, 2):
            xd = torch.from_numpy(x).cuda().to(torch.complex128 if prec == 0 else torch.complex64)
            for v in (xd, unaligned(xd)):
                y = dev.schur(v, precision=prec).cpu().numpy()
                check_schur_entrywise(y, xd.cpu().numpy(), s, h, dims, prec, 0.02, f"aligned to {v.data_ptr() % 16}")
    dev.close()


@pytest.mark.parametrize("nv,fdims,mu", CASES)
def test_half_apply_and_solves(tmp_path, nv, fdims, mu):
    _run(tmp_path, 7, nv, fdims, mu)
