"""FP64 stencil through exact digit products (csrc/digits.cu) against the oracle, entry by entry.

Tolerance: the FP64 bound of the other stencil tests, (K + 4) 2^-53 of sum_j |a_ij| |x_j| with K = 9n + 1
(gpu_helpers.stencil_factor).  The digit products stay far inside it: two conversions to 62 bits below the
largest entry of a block / site vector and dropped levels of the same size, while the sites for which
that is not enough (entries of very different size, scales near the FP64 range's ends, non-finite
values) are summed on the FP64 pipe.
"""
import numpy as np
import pytest
import torch

from gpu_helpers import abs_apply, assert_entrywise, stencil_factor
from oracle import coarse as ocoarse
from oracle.lattice import neighbours

pytestmark = pytest.mark.gpu


def blocks(dims, nv, seed):
    """Random sigma3-Hermitian self blocks and forward hops with their backward hops, [V, n, n], [V, 8, n, n]."""
    rng = np.random.default_rng(seed)
    V, n = int(np.prod(dims)), 2 * nv
    g = rng.standard_normal((V, n, n)) + 1j * rng.standard_normal((V, n, n))
    f = rng.standard_normal((V, 4, n, n)) + 1j * rng.standard_normal((V, 4, n, n))
    s3 = np.repeat([1.0, -1.0], nv)
    return 0.1 * (g + s3[:, None] * g.conj().transpose(0, 2, 1) * s3) + 2.5 * np.eye(n), 0.1 * f


def canonical(f, dims):
    n = f.shape[-1]
    s3 = np.repeat([1.0, -1.0], n // 2)
    nb = neighbours(dims)
    h = np.empty((f.shape[0], 8, n, n), dtype=complex)
    h[:, :4] = f
    for mu in range(4):
        h[:, 4 + mu] = s3[:, None] * f[nb[:, 4 + mu], mu].conj().transpose(0, 2, 1) * s3
    return h


def device_op(s, f, dims, nv, mu, cols):
    from paper_2205_09104_gb300 import CoarseOp
    return CoarseOp(torch.from_numpy(s).cuda(), torch.from_numpy(np.ascontiguousarray(f)).cuda(), dims, nv, mu=mu,
                    precisions=(), max_nrhs=cols, assume_gamma5=True)


def check(s, f, dims, nv, mu, X, adjoint, what):
    dev = device_op(s, f, dims, nv, mu, X.shape[0])
    y = dev.apply(torch.from_numpy(X).cuda(), precision=0, adjoint=adjoint).cpu().numpy()
    h = canonical(f, dims)
    ref_of = ocoarse.apply_adjoint if adjoint else ocoarse.apply
    for c in range(X.shape[0]):
        ref = ref_of(s, h, dims, X[c], mu)
        bound = stencil_factor(0, 2 * nv) * abs_apply(s, h, dims, X[c], mu, adjoint=adjoint)
        assert_entrywise(y[c], ref, bound, f"{what} column {c}")
    dev.close()


def columns(cols, N, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((cols, N)) + 1j * rng.standard_normal((cols, N))


@pytest.mark.parametrize("dims,nv,cols", [((2, 2, 2, 2), 8, 1), ((3, 2, 5, 2), 8, 4), ((2, 3, 2, 4), 16, 1),
                                          ((5, 2, 2, 3), 16, 3), ((2, 2, 3, 2), 24, 1), ((3, 3, 2, 2), 24, 5),
                                          # from 1024 sites on one column takes the kernel that reads a block once
                                          ((4, 4, 8, 8), 8, 1), ((7, 5, 6, 5), 16, 1), ((3, 7, 7, 7), 24, 1)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_digit_products_match_oracle(dims, nv, cols, adjoint):
    s, f = blocks(dims, nv, 11)
    X = columns(cols, s.shape[0] * 2 * nv, 12)
    X[-1] *= np.repeat(np.exp2(np.arange(s.shape[0]) % 40 - 20.0), 2 * nv)  # sites of very different size
    check(s, f, dims, nv, 0.02, X, adjoint, f"dims={dims} nv={nv}")


@pytest.mark.parametrize("nv", [8, 16, 24])
@pytest.mark.parametrize("what", ["equal", "zeros", "halves", "row", "column", "tiny", "huge"])
def test_digit_products_hard_values(nv, what):
    dims = (3, 2, 2, 2)
    s, f = blocks(dims, nv, 21)
    V, n = s.shape[0], 2 * nv
    X = columns(2, V * n, 22)
    x = X[0].reshape(V, n)
    if what == "equal":       # every digit of a block and of a vector the same: the largest level sums
        f[:] = -(0.5 + 0.5 / 255) * (1 + 1j)
        X[:] = (0.5 - 0.5 / 255) * (1 - 1j)
    elif what == "zeros":
        f[1, 2] = 0.0
        x[3] = 0.0
        x[5, nv:] = 0.0
    elif what == "halves":    # one chirality far below the other
        x[2, :nv] *= 2.0 ** -40
        f[2] *= np.where((np.arange(n) < nv)[:, None] == (np.arange(n) < nv), 1.0, 0.0)
    elif what == "row":
        f[4, 1, 3] *= 2.0 ** -30
    elif what == "column":
        f[4, 1, :, 5] *= 2.0 ** -30
    elif what == "tiny":
        X *= 2.0 ** -960
    elif what == "huge":
        f[0, 3] *= 2.0 ** 950
    check(s, f, dims, nv, 0.0, X, False, f"{what} nv={nv}")


@pytest.mark.parametrize("adjoint", [False, True])
def test_digit_products_hard_values_push(adjoint):
    """The hard values above on a lattice of the push kernel."""
    dims, nv = (5, 6, 7, 5), 8
    s, f = blocks(dims, nv, 25)
    V, n = s.shape[0], 2 * nv
    X = columns(1, V * n, 26)
    x = X[0].reshape(V, n)
    f[7, 2] = 0.0
    x[3] = 0.0
    x[5, nv:] = 0.0
    x[20, :nv] *= 2.0 ** -40
    f[40, 1, 3] *= 2.0 ** -30
    f[60, 3, :, 5] *= 2.0 ** -30
    x[100] *= 2.0 ** -980
    f[200, 0] *= 2.0 ** 930
    check(s, f, dims, nv, 0.02, X, adjoint, "push, hard values")


@pytest.mark.parametrize("dims", [(4, 2, 4, 2), (5, 6, 7, 5)])
def test_digit_products_non_finite(dims):
    nv = 8
    s, f = blocks(dims, nv, 31)
    V, n = s.shape[0], 2 * nv
    X = columns(3, V * n, 32)
    X[0].reshape(V, n)[5, 3] = np.inf
    X[1].reshape(V, n)[0, 9] = np.nan
    dev = device_op(s, f, dims, nv, 0.0, 3)
    if V < 1024:
        y = dev.apply(torch.from_numpy(X).cuda(), precision=0).cpu().numpy().reshape(3, V, n)
    else:
        y = np.stack([dev.apply(torch.from_numpy(x).cuda(), precision=0).cpu().numpy().reshape(V, n) for x in X])
    nb = neighbours(dims)
    for c, site in ((0, 5), (1, 0)):
        hit = np.zeros(V, dtype=bool)
        hit[[site, *nb[site]]] = True
        assert not np.isfinite(y[c][hit]).any()
        assert np.isfinite(y[c][~hit]).all()
    assert np.isfinite(y[2]).all()
    dev.close()
