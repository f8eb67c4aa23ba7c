"""FP64 stencil on digits, row by row: inputs whose products are far below their block's and their site's largest
entries, products near the lower end of the FP64 range, and the exactness of well-scaled sums.

Tolerances.  Every entry keeps the FP64 bound of the other stencil tests (gpu_helpers.stencil_factor) whatever
the sizes of the entries.  Results near the range's end may also be off by the smallest subnormal per product.
On Gaussian data the digits leave one rounding per block sum and the additions of the nine blocks, about
sqrt(1 + (2 + .. + 9) / 9) / sqrt(3) = 1.4 units of 2^-53 relative to |y| in the mean square: at most 4 units are
allowed, where a lost digit level (256^-7 of the product of the largest entries) costs about 30.
"""
import numpy as np
import pytest
import torch

from gpu_helpers import U64, abs_apply, assert_entrywise, stencil_factor
from oracle import coarse as ocoarse
from oracle.lattice import neighbours
from test_gpu_digits import blocks, canonical, check, columns, device_op

pytestmark = pytest.mark.gpu

# the pull kernel, two columns in one pass, the push kernel (from 1024 sites on)
LAYOUTS = [((3, 2, 2, 2), 1), ((2, 3, 2, 2), 2), ((4, 4, 8, 8), 1)]


@pytest.mark.parametrize("dims,cols", LAYOUTS)
@pytest.mark.parametrize("nv", [8, 16, 24])
@pytest.mark.parametrize("k", [12, 20, 30, 40, 70])
def test_operator_column(dims, cols, nv, k):
    """One column of the operator: an entry 2^-k below its block's diagonal, alone with x's only entry."""
    V, n = int(np.prod(dims)), 2 * nv
    s, f = blocks(dims, nv, 71)
    s[:] = 2.5 * np.eye(n)
    s[3, 0, 1], s[3, 1, 0] = (1.0 + 1.0 / 3.0) * 2.0 ** -k, (1.0 + 1.0 / 3.0) * 2.0 ** -k
    f[:] = 0.0
    X = np.zeros((cols, V * n), dtype=complex)
    X[:, 3 * n + 1] = 0.7 - 0.2j
    for adjoint in (False, True):
        check(s, f, dims, nv, 0.0, X, adjoint, f"column k={k} nv={nv}")


@pytest.mark.parametrize("dims,cols", LAYOUTS)
@pytest.mark.parametrize("nv", [8, 16, 24])
def test_diagonal_blocks_and_graded_vector(dims, cols, nv):
    """Diagonal self and hop blocks, site vectors graded over 75 binary orders inside each chirality half."""
    n = 2 * nv
    s, f = blocks(dims, nv, 72)
    V = s.shape[0]
    s[:] = 2.7 * np.eye(n)
    f *= np.where(np.arange(V)[:, None, None, None] % 2, np.eye(n), 0.0)
    X = columns(cols, V * n, 73)
    X *= np.tile(np.exp2(-75.0 * (np.arange(n) % nv) / (nv - 1)), V)
    for adjoint in (False, True):
        check(s, f, dims, nv, 0.01, X, adjoint, f"graded nv={nv}")


@pytest.mark.parametrize("dims,cols", LAYOUTS)
@pytest.mark.parametrize("orders", [(-500, -505), (-500, -540), (-300, -700), (470, 480)])
def test_products_near_the_range_ends(dims, cols, orders):
    nv = 8
    s, f = blocks(dims, nv, 74)
    V, n = s.shape[0], 2 * nv
    X = columns(cols, V * n, 75) * 2.0 ** orders[1]
    s *= 2.0 ** orders[0]
    f *= 2.0 ** orders[0]
    dev = device_op(s, f, dims, nv, 0.0, cols)
    y = dev.apply(torch.from_numpy(X).cuda(), precision=0).cpu().numpy()
    dev.close()
    # the oracle at an ordinary scale, scaled back (exact but for subnormal results)
    h = canonical(f, dims) * 2.0 ** -orders[0]
    for c in range(cols):
        x = X[c] * 2.0 ** -orders[1]
        ref = ocoarse.apply(s * 2.0 ** -orders[0], h, dims, x, 0.0)
        bound = stencil_factor(0, n) * abs_apply(s * 2.0 ** -orders[0], h, dims, x, 0.0)
        back = 2.0 ** (sum(orders) / 2)
        yb = y[c] / back
        assert_entrywise(yb, ref * back, bound * back + (9 * n + 5) * 4 * 2.0 ** -1074 / back, f"{orders} column {c}")


@pytest.mark.parametrize("dims,cols", LAYOUTS)
@pytest.mark.parametrize("nv", [8, 16, 24])
def test_well_scaled_sums_are_nearly_exact(dims, cols, nv):
    s, f = blocks(dims, nv, 76)
    V, n = s.shape[0], 2 * nv
    X = columns(cols, V * n, 77)
    dev = device_op(s, f, dims, nv, 0.0, cols)
    y = dev.apply(torch.from_numpy(X).cuda(), precision=0).cpu().numpy()
    dev.close()
    # 64 bits or more of mantissa, on sites spread over the lattice
    sites = np.unique(np.linspace(0, V - 1, 40).astype(int))
    h, nb = canonical(f, dims), neighbours(dims)
    for c in range(cols):
        x = X[c].reshape(V, n).astype(np.clongdouble)
        got = y[c].reshape(V, n)[sites]
        ref = np.empty((len(sites), n), dtype=np.clongdouble)
        for i, q in enumerate(sites):
            ref[i] = (s[q].astype(np.clongdouble) * x[q]).sum(1)
            for d in range(8):
                ref[i] += (h[q, d].astype(np.clongdouble) * x[nb[q, d]]).sum(1)
        err = np.sqrt((np.abs(got - ref) ** 2).sum() / (np.abs(ref) ** 2).sum())
        assert err <= 4 * U64, f"nv={nv} column {c}: {float(err / U64)} units"
