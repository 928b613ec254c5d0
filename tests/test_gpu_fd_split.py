"""The FP64 FD on the tensor cores (every n_k <= 256) against mode products in
80-bit arithmetic with the library's own U_k and D_k, so that only the
products' rounding is seen.

Tolerance: a product's error is at most about 5 x 2^-53 of its result's norm
(that of an FP64 FMA chain of 128 terms); six products and the divide, each
amplified by the condition of the factors that follow (for these spaces
cond(U_k)^2 <= 30), give 6 x 5 x 30 x 2^-53 = 1e-13.
"""
import numpy as np
import pytest

import synth
from gpu_util import need_gpu, to_dev, rel, maxrel

pytestmark = pytest.mark.gpu

# tile edges: K padded to 32 (one and two 64-wide chunks), columns to 16 and in
# blocks of 64, rows in tiles of 128, column splits of small problems
CASES = [(3, (32, 32, 32), 3), (3, (33, 31, 65), 2), (3, (64, 17, 97), 3), (3, (127, 3, 128), 1),
         (3, (2, 1, 5), 1), (3, (128, 112, 40), 3), (2, (128, 17), 3), (2, (1, 129 - 1), 2), (2, (96, 95), 4),
         # two parts (K > 128): every padded length, one and several column blocks
         (2, (129, 160), 3), (3, (150, 24, 20), 2), (2, (193, 40), 2), (2, (256, 225), 3), (3, (10, 161, 9), 3)]


def reference(patch, r):
    """P^{-1} r in extended precision from the patch's eigenpairs."""
    L = np.longdouble
    d, n = patch.dim, patch.n
    eig = [patch.eigen(k) for k in range(d)]
    x = r.astype(L).reshape(n[::-1])
    lam = L(0)
    for k, (D, U) in enumerate(eig):
        ax = d - 1 - k
        x = np.moveaxis(np.tensordot(U.astype(L).T, x, axes=([1], [ax])), 0, ax)
        lam = lam + D.astype(L).reshape([-1] + [1] * k)
    x = x / lam
    for k, (_, U) in enumerate(eig):
        ax = d - 1 - k
        x = np.moveaxis(np.tensordot(U.astype(L), x, axes=([1], [ax])), 0, ax)
    return x.reshape(-1)


@pytest.mark.parametrize("dim,n,p", CASES)
def test_split_products(dim, n, p):
    torch = need_gpu()
    from paper_1602_01636_gb300 import igafd
    patch = igafd.Patch.from_problem(synth.Problem(dim, n, p), stencil=False)
    rng = np.random.default_rng(7)
    smooth = np.ones(patch.N)
    wide = rng.standard_normal(patch.N) * 10.0 ** rng.integers(-8, 9, patch.N)
    for r in (rng.standard_normal(patch.N), smooth, wide):
        z = patch.apply_prec(to_dev(r)).cpu().numpy()
        want = reference(patch, r).astype(np.float64)
        assert rel(z, want) <= 1e-13 and maxrel(z, want) <= 1e-13
    # powers of two pass through exactly, also out to the ends of the range
    z = patch.apply_prec(to_dev(wide)).cpu().numpy()
    for e in (-900, 900):
        assert np.array_equal(patch.apply_prec(to_dev(np.ldexp(wide, e))).cpu().numpy(), np.ldexp(z, e))
    tiny = patch.apply_prec(to_dev(np.ldexp(wide, -1040))).cpu().numpy()    # subnormal entries
    assert np.abs(tiny - np.ldexp(z, -1040)).max() <= 1e-12 * np.abs(np.ldexp(z, -1040)).max() + 5e-322
    assert not patch.apply_prec(to_dev(np.zeros(patch.N))).any().item()
    for bad in (np.nan, np.inf, -np.inf):
        r = rng.standard_normal(patch.N)
        r[patch.N // 2] = bad
        assert not torch.isfinite(patch.apply_prec(to_dev(r))).any().item()
    patch.close()
