"""Eigendecompositions of pencils with n_k > 128 (the FP32 start from L2 and its
FP64 refinement): the oracle's invariants and eigenvalues, to the tolerance of
the smaller pencils' tests (the route accepts only what meets 1e-12). The
route takes degrees 1 and 2; higher ones keep the FP64 Jacobi."""
import numpy as np
import pytest

import synth
from oracle import assemble, fd
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p", [((129, 160), 2), ((150, 257), 2), ((192, 131), 1), ((256, 40), 1),
                                 ((300, 513), 2), ((129, 64), 3)])
def test_large_pencils(n, p):
    need_gpu()
    from paper_1602_01636_gb300 import igafd
    prob = synth.Problem(2, n, p)
    patch = igafd.Patch.from_problem(prob, stencil=False)
    disc = assemble.Discretization.from_problem(prob)
    assert list(patch.info.eig_refined)[:2] == [int(m <= 128 or p <= 2) for m in n]
    first = [patch.eigen(k) for k in range(2)]
    for k in range(2):
        K, M = disc.pencil(k)
        D, U = first[k]
        Do, _ = fd.generalized_eig(K, M)
        assert np.abs(D - Do).max() <= 1e-12 * Do.max()
        assert np.abs(U.T @ M @ U - np.eye(len(D))).max() <= 1e-12
        assert np.abs(U.T @ K @ U - np.diag(D)).max() <= 1e-12 * D.max()
    patch.setup_prec()                       # reproducible
    for k in range(2):
        D, U = patch.eigen(k)
        assert np.array_equal(D, first[k][0]) and np.array_equal(U, first[k][1])
    patch.close()
