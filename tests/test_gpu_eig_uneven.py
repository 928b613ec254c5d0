"""Eigendecompositions of pencils with n_k > 128 on uneven, graded and repeated
knots and with span scalings: the oracle's invariants whichever route is taken
(tolerances of the other eigen tests), and no set-up slower than the FP64
Jacobi alone where the refinement would not hold."""
import time

import numpy as np
import pytest

import synth
from oracle import assemble, learned
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def knots(kind, n, p):
    """Knots with n interior functions."""
    mult = np.ones(n - p + 1, int)
    if kind == "repeated":                     # C^0 at every knot
        mult = np.full((n - p + 1) // p, p)
        mult = np.concatenate([mult, np.ones(n - p + 1 - mult.sum(), int)])
    x = np.linspace(0.0, 1.0, len(mult) + 2)
    if kind == "graded":                       # spans from 1 to 10^3
        x = np.sinh(8.0 * x) / np.sinh(8.0)
    elif kind == "uneven":
        w = np.random.default_rng(8).uniform(0.1, 1.0, len(x) - 1)
        x = np.concatenate([[0.0], np.cumsum(w) / w.sum()])
        x[-1] = 1.0
    return np.concatenate([np.zeros(p + 1), np.repeat(x[1:-1], mult), np.ones(p + 1)])


def patch_of(kinds, n, p):
    from paper_1602_01636_gb300 import igafd
    kn = [knots(kind, v, p) for kind, v in zip(kinds, n)]
    ctrl = synth.control_net(kn, p)
    disc = assemble.Discretization(kn, p, assemble.Geometry(ctrl, kn, p))
    return igafd.Patch(kn, p, ctrl, stencil=False), disc


def check(patch, pencils):
    for k, (K, M) in enumerate(pencils):
        D, U = patch.eigen(k)
        assert np.all(np.diff(D) >= 0)
        assert np.abs(U.T @ M @ U - np.eye(len(D))).max() <= 1e-12
        assert np.abs(U.T @ K @ U - np.diag(D)).max() <= 1e-12 * D.max()


@pytest.mark.parametrize("kinds,n,p,refined", [
    (("graded", "uneven"), (150, 140), 2, (0, None)), (("graded", "graded"), (257, 130), 1, (0, 0)),
    (("repeated", "uneven"), (150, 161), 2, (1, None)), (("uniform", "graded"), (640, 40), 2, (None, None))])
def test_uneven_knots(kinds, n, p, refined):
    need_gpu()
    patch, disc = patch_of(kinds, n, p)
    for k, want in enumerate(refined):
        assert want is None or patch.info.eig_refined[k] == want
    check(patch, [disc.pencil(k) for k in range(2)])
    patch.close()


def test_scaled_pencils():
    torch = need_gpu()
    patch, disc = patch_of(("uniform", "uneven"), (150, 200), 2)
    logw = np.random.default_rng(9).standard_normal((patch.scaling_rows(), 2)).astype(np.float32)
    patch.set_scalings(torch.from_numpy(logw).cuda())
    check(patch, learned.scaled_pencils(disc, logw.astype(np.float64)))
    patch.close()


def test_graded_set_up_not_slower_than_jacobi():
    torch = need_gpu()
    patch, _ = patch_of(("graded", "uniform"), (300, 8), 2)

    def best(route):
        patch.set_eig_route(route)
        t = []
        for _ in range(3):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            patch.setup_prec()
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        return min(t)

    assert best(0) <= 1.15 * best(1)
    patch.close()
