"""Products with A over the tile heights and last tiles that the sizes select,
with one and two rows per thread, every ring depth and the half-stored stencil,
against the same sums formed from the copied-out stencil.

Tolerance: (2p+1)^d terms summed in another order, at most that many units of
2^-53 of sum |a_ij| |x_j|.
"""
import numpy as np
import pytest

import synth
from gpu_util import need_gpu, to_dev

pytestmark = pytest.mark.gpu


def reference(S, x, n, p):
    """y and sum |a||x| from S[o][row] on the box n (direction 1 first)."""
    import torch
    d, W = len(n), 2 * p + 1
    shape = list(n[::-1])
    pad = torch.zeros([v + 2 * p for v in shape], dtype=torch.float64, device=x.device)
    pad[tuple(slice(p, p + v) for v in shape)] = x.reshape(shape)
    y = torch.zeros(shape, dtype=torch.float64, device=x.device)
    size = torch.zeros_like(y)
    for o in range(W ** d):
        at = [(o // W ** k) % W for k in range(d)][::-1]            # slowest direction first
        t = S[o].reshape(shape) * pad[tuple(slice(a, a + v) for a, v in zip(at, shape))]
        y += t
        size += t.abs()
    return y.reshape(-1), size.reshape(-1)


# from one tile to several rounds of 256-row tiles, lengths that leave short last tiles
@pytest.mark.parametrize("n,p", [((3, 5, 4), 2), ((11, 13, 17), 2), ((20, 20, 20), 3), ((29, 31, 37), 2),
                                 ((33, 40, 29), 1), ((47, 53, 41), 3), ((61, 30, 47), 4), ((70, 67, 59), 2),
                                 ((23, 19, 31), 5), ((101, 97), 3), ((257, 130), 2)])
def test_tiles(n, p):
    torch = need_gpu()
    from paper_1602_01636_gb300 import igafd
    d = len(n)
    prob = synth.Problem(d, n, p, [0.03, -0.02, 0.015] if d == 3 else None)
    x = to_dev(np.random.default_rng(1).standard_normal(int(np.prod(n))))
    for half in (False, True):
        patch = igafd.Patch(prob.knots, p, prob.ctrl, half_stencil=half)
        S = patch.stencil()
        y, size = reference(S, x, n, p)
        bound = size * ((2 * p + 1) ** d * 2.0 ** -53)
        assert bool(((patch.apply_A(x) - y).abs() <= bound).all())     # the defaults
        for rows in (1, 2) if d == 3 else (1,):
            patch.set_stencil_rows(rows)
            for stages in (4,) if half else (3, 4, 6):
                patch.set_stencil_stages(stages)
                assert bool(((patch.apply_A(x) - y).abs() <= bound).all()), (half, rows, stages)
        patch.close()
