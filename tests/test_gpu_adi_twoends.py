"""The FP64 ADI line solve, which eliminates a line from both ends towards a
middle block of p rows, at the line lengths where its parts vanish or are
uneven: shorter than the middle block, exactly its size, one row on one end
only, odd and even remainders, the longest line.

Tolerance: both sides solve the same systems K_k + w M_k and M_k, each with a
forward error of at most (terms per row) x 2^-53 x its condition number; the
largest is M_k's. With at most 2 p + 1 = 11 terms, three directions and two
solves per direction: 64 x 2^-53 x max_k cond(M_k) of max|z|, and not below the
1e-12 of the other ADI tests."""
import numpy as np
import pytest

import synth
from oracle import adi, assemble
from gpu_util import need_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p", [((1, 2, 33), 1), ((1, 2, 3), 2), ((2, 3, 4), 3), ((5, 6, 7), 3),
                                 ((4, 5, 6), 5), ((9, 10, 11), 5), ((256, 3, 8), 3)])
def test_line_lengths_match_oracle(n, p):
    need_gpu()
    from paper_1602_01636_gb300 import igafd
    omega = [0.7, 25.0, 3.0]
    prob = synth.Problem(3, n, p, None)
    disc = assemble.Discretization.from_problem(prob)
    pens = [disc.pencil(k) for k in range(3)]
    r = synth.random_vector(disc.N, 21)
    ref = adi.ADI3D(pens, omega=np.array(omega)).apply(r)
    patch = igafd.Patch.from_problem(prob, stencil=False)
    patch.adi_setup(omega, "fp64")
    z = patch.apply_prec_adi(to_dev(r)).cpu().numpy()
    cond = max(np.linalg.cond(pen[1]) for pen in pens)
    assert np.abs(z - ref).max() <= max(1e-12, 64 * 2.0 ** -53 * cond) * np.abs(ref).max()
