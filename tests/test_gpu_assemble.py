"""3D assembly by patch-wide sum factorisation and the load vector's row kernel
against the oracle on the spaces where their indexing can go wrong: every
degree, single elements, repeated interior knots (supports of few elements),
geometry and coefficient nets on other knots, tiles of direction 1, the full
space, and i2 taken in chunks.

Tolerance: the same quadrature sums in another order (at most (p + 1)^6 terms,
observed a few ulps of the largest), as for the other assembly tests: 1e-13.
"""
import numpy as np
import pytest

import synth
from oracle import assemble
from gpu_util import need_gpu, to_dev, rel

pytestmark = pytest.mark.gpu


def knots(p, spans):
    """Open knots over spans = [multiplicity after each span, ...], uneven spans."""
    inner, x = [], 0.0
    for i, mult in enumerate(spans[:-1]):
        x += 1.0 + 0.3 * (i % 3)
        inner += [x] * mult
    end = x + 1.0
    return np.concatenate([np.zeros(p + 1), np.array(inner) / end, np.ones(p + 1)])


CASES = [
    # p, spans per direction, geometry (degree, elements) or None (isoparametric), coefficient, full space
    (1, ([1] * 70, [1, 1, 1], [1, 1]), None, False, False),
    (2, ([1, 2, 1, 1], [2, 2, 1], [1] * 5), (1, 3), False, False),
    (3, ([1], [1, 1], [3, 1, 2, 1]), (2, 9), True, False),
    (3, ([1] * 34, [1], [1, 1, 1]), None, True, False),
    (4, ([1, 1, 4, 1], [1], [1, 1]), None, False, True),
    (5, ([1, 1], [1, 5, 1], [1]), (3, 2), False, False),
    (6, ([1, 1], [1], [1, 1, 1]), None, False, False),
]


@pytest.mark.parametrize("p,spans,geo,coef,full", CASES)
def test_assembly_and_load(p, spans, geo, coef, full):
    need_gpu()
    from paper_1602_01636_gb300 import igafd
    kn = [knots(p, s) for s in spans]
    gp, gk = (p, kn) if geo is None else (geo[0], [synth.uniform_open_knots(geo[1], geo[0])] * 3)
    ctrl = synth.control_net(gk, gp, [0.03, -0.02, 0.015])
    rng = np.random.default_rng(3)
    field = ofield = None
    if coef:
        ck = [synth.uniform_open_knots(4, 2)] * 3
        cv = np.exp(0.4 * rng.standard_normal((6, 6, 6)))
        field, ofield = (ck, 2, cv), assemble.ScalarSpline(cv, ck, 2)
    disc = assemble.Discretization(kn, p, assemble.Geometry(ctrl, gk, gp), kappa=1.3, kappa_field=ofield)
    f = lambda x, y, z: 1.0 + x * y - z
    if full:                                   # (the oracle assembles the interior space)
        patch = igafd.Patch(kn, p, ctrl, 1.3, geo_knots=gk, geo_p=gp, kappa_field=field, full_space=True)
        m = [len(k) - p - 1 for k in kn]
        keep = np.zeros(m[::-1], bool)
        keep[1:-1, 1:-1, 1:-1] = True
        S = patch.stencil().cpu().numpy()[:, keep.ravel()]
        want = disc.assemble_stencil().reshape(S.shape)
        S[want == 0.0] = 0.0                   # couplings to boundary functions
        assert np.abs(S - want).max() <= 1e-13 * np.abs(want).max()
        patch.close()
        return
    want = disc.assemble_stencil()
    want = want.reshape(want.shape[0], -1)
    J = disc.geo.eval_grid([z.ravel() for z in disc.qz])[1]
    kap = 1.3 * (ofield.eval_grid([z.ravel() for z in disc.qz]) if coef else 1.0)
    Q, det = assemble.q_matrix(J, kap)
    lam = np.linalg.eigvalsh(Q.reshape(-1, 3, 3))
    for half in (False, True):
        patch = igafd.Patch(kn, p, ctrl, 1.3, geo_knots=gk, geo_p=gp, kappa_field=field, half_stencil=half)
        S = patch.stencil().cpu().numpy()
        assert np.abs(S - want).max() <= 1e-13 * np.abs(want).max()
        assert not S[want == 0.0].any()      # outside the box, or functions without a shared element
        assert abs(patch.info.min_detJ - det.min()) <= 1e-12 * det.max()
        q = lam[:, -1].max() / lam[:, 0].min()
        assert abs(patch.info.q_bound - q) <= 1e-9 * q
        X = patch.quad_points()
        b = patch.load_rhs((1.0 + X[0] * X[1] - X[2]).contiguous()).cpu().numpy()
        bo = disc.assemble_rhs(f)
        assert np.abs(b - bo).max() <= 1e-13 * np.abs(bo).max()
        patch.close()


def test_chunks_of_direction_2():
    """A layer whose scratch is over the limit (p = 6, 665 x 665 points) is
    assembled in chunks of i_2: on the identity map A = P, so A P^{-1} r = r."""
    need_gpu()
    from paper_1602_01636_gb300 import igafd
    patch = igafd.Patch.from_problem(synth.Problem(3, (100, 100, 5), 6))
    r = to_dev(np.random.default_rng(0).standard_normal(patch.N))
    assert rel(patch.apply_A(patch.apply_prec(r)).cpu().numpy(), r.cpu().numpy()) <= 1e-10
    patch.close()


def test_folded_map_is_refused():
    need_gpu()
    from paper_1602_01636_gb300 import igafd
    prob = synth.Problem(3, (9, 8, 10), 2, [0.9, -0.7, 0.8])
    with pytest.raises(igafd.IgafdError) as e:
        igafd.Patch.from_problem(prob)
    assert e.value.status == igafd.ERR_FOLDED
