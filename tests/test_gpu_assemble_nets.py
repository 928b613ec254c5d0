"""3D assembly and load vector on nets much finer than the solution space, and
set-ups from several host threads at once."""
import threading

import numpy as np
import pytest

import synth
from oracle import assemble
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def fine_net(elements, p=2, gp=1):
    """Solution knots, geometry knots with `elements` spans in direction 1, control net."""
    kn = [synth.uniform_open_knots(e, p) for e in (5, 3, 4)]
    gk = [synth.uniform_open_knots(e, gp) for e in (elements, 2, 3)]
    return kn, gk, synth.control_net(gk, gp, [0.03, -0.02, 0.015])


def test_set_ups_from_two_threads():
    """Nets of different sizes, whose kernels ask for more and less than 48 KB
    of shared memory, set up and loaded by two threads at once: every call
    succeeds and gives the bits of a call alone."""
    torch = need_gpu()
    from paper_1602_01636_gb300 import igafd
    nets = [fine_net(900), fine_net(6)]

    def once(kn, gk, ctrl):
        patch = igafd.Patch(kn, 2, ctrl, geo_knots=gk, geo_p=1)
        out = [patch.stencil(), patch.load_rhs_sine()]
        patch.close()
        return out

    want = [once(*net) for net in nets]
    torch.cuda.synchronize()
    failed = []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(40):
                    got = once(*nets[i])
                    torch.cuda.current_stream().synchronize()
                    assert all(torch.equal(a, b) for a, b in zip(got, want[i]))
        except BaseException as e:
            failed.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed


# nets whose rows fit in shared memory for all, for one and for no group of
# threads; a fine coefficient net beside a coarse map
@pytest.mark.parametrize("p,gp,elements,kel", [(2, 1, 720, 0), (2, 1, 2900, 0), (2, 2, 3400, 6), (3, 1, 5, 26000),
                                               (5, 1, 6000, 0)])
def test_nets_finer_than_the_space(p, gp, elements, kel):
    """Stencil, load vector and diagnostics against the oracle.

    Tolerance: 1e-13 as for the other assembly tests, and what rounding leaves
    of the map's derivatives along direction 1: differences of control values up
    to 1 over spans 1 / elements are off by up to 2 x 2^-53 elements; Q is formed
    of up to seven of them (two cofactors, the determinant), on both sides: 28,
    with margin 40 x 2^-53 elements."""
    need_gpu()
    tol = 1e-13 + 40 * 2.0 ** -53 * elements
    from paper_1602_01636_gb300 import igafd
    kn, gk, ctrl = fine_net(elements, p, gp)
    field = ofield = None
    if kel:
        ck = [synth.uniform_open_knots(e, 2) for e in (kel, 3, 2)]
        rng = np.random.default_rng(3)
        cv = np.exp(0.2 * rng.standard_normal([len(k) - 3 for k in ck[::-1]]))
        field, ofield = (ck, 2, cv), assemble.ScalarSpline(cv, ck, 2)
    disc = assemble.Discretization(kn, p, assemble.Geometry(ctrl, gk, gp), kappa=1.3, kappa_field=ofield)
    patch = igafd.Patch(kn, p, ctrl, 1.3, geo_knots=gk, geo_p=gp, kappa_field=field)
    want = disc.assemble_stencil()
    S = patch.stencil().cpu().numpy()
    assert np.abs(S - want.reshape(S.shape)).max() <= tol * np.abs(want).max()
    det = assemble.q_matrix(disc.geo.eval_grid([z.ravel() for z in disc.qz])[1])[1]
    assert abs(patch.info.min_detJ - det.min()) <= max(1e-12, tol) * det.max()
    X = patch.quad_points()
    b = patch.load_rhs((1.0 + X[0] * X[1] - X[2]).contiguous()).cpu().numpy()
    bo = disc.assemble_rhs(lambda x, y, z: 1.0 + x * y - z)
    assert np.abs(b - bo).max() <= tol * np.abs(bo).max()
    patch.close()
