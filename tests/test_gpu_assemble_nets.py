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
