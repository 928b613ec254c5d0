"""The split FP64 FD where its schedule, its exactness and its accuracy could
go wrong."""
import numpy as np
import pytest

import synth
from gpu_util import need_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,p", [(3, (24, 40, 31), 2), (3, (70, 96, 65), 3), (2, (128, 100), 3),
                                     (2, (150, 256), 2)])
def test_cold_digits_beside_other_traffic(dim, n, p):
    """B's digits out of L2 and the memory system busy, so that their copies
    come late: the same bits as with everything at hand."""
    torch = need_gpu()
    from paper_1602_01636_gb300 import igafd
    patch = igafd.Patch.from_problem(synth.Problem(dim, n, p), stencil=False)
    r = to_dev(np.random.default_rng(1).standard_normal(patch.N))
    patch.apply_prec(r)
    want = patch.apply_prec(r).clone()
    big = torch.empty(1 << 27, dtype=torch.float64, device="cuda")      # 1 GB, larger than L2
    other = torch.cuda.Stream()
    for _ in range(20):
        big.fill_(1.0)
        other.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(other):
            for _ in range(4):
                big.mul_(1.0)
        assert torch.equal(patch.apply_prec(r), want)
        torch.cuda.current_stream().wait_stream(other)
    torch.cuda.synchronize()
    patch.close()
