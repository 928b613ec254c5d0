"""The split FP64 FD where its schedule, its exactness and its accuracy could
go wrong."""
import numpy as np
import pytest

import synth
from gpu_util import need_gpu, rel, to_dev
from test_gpu_fd_split import reference

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


@pytest.mark.parametrize("n", [(119, 128), (128, 119)])
def test_rows_along_an_eigenvector(n):
    """Rows and columns of equal digits: scaled eigenvectors of degree 1, many
    of whose entries have one size, so that the digits' products add up with
    one sign.

    Tolerance: 5 x 2^-53 of the norms per product (an FP64 chain of 128 terms),
    four products, cond(U_k)^2 = cond(M_k) <= 3 for degree 1: 60 x 2^-53."""
    need_gpu()
    from paper_1602_01636_gb300 import igafd
    patch = igafd.Patch.from_problem(synth.Problem(2, n, 1), stencil=False)
    U = [patch.eigen(k)[1] for k in range(2)]
    rng = np.random.default_rng(5)
    for num, den in ((1, 3), (2, 3), (1, 2)):
        u = [U[k][:, num * (n[k] + 1) // den - 1] for k in range(2)]
        for scale in rng.uniform(1.0, 2.0, 16):
            r = (scale * np.outer(u[1], u[0])).ravel()
            z = patch.apply_prec(to_dev(r)).cpu().numpy()
            assert rel(z, reference(patch, r).astype(np.float64)) <= 60 * 2.0 ** -53
    patch.close()
