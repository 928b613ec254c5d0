"""The split FP64 FD where its schedule, its exactness and its accuracy could
go wrong."""
import numpy as np
import pytest

import synth
from gpu_util import maxrel, need_gpu, rel, to_dev
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


def _knots(n, p, grading):
    x = np.linspace(0.0, 1.0, n - p + 3)
    x = np.sinh(grading * x) / np.sinh(grading) if grading else x
    return np.concatenate([np.zeros(p), x, np.ones(p)])


# graded spans (the smallest 1e-3, 2e-4, 1e-6 of the largest), span scalings
# (standard deviation of their logarithms), and both
@pytest.mark.parametrize("n,p,grading,scaling", [((64, 50), 3, 8.0, 0.0), ((40, 128), 2, 10.0, 0.0),
                                                 ((64, 64), 1, 14.0, 0.0), ((64, 33), 3, 0.0, 2.0),
                                                 ((96, 64), 2, 0.0, 5.0), ((31, 60), 4, 4.0, 4.0),
                                                 ((129, 40), 2, 8.0, 0.0)])
def test_graded_and_scaled_pencils(n, p, grading, scaling):
    """Eigenvectors whose entries differ by orders of magnitude, and right-hand
    sides that meet their smallest ones.

    Tolerance: 10 x 2^-53 of the norms for each of four products (an FP64 chain
    of 128 terms has 5), no amplification: 40 x 2^-53 = 4.4e-15."""
    torch = need_gpu()
    from paper_1602_01636_gb300 import igafd
    kn = [_knots(v, p, grading) for v in n]
    patch = igafd.Patch(kn, p, synth.control_net(kn, p), stencil=False)
    rng = np.random.default_rng(2)
    if scaling:
        logw = scaling * rng.standard_normal((patch.scaling_rows(), 2))
        patch.set_scalings(torch.from_numpy(logw.astype(np.float32)).cuda())
    U = [patch.eigen(k)[1] for k in range(2)]
    size = [np.abs(u).max(axis=1) for u in U]
    cases = [rng.standard_normal(n[::-1]), np.ones(n[::-1]), np.outer(1 / size[1], 1 / size[0])]
    for at in ([s.argmin() for s in size], [s.argmax() for s in size], [v // 2 for v in n]):
        r = np.zeros(n[::-1])
        r[at[1], at[0]] = 1.0
        cases.append(r)
    for r in cases:
        z = patch.apply_prec(to_dev(r.ravel())).cpu().numpy()
        want = reference(patch, r.ravel()).astype(np.float64)
        assert rel(z, want) <= 40 * 2.0 ** -53 and maxrel(z, want) <= 40 * 2.0 ** -53
    patch.close()


def test_eigenvector_images_follow_the_scalings():
    """A pencil within the digits' range, beyond it and back: the route follows
    without a new plan, also in a solve whose iterations are replayed."""
    torch = need_gpu()
    from paper_1602_01636_gb300 import igafd
    patch = igafd.Patch.from_problem(synth.Problem(2, (40, 33), 2))
    b = to_dev(np.random.default_rng(3).standard_normal(patch.N))
    z0, x0 = patch.apply_prec(b).clone(), patch.pcg(b, tol=1e-10)[0].clone()
    logw = 5.0 * np.random.default_rng(4).standard_normal((patch.scaling_rows(), 2))
    patch.set_scalings(torch.from_numpy(logw.astype(np.float32)).cuda())
    z = patch.apply_prec(b).cpu().numpy()
    assert rel(z, reference(patch, b.cpu().numpy()).astype(np.float64)) <= 40 * 2.0 ** -53
    info = patch.pcg(b, tol=1e-10, max_iter=20)[1]         # (a poor P: only that it runs)
    assert info.status in (igafd.OK, igafd.ERR_NOT_CONVERGED)
    patch.set_scalings(None)
    assert torch.equal(patch.apply_prec(b), z0) and torch.equal(patch.pcg(b, tol=1e-10)[0], x0)
    patch.close()


# one and two parts, one and two column blocks, the early slices of each length
@pytest.mark.parametrize("dim,n,p", [(3, (20, 33, 8), 2), (2, (96, 128), 3), (2, (200, 129), 2)])
def test_waits_that_give_up(dim, n, p):
    """Every wait gives up at once: NaN in place of what the buffers held, an
    error from a solve, and a patch that works as before afterwards."""
    torch = need_gpu()
    from paper_1602_01636_gb300 import igafd
    patch = igafd.Patch.from_problem(synth.Problem(dim, n, p))
    r = to_dev(np.random.default_rng(6).standard_normal(patch.N))
    want = patch.apply_prec(r).clone()
    patch.set_wait_polls(0)
    assert torch.isnan(patch.apply_prec(r)).all().item()
    with pytest.raises(igafd.IgafdError):
        patch.pcg(r)
    patch.set_wait_polls()
    assert torch.equal(patch.apply_prec(r), want)
    fresh = igafd.Patch.from_problem(synth.Problem(dim, n, p))
    assert torch.equal(patch.pcg(r)[0], fresh.pcg(r)[0])
    patch.close()
    fresh.close()
