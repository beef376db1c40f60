"""The pivoted Cholesky factor against its definition, at the edges of its launch shapes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()
    import paper_2309_08572_gb300 as pkg
    return pkg


def _psd(n, rank):
    """B B^+ with the columns of B over seven decades."""
    rng = np.random.default_rng(1000 * n + rank)
    b = rng.standard_normal((n, rank)) + 1j * rng.standard_normal((n, rank))
    b *= 10.0 ** -np.linspace(0, 7, rank)
    return b @ b.conj().T


# one CTA, four, eight (8 and 4 lanes a row), sixteen, and the pivot's row by a second hop; full
# rank, a rank cut short by the tolerance, and more than the columns allowed
@pytest.mark.parametrize("n,rank,rmax", [(1, 1, 168), (2, 2, 1), (31, 9, 168), (32, 32, 168),
                                         (33, 33, 168), (64, 20, 7), (65, 65, 168), (160, 50, 168),
                                         (161, 161, 161), (256, 30, 168), (257, 200, 168),
                                         (832, 40, 168), (833, 40, 168), (1024, 190, 168)])
def test_factor(lib, n, rank, rmax):
    w = _psd(n, rank)
    tol = 1e-13
    ld = min(n, rmax) + 3
    dw = torch.from_numpy(w).cuda()
    L = torch.full((n, ld), 7.0, dtype=torch.complex128, device="cuda")
    piv = torch.zeros(min(n, rmax), dtype=torch.int32, device="cuda")
    r, resid = lib.kernel_pchol(n, dw, rmax, tol, L, piv)
    assert 1 <= r <= min(n, rmax)
    got = L.cpu().numpy()
    assert (got[:, r:] == 7.0).all()                    # nothing beyond the factor is written
    got, p, tr = got[:, :r], piv.cpu().numpy()[:r], np.trace(w).real
    assert len(set(p)) == r
    # the rounding of a remainder's entry: r products and one subtraction, each of a term that is
    # at most the largest diagonal, a few units in the last place each
    eps = 4 * (r + 2) * 2.0 ** -53 * np.diag(w).real.max()
    rem = np.diag(w).real.copy()
    for j in range(r):
        assert rem[p[j]] >= rem.max() - 2 * eps          # the largest remaining diagonal
        assert abs(got[p[j], j].real ** 2 - rem[p[j]]) <= eps
        rem -= np.abs(got[:, j]) ** 2
        rem[p[: j + 1]] = 0
    left = w - got @ got.conj().T
    if r < min(n, rmax):
        assert rem.max() <= tol * tr + eps
    # the remainder is PSD: no entry beyond its largest diagonal
    assert np.abs(left).max() <= max(rem.max(), 0) + 3 * eps
    assert abs(resid * tr - max(rem.max(), 0)) <= 2 * eps
