"""The graded eigensolver on matrices L^+ L with runs of nearly equal eigenvalues of any length, and
with spectra whose close pairs are a matter of chance, against numpy in FP64."""
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


def _factor(h):
    """Columns of the pivoted Cholesky factor of h."""
    d, L = np.diag(h).real.copy(), np.zeros(h.shape, dtype=complex)
    for j in range(len(h)):
        p = int(np.argmax(d))
        c = h[:, p] - L[:, :j] @ L[p, :j].conj()
        L[:, j] = c / np.sqrt(d[p])
        d = np.maximum(d - np.abs(L[:, j]) ** 2, 0)
        d[p] = 0
        if d.max() <= 1e-16 * np.trace(h).real:
            return L[:, :j + 1]
    return L


def _spectra():
    for run in (2, 14, 16, 17, 20, 40):
        for gap in (1e-9, 1e-7, 1e-6, 1e-4, 1e-3):
            yield 60, run, gap
    for n, run, gap in ((168, 100, 1e-7), (168, 168, 1e-6), (33, 33, 1e-8), (19, 18, 0.0)):
        yield n, run, gap
    for n in (100, 160):
        yield n, 0, 0.0


@pytest.mark.parametrize("n,run,gap", list(_spectra()))
def test_runs(lib, n, run, gap):
    """Three decades, `run` values a relative `gap` apart (run = 0: all within one decade).  The last
    pass leaves pairs at angles of at most 1e-6, hence norms, angles and relative couplings
    |v_i^+ A v_j| / sqrt(l_i l_j) of 1e-12 a pair, ten of which are allowed; eigenvalues are off by
    the square of a coupling, a norm, or the rounding of A and of the reference, 4 n eps ||A||."""
    rng = np.random.default_rng(1000 * n + run)
    w = 1 + 9 * rng.random(n) if run == 0 else 10.0 ** (-3 * rng.random(n))
    w[:run] = 0.3 * (1 + gap * np.arange(run))
    w = np.sort(w)[::-1]
    x = rng.standard_normal((n + 20, n)) + 1j * rng.standard_normal((n + 20, n))
    q, _ = np.linalg.qr(x)
    L = _factor((q * w) @ q.conj().T)[:, :n]
    a = L.conj().T @ L
    a = 0.5 * (a + a.conj().T)
    m = len(a)
    ta = torch.tensor(a, device="cuda")
    tv, tw = torch.zeros_like(ta), torch.zeros(m, dtype=torch.float64, device="cuda")
    lib.kernel_heig_graded(m, ta, tv, tw)
    got, v = tw.cpu().numpy(), tv.cpu().numpy()
    o = np.argsort(got)[::-1]
    got, v = got[o], v[:, o]
    ref = np.linalg.eigvalsh(a)[::-1]
    tol = 1e-11
    assert np.abs(v.conj().T @ v - np.eye(m)).max() < tol
    assert (np.abs(got - ref) < tol * ref + 4 * m * 2.0 ** -53 * ref[0]).all()
    s = np.abs(v.conj().T @ a @ v)
    np.fill_diagonal(s, 0)
    # the products that form s round to 4 m eps ||A||
    lim = tol * np.sqrt(np.outer(got, got)) + 4 * m * 2.0 ** -53 * ref[0]
    assert (s < lim).all()
