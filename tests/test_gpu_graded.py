"""The graded eigensolver (L^+ L of pivoted Cholesky factors) against numpy in FP64."""
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


def _rand(rng, shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def _graded(n, kind):
    """L^+ L of a factor with columns falling over 14 decades (seven of the square root) whose
    normalised columns are well conditioned: generic; with equal and nearly equal sizes (one
    run longer than a Ritz cluster); or already diagonal."""
    rng = np.random.default_rng(n)
    q, _ = np.linalg.qr(_rand(rng, (2 * n + 3, n)))
    d = 10.0 ** (-np.linspace(0, 7, n))
    if kind == "clusters":
        d[n // 3: n // 3 + 20] = d[n // 3]
        d[:2] = (1.0, 1.0 + 1e-9)[: len(d)]
    if kind == "diagonal":
        return q * d
    mix = np.eye(n) + 0.3 / np.sqrt(n) * _rand(rng, (n, n))
    return (q @ mix) * d


@pytest.mark.parametrize("kind", ["generic", "clusters", "diagonal"])
@pytest.mark.parametrize("n", [1, 2, 3, 17, 64, 65, 118, 119, 167, 168])
def test_graded_pairs_relative_to_their_size(lib, n, kind):
    """Bounds, with eps = 2^-53 and C = D^-1 A D^-1 the scaled matrix: FP64 products of length n
    perturb C by at most 8 n eps entrywise, hence the eigenvalues relatively by 8 n eps
    cond(C) n (Demmel and Veselic), and the eigenvectors' overlaps and graded couplings
    |v_i^+ A v_j| / sqrt(l_i l_j) by as much over the relative gap; inside a run of equal
    values only the couplings' size against the FP32 sweeps (1e-5) is promised."""
    L = _graded(n, kind)
    a = L.conj().T @ L
    a = 0.5 * (a + a.conj().T)
    ta = torch.tensor(a, device="cuda")
    tv = torch.zeros_like(ta)
    tw = torch.zeros(n, dtype=torch.float64, device="cuda")
    lib.kernel_heig_graded(n, ta, tv, tw)
    w, v = tw.cpu().numpy(), tv.cpu().numpy()
    d = np.sqrt(np.diag(a).real)
    cond = np.linalg.cond(a / d[:, None] / d)
    tol = 8 * n * 2.0 ** -53 * cond * n + 1e-14
    ref = np.linalg.svd(L, compute_uv=False) ** 2
    w, o = np.sort(w)[::-1], np.argsort(w)[::-1]
    v = v[:, o]
    assert np.max(np.abs(w / ref - 1)) < tol
    g = np.abs(v.conj().T @ v - np.eye(n))
    s = np.abs(v.conj().T @ a @ v) / np.sqrt(np.outer(w, w))
    np.fill_diagonal(s, 0)
    gap = np.abs(w[:, None] - w) / np.maximum(w[:, None], w)
    far = gap > 1e-6
    print(n, kind, "cond", cond, "eig", np.max(np.abs(w / ref - 1)), "ortho", g.max(),
          "coupling", (s * far * gap).max(), "near", (s * ~far).max())
    assert g.max() < 1e-8
    assert (s * far * gap).max() < max(tol, 1e-12)
    assert (s * ~far).max() < 1e-5
