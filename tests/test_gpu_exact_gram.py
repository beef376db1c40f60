"""Exact-slice products at the edges of their tiles, drains and K splits: Gram matrices (one
packed operand, upper half mirrored) and general products against numpy in FP64, and rows
with a non-finite entry."""
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
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("n,k", [(1, 1), (31, 7), (33, 80), (128, 81), (129, 160), (160, 1000),
                                 (257, 513), (400, 5043), (700, 1500)])
def test_gram(lib, n, k, side):
    """C = A^+ A (side 0) or A A^+ with rows of A scaled over eight decades, within the bound that
    the exact products are held to (|err| <= 2^-40 sum |a||b|); C is exactly Hermitian."""
    rng = np.random.default_rng(n + k)
    a = _rand(rng, (n, k)) * (10.0 ** rng.uniform(-8, 0, (n, 1))).astype(np.float32)
    x = np.ascontiguousarray(a.conj().T) if side == 0 else a       # stored: k x n or n x k
    t = torch.tensor(x, device="cuda")
    c = torch.full((n, n), float("nan"), dtype=torch.complex128, device="cuda")
    ld = x.shape[1]
    lib.kernel_tcgemm_exact(*((2, 0) if side == 0 else (0, 2)), n, n, k, t, ld, 0, t, ld, 0, c, n, 0, 1)
    got = c.cpu().numpy()
    a64 = a.astype(np.complex128)
    err = np.abs(got - a64 @ a64.conj().T) / (np.abs(a64) @ np.abs(a64).T)
    assert err.max() < 2.0 ** -40
    assert np.array_equal(got, got.conj().T)


@pytest.mark.parametrize("m,n,k,batch", [(1, 1, 1, 1), (128, 32, 16, 1), (129, 33, 17, 2),
                                         (64, 64, 2500, 1), (300, 100, 400, 3),
                                         (2100, 600, 40, 1), (500, 500, 300, 2)])
def test_general(lib, m, n, k, batch):
    """The same bound; K = 2500 with two tiles, and tiles that do not deal out evenly, share
    tiles between CTAs as integer sums; 2100 x 600 gives each CTA several tiles."""
    rng = np.random.default_rng(m + n + k)
    a, b = _rand(rng, (batch, m, k)), _rand(rng, (batch, k, n))
    c = torch.full((batch, m, n), float("nan"), dtype=torch.complex128, device="cuda")
    lib.kernel_tcgemm_exact(0, 0, m, n, k, torch.tensor(a, device="cuda"), k, m * k,
                            torch.tensor(b, device="cuda"), n, k * n, c, n, m * n, batch)
    a64, b64 = a.astype(np.complex128), b.astype(np.complex128)
    err = np.abs(c.cpu().numpy() - a64 @ b64) / (np.abs(a64) @ np.abs(b64))
    assert err.max() < 2.0 ** -40


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_rows(lib, bad):
    """A NaN or an infinity makes its row and column of the product NaN and nothing else; a zero
    row gives zeros; denormal entries do not disturb."""
    rng = np.random.default_rng(3)
    a = _rand(rng, (200, 70))
    a[7, 3] = bad
    a[9] = 0
    a[11] *= 1e-42
    t = torch.tensor(a, device="cuda")
    c = torch.zeros((200, 200), dtype=torch.complex128, device="cuda")
    lib.kernel_tcgemm_exact(0, 2, 200, 200, 70, t, 70, 0, t, 70, 0, c, 200, 0, 1)
    got = c.cpu().numpy()
    hit = np.zeros((200, 200), dtype=bool)
    hit[7] = hit[:, 7] = True
    assert np.all(np.isnan(got[hit].real)) and np.all(np.isfinite(got[~hit]))
    assert np.all(got[9][np.arange(200) != 7] == 0)
