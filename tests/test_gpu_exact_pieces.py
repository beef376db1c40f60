"""Exact-slice products whose K is cut into pieces, at sizes whose shorter pieces need more parts
than the longer ones."""
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


@pytest.mark.parametrize("m,n,k,batch,gram", [(2, 2, 8740, 1, True), (9, 9, 18704, 1, True),
                                              (10, 2, 8123, 3, False), (105, 105, 10962, 1, True),
                                              (200, 20, 9001, 2, False), (33, 33, 4097, 1, True)])
def test_long_k(lib, m, n, k, batch, gram):
    """Within the bound that the exact products are held to, |err| <= 2^-40 sum |a||b|."""
    rng = np.random.default_rng(m + k)
    a = _rand(rng, (batch, m, k))
    b = np.ascontiguousarray(a.conj().swapaxes(1, 2)) if gram else _rand(rng, (batch, k, n))
    c = torch.full((batch, m, n), float("nan"), dtype=torch.complex128, device="cuda")
    ta = torch.tensor(a, device="cuda")
    if gram:
        lib.kernel_tcgemm_exact(0, 2, m, n, k, ta, k, m * k, ta, k, m * k, c, n, m * n, batch)
    else:
        tb = torch.tensor(b, device="cuda")
        lib.kernel_tcgemm_exact(0, 0, m, n, k, ta, k, m * k, tb, n, k * n, c, n, m * n, batch)
    a64, b64 = a.astype(np.complex128), b.astype(np.complex128)
    err = np.abs(c.cpu().numpy() - a64 @ b64) / (np.abs(a64) @ np.abs(b64))
    assert err.max() < 2.0 ** -40


@pytest.mark.parametrize("n,k", [(768, 1024), (740, 900), (713, 1720), (423, 235)])
def test_gram_in_one_piece(lib, n, k):
    """A Gram whose plan wants parts where the general product's does not: exponents, packing (one
    launch up to K = 256), the product and its parts, once."""
    rng = np.random.default_rng(n)
    t = torch.tensor(_rand(rng, (k, n)), device="cuda")
    c = torch.zeros((n, n), dtype=torch.complex128, device="cuda")
    before = lib.kernel_launches()
    lib.kernel_tcgemm_exact(2, 0, n, n, k, t, n, 0, t, n, 0, c, n, 0, 1)
    assert lib.kernel_launches() - before <= 4
    a = t.cpu().numpy().astype(np.complex128)
    err = np.abs(c.cpu().numpy() - a.conj().T @ a) / (np.abs(a).T @ np.abs(a))
    assert err.max() < 2.0 ** -40


def test_batch_of_40000(lib):
    """More entries than half of a grid's z extent, which both operands of a short product share."""
    rng = np.random.default_rng(5)
    batch, m, n, k = 40000, 2, 2, 3
    a, b = _rand(rng, (batch, m, k)), _rand(rng, (batch, k, n))
    c = torch.full((batch, m, n), float("nan"), dtype=torch.complex128, device="cuda")
    lib.kernel_tcgemm_exact(0, 0, m, n, k, torch.tensor(a, device="cuda"), k, m * k,
                            torch.tensor(b, device="cuda"), n, k * n, c, n, m * n, batch)
    a64, b64 = a.astype(np.complex128), b.astype(np.complex128)
    err = np.abs(c.cpu().numpy() - a64 @ b64) / (np.abs(a64) @ np.abs(b64))
    assert err.max() < 2.0 ** -40
