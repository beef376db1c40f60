"""Split-precision products whose tile rule takes 192 columns, with ragged last tiles."""
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


@pytest.mark.parametrize("mode,unit", [("tf32x3", 2.0 ** -22), ("bf16x3", 2.0 ** -16)])
@pytest.mark.parametrize("m,n,k", [(1300, 1241, 37), (1281, 1248, 16)])
def test_wide_tiles(lib, mode, unit, m, n, k):
    rng = np.random.default_rng(m + n)
    a = (rng.standard_normal((m, k)) + 1j * rng.standard_normal((m, k))).astype(np.complex64)
    b = (rng.standard_normal((k, n)) + 1j * rng.standard_normal((k, n))).astype(np.complex64)
    c = torch.full((m, n), float("nan"), dtype=torch.complex64, device="cuda")
    lib.kernel_tcgemm(mode, 0, 0, m, n, k, torch.tensor(a, device="cuda"), k, 0,
                      torch.tensor(b, device="cuda"), n, 0, c, n, 0, 1)
    # the dropped low parts and the parts' own rounding, four units a product at the most, and one
    # FP32 rounding for each of the 3 x 2k terms of a sum; |re| + |im| bounds either part
    s = lambda x: np.abs(x.real).astype(float) + np.abs(x.imag)
    lim = (4 * unit + 6 * k * 2.0 ** -24) * (s(a) @ s(b))
    err = c.cpu().numpy().astype(complex) - a.astype(complex) @ b.astype(complex)
    assert (np.maximum(np.abs(err.real), np.abs(err.imag)) <= lim).all()
