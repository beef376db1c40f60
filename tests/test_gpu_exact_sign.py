"""The exact-slice products have no preferred sign."""
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


@pytest.mark.parametrize("m,n,k", [(40, 33, 200), (64, 64, 2000)])
def test_negated_operand(lib, m, n, k):
    """The slices of -x are those of x negated, so (-A) B is -(A B) to the last bit; the error
    against FP64 sums stays that of the dropped pairs, with no common shift."""
    rng = np.random.default_rng(k)

    def rand(*s):
        x = (rng.standard_normal(s) + 1j * rng.standard_normal(s)).astype(np.complex64)
        return torch.tensor(x, device="cuda")
    a, b = rand(m, k), rand(k, n)
    out = []
    for x in (a, -a):
        c = torch.zeros((m, n), dtype=torch.complex128, device="cuda")
        lib.kernel_tcgemm_exact(0, 0, m, n, k, x.contiguous(), k, 0, b, n, 0, c, n, 0, 1)
        out.append(c.cpu().numpy())
    assert np.array_equal(out[0], -out[1])
