"""The FP32 block Jacobi solver keeps the spectrum's scale over its many rounds."""
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


@pytest.mark.parametrize("n", [200, 400, 700])
@pytest.mark.parametrize("decades", [None, 1, 4])
def test_scale(lib, n, decades):
    """A round multiplies A by unitaries rounded to FP32, whose columns' norms are off by at most
    eps = 2^-24 either way: over the rounds a random walk, four standard deviations of which are
    allowed for the mean relative shift of the eigenvalues."""
    rng = np.random.default_rng(10 * n)
    x = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    if decades is None:
        h = x + x.conj().T
    else:
        q, _ = np.linalg.qr(x)
        h = (q * 10.0 ** -np.linspace(0, decades, n)) @ q.conj().T
    h = h.astype(np.complex64)
    h = (h + h.conj().T) / 2
    a = torch.tensor(h, device="cuda")
    v, w = torch.zeros_like(a), torch.zeros(n, dtype=torch.float64, device="cuda")
    sweeps = lib.kernel_heig(1, n, a, v, w)
    ref = np.sort(np.linalg.eigvalsh(h.astype(complex)))[::-1]
    d = w.cpu().numpy() - ref
    rounds = sweeps * ((n + 15) // 16 * 2 - 1)
    assert abs((d * ref).sum() / (ref * ref).sum()) < 4 * np.sqrt(rounds) * 2.0 ** -24
