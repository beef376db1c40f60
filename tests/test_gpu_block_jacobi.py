"""The block Jacobi solver at the edges of its blocks, pairs and tiles, against numpy in FP64."""
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


# beyond the one-CTA solver (84 in FP64, 118 in FP32): one column into a block, a pair, a tile of
# the vectors; more pairs than CTAs' first items; a matrix that needs no rotation; indefinite and
# rank-deficient ones
@pytest.mark.parametrize("kind", ["indefinite", "low_rank", "diagonal"])
@pytest.mark.parametrize("prec,n", [(0, 85), (0, 96), (0, 97), (0, 200), (1, 119), (1, 128),
                                    (1, 129), (1, 145), (1, 193), (1, 517)])
def test_block_jacobi(lib, prec, n, kind):
    rng = np.random.default_rng(n)
    x = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    if kind == "indefinite":
        h = x + x.conj().T
    elif kind == "low_rank":
        h = x[:, :7] @ x[:, :7].conj().T
    else:
        h = np.diag(np.arange(n, 0, -1.0)).astype(complex)
    ct = torch.complex128 if prec == 0 else torch.complex64
    h = torch.tensor(h, dtype=ct).to(torch.complex128).numpy()
    ta = torch.tensor(h, dtype=ct, device="cuda")
    tv, tw = torch.zeros_like(ta), torch.zeros(n, dtype=torch.float64, device="cuda")
    lib.kernel_heig(prec, n, ta, tv, tw)
    torch.cuda.synchronize()
    w, v = tw.cpu().numpy(), tv.cpu().numpy().astype(complex)
    # backward stability, n eps ||H||, as the solver is held to elsewhere
    tol = (4e-16 if prec == 0 else 2e-7) * n
    nrm = np.abs(np.linalg.eigvalsh(h)).max()
    assert np.abs(w - np.sort(np.linalg.eigvalsh(h))[::-1]).max() < tol * nrm
    assert np.abs(h @ v - v * w[None, :]).max() < 10 * tol * nrm
    assert np.abs(v.conj().T @ v - np.eye(n)).max() < 10 * tol
