"""Small FP64 products (tiles of 8 x 8, 4 x 8 and 4 x 4, and the K loop split over a cluster)
against numpy."""
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


@pytest.mark.parametrize("m,n,k,batch", [(8, 8, 1, 1), (9, 7, 33, 1), (60, 60, 60, 2), (33, 17, 31, 1),
                                         (64, 96, 32, 1), (1, 250, 65, 1), (120, 121, 95, 1),
                                         (41, 41, 1968, 1), (13, 5, 517, 3), (20, 20, 160, 70),
                                         (300, 260, 500, 1)])
@pytest.mark.parametrize("opa,opb", [(0, 0), (2, 0), (0, 2), (1, 3)])
def test_small_fp64_tiles(lib, m, n, k, batch, opa, opb):
    """Products on the 8 x 8, 4 x 8 and 4 x 4 tiles, edges included: FP64 rounding of numpy."""
    rng = np.random.default_rng(m + n + k)
    op = {0: lambda x: x, 1: lambda x: x.T, 2: lambda x: x.conj().T, 3: lambda x: x.conj()}
    a = _rand(rng, (batch,) + ((m, k) if opa in (0, 3) else (k, m)))
    b = _rand(rng, (batch,) + ((k, n) if opb in (0, 3) else (n, k)))
    ta, tb = torch.tensor(a, device="cuda"), torch.tensor(b, device="cuda")
    tc = torch.full((batch, m, n), float("nan"), dtype=torch.complex128, device="cuda")
    lib.kernel_cgemm(0, opa, opb, m, n, k, ta, a.shape[2], m * k, tb, b.shape[2], k * n, tc, n,
                     m * n, batch)
    torch.cuda.synchronize()
    want = np.stack([op[opa](x) @ op[opb](y) for x, y in zip(a, b)])
    scale = np.stack([np.abs(op[opa](x)) @ np.abs(op[opb](y)) for x, y in zip(a, b)])
    assert (np.abs(tc.cpu().numpy() - want) / scale).max() < 4 * (k + 4) * 2.0 ** -53
