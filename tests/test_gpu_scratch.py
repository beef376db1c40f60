"""Pooled scratch of the product entry points: calls from several threads on streams of their own,
larger and smaller in turn, with the pool given back in between."""
import threading

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


def test_threads_and_trim(lib):
    def one(seed, out):
        rng = np.random.default_rng(seed)
        st = torch.cuda.Stream()
        for n, k in ((40, 300), (130, 1100), (40, 300), (257, 200)):
            a = (rng.standard_normal((k, n)) + 1j * rng.standard_normal((k, n))).astype(np.complex64)
            with torch.cuda.stream(st):
                d = torch.from_numpy(a).cuda()
                c = torch.zeros((n, n), dtype=torch.complex128, device="cuda")
                lib.kernel_tcgemm_exact(2, 0, n, n, k, d, n, 0, d, n, 0, c, n, 0, 1,
                                        stream=st.cuda_stream)
                got = c.cpu().numpy()
            w = a.astype(complex)
            # 2^-40 of the sum of the moduli, as for the product itself
            lim = 2.0 ** -40 * (np.abs(w).T @ np.abs(w))
            out.append(bool((np.abs(got - w.conj().T @ w) <= lim).all()))
            lib.kernel_trim()
    res = [[] for _ in range(4)]
    ts = [threading.Thread(target=one, args=(i, res[i])) for i in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert res == [[True] * 4] * 4
