"""Second-order observables from the library's own site tensors, at the edges of the products'
tiles: bond dimensions whose squares lie below, at and above 32 and 64, odd ones, every cut."""
import types

import numpy as np
import pytest

import synth
from oracle import second_order as so

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


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-11), ("c64", 1e-4)])
@pytest.mark.parametrize("chi", [1, 3, 5, 6, 8, 9])
def test_from_sites(lib, prec, tol, chi):
    # FP64: sums of up to 9 chi^2 products a site, six sites, all of one sign at the end: some
    # 4000 rounding errors of 1e-16 at the most; FP32 environments as elsewhere 1e-4
    c = synth.scaled(synth.chain40(), n_sites=6, chi_max=chi, k_max=5)
    g = lib.Mpdo(c.n_sites, c.chi_max, c.k_max, prec=prec)
    for layer in 3 * lib.circuit_layers(c):   # deep enough for the bonds to reach chi in FP32 too
        g.apply_layer(layer)
    A = [g.site(n) for n in range(c.n_sites)]
    m = types.SimpleNamespace(n=c.n_sites, A=[np.asarray(a, dtype=complex) for a in A])
    assert max(a.shape[0] for a in A) == chi
    for cut in range(1, c.n_sites):
        got, want = g.second_order(cut), so.second_order(m, cut)
        for key in ("xi", "collision"):
            assert abs(got[key] - want[key]) <= tol * abs(want[key]), (cut, key)
        for key in ("s2_left", "s2_right", "i2"):
            assert abs(got[key] - want[key]) <= 4 * tol, (cut, key)
    g.close()
