"""The vectorized MPO at cuts of every size, from nearly none to coarse, against the oracle's SVD."""
import numpy as np
import pytest

import synth
from oracle import rcs as orcs
from oracle import vmpo as ovmpo

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


@pytest.mark.parametrize("tc", [False, True])
@pytest.mark.parametrize("ppt", [True, False])
@pytest.mark.parametrize("cut", [1e-5, 1e-4, 1e-3, 1e-2])
def test_cut(lib, cut, ppt, tc):
    """FP64: the engine's 1e-9, whatever the cut.  Tensor-core form: as elsewhere 10 eps / gap, the
    products' eps = 2^-48 sqrt(9 chi) against the smallest gap at a truncation, floor 1e-9."""
    c = synth.rcs(8, 6, 24, 1, gamma_diss=0.1, seed=5, delta_pp=0.01)
    ref = ovmpo.VMPO(c.n_sites, orcs.zero_state(), c.chi_max, mode="ppt" if ppt else "naive",
                     sv_cutoff=cut)
    for i, k in orcs.circuit_ops(c):
        ref.apply_two_site(i, k)
    tol = 1e-9
    if tc:
        tol = max(tol, 10 * 2.0 ** -48 * np.sqrt(9 * c.chi_max) / ref.cut_gap_min)
    g = lib.Vmpo(c.n_sites, c.chi_max, ppt=ppt, sv_cutoff=cut, init_vec=[1, 0, 0], tc=tc)
    for layer in lib.circuit_layers(c):
        g.apply_layer(layer)
    e, r = g.expect_energy(1.0, 1.0, 0.0), ref.expect_energy(1.0, 1.0, 0.0)
    print("cut", cut, ppt, tc, "tol", tol, {k: abs(e[k] - r[k]) for k in r})
    b, _ = g.dims()
    assert list(b) == [a.shape[2] for a in ref.A[:-1]]
    for key in r:
        assert abs(e[key] - r[key]) < tol * max(1.0, abs(r[key])), (key, e[key], r[key])
    assert abs(g.purity() - ref.purity()) < tol * ref.purity()
    assert abs(g.collision() - ref.collision()) < tol * ref.collision()
    g.close()
