"""The surrogate network's passes at the edges of their tiles, against FP64 sums of the same rounded
operands."""
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


def _passes(w, c, x, t, wout, rnd):
    """Output, loss, gradients of the parameters and of x . wout, products of rnd(.) operands."""
    acts, a = [x], x
    for i, (wi, ci) in enumerate(zip(w, c)):
        z = rnd(a) @ rnd(wi) + ci
        a = np.tanh(z) if i < len(w) - 1 else z
        acts.append(a)

    def back(dz, params):
        grads = []
        for i in range(len(w) - 1, -1, -1):
            grads.append((rnd(acts[i]).T @ rnd(dz), dz.sum(0)))
            da = rnd(dz) @ rnd(w[i]).T
            dz = da * (1 - acts[i] ** 2) if i else da
        return grads[::-1] if params else dz
    loss = ((acts[-1] - t) ** 2).mean()
    g = back(2 * (acts[-1] - t) / t.size, True)
    return acts[-1], loss, g, back(np.tile(wout, (len(x), 1)), False)


# below, at and above a warp's rows, a tile's rows and columns, and rows of 16 bytes; one layer;
# an output wider than one epilogue step
@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("widths,batch", [((3, 2), 1), ((24, 256, 256, 256, 2), 33),
                                          ((7, 33, 65, 5), 129), ((9, 128, 40), 128),
                                          ((64, 64, 1), 31), ((5, 17, 300, 70), 257)])
def test_passes(lib, widths, batch, bf16):
    rng = np.random.default_rng(sum(widths) + batch)
    w = [(rng.standard_normal((a, b)) / np.sqrt(a)).astype(np.float32)
         for a, b in zip(widths[:-1], widths[1:])]
    c = [(0.1 * rng.standard_normal(b)).astype(np.float32) for b in widths[1:]]
    x = rng.uniform(-1, 1, (batch, widths[0])).astype(np.float32)
    t = rng.standard_normal((batch, widths[-1])).astype(np.float32)
    wout = rng.standard_normal(widths[-1]).astype(np.float32)

    def rnd(a):
        if not bf16:
            return np.asarray(a, dtype=float)
        return torch.from_numpy(np.asarray(a, dtype=np.float32)).bfloat16().double().numpy()
    y, loss, g, gx = _passes([v.astype(float) for v in w], [v.astype(float) for v in c],
                             x.astype(float), t.astype(float), wout.astype(float), rnd)
    net = lib.Mlp(list(widths), max_batch=batch + 3, bf16=bf16)
    net.set_params(lib.mlp_flat(list(zip(w, c))))
    xd, td = torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda")
    gxd, yd = torch.full_like(xd, 7.0), torch.zeros((batch, widths[-1]), device="cuda")
    torch.cuda.synchronize()
    got_loss, got = net.loss_grad(xd, td, want_grad=True)
    net.input_grad(xd, wout, gxd)
    net.forward(xd, yd)
    torch.cuda.synchronize()
    # an FP32 sum may put an operand of the next product on the other side of a BF16 rounding, one
    # part in 256 of one term; sums of FP32 products themselves are good to a few 1e-7
    tol = 1.0 / 256 if bf16 else 1e-5
    want = np.concatenate([np.concatenate([a.ravel(), b]) for a, b in g])
    assert np.isfinite(got).all()
    off = 0
    for a, b in g:                                   # each layer's weights and biases
        for v in (a.ravel(), b):
            assert np.abs(got[off:off + v.size] - v).max() <= tol * np.abs(v).max(), off
            off += v.size
    assert off == want.size
    assert abs(got_loss - loss) <= tol * loss
    assert np.abs(yd.cpu().numpy() - y).max() <= tol * np.abs(y).max()
    assert np.abs(gxd.cpu().numpy() - gx).max() <= tol * np.abs(gx).max()
