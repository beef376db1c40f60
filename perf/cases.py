"""The measured cases: what a user of this library has the GPU do, through its public entry
points, over the sizes that the workloads, the tests and the benchmark of this repository use.

  circuits     one noisy QAOA chain (reset, its layers, the energies) in the default FP64 form
               and in the tensor-core mixed form, and a batch of ragged chains through the
               batch executor
  engine two   the vectorized MPO with purity-preserving truncation on a random circuit
  observables  sampling with energies, and the second-order quantities of a prepared state
  surrogate    one training step and one input gradient of the network that learns energies
  deep chains  the eigensolver and the two tensor-core products at the bond sizes n = 9 D that
               eight-layer chains reach (one such circuit runs for minutes)

Angles, gates and noise rates are drawn from the seed.  Observables of a complex64 state are
returned in 32 bits, the storage precision of the state they are computed from.
"""
import math

import numpy as np
import torch

import paper_2309_08572_gb300 as lib

M_MAX = 25                      # Kraus operators of a noisy QAOA block
FORMS = {"fp64": dict(prec="fp64"),
         # complex64 sites, FP64 Grams, large products on the tensor cores, cut s > 1e-7 s_max
         "mixed_tc": dict(prec="tf32x3", gram_fp64=True, sv_cutoff=1e-7)}


def listed():
    return [
        # the smallest circuit a user checks a setup with: six atoms, one layer, no truncation
        dict(name="circuit_tiny_fp64", kind="circuit", form="fp64", n=6, p=1, chi=64, k=40),
        # the default form on the 40-atom workload
        dict(name="circuit_chain40_fp64", kind="circuit", form="fp64", n=40, p=2, chi=64, k=8),
        # the headline workload: one 100-atom circuit, three layers, energies after each
        dict(name="circuit_chain100", kind="circuit", form="mixed_tc", n=100, p=3, chi=256, k=16),
        # sample generation and angle scans: ragged chains on a pool of eight handles
        dict(name="batch_ragged", kind="batch", count=16, n_min=20, n_max=100, p=2, chi=128, k=8),
        # the vectorized engine with PPT on the bond, on the 8-site random circuit
        dict(name="vmpo_rcs8", kind="vmpo", n=8, layers=4, chi=16, ppt=True),
        # measurement outcomes and energies of a prepared 40-atom state
        dict(name="sample_chain40", kind="sample", n=40, p=2, chi=64, k=8, shots=256),
        # purity, collision probability and mutual information of a prepared state
        dict(name="second_order_n24", kind="second_order", n=24, p=2, chi=16, k=8),
        # one step of surrogate training at its usual batch (BF16 products)
        dict(name="surrogate_train", kind="train", batch=512, p=2, bf16=True),
        # one descent step of the angle search: few rows, latency
        dict(name="surrogate_input_grad", kind="input_grad", batch=64, p=2, bf16=True),
        # bond eigenproblem of a deep chain at D = 150
        dict(name="eig_bond_1350", kind="eig", n=1350),
        # bond Gram of FP32 tensors to FP64 accuracy at D = 256 (3 D columns of D_l K rows)
        dict(name="gram_exact_768", kind="gram", n=768, rows=4096),
        # FP32 product of the new centre in split precision at D = 256
        dict(name="product_tf32x3_2304", kind="product", m=2304, n=2304, k=768),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["circuit_fp64", "circuit_mixed", "batch", "vmpo", "sample", "second_order",
                       "train", "input_grad", "eig", "gram", "product"])
    if kind == "circuit_fp64":
        return dict(kind="circuit", form="fp64", n=rng.randint(6, 40), p=rng.randint(1, 2),
                    chi=rng.choice([16, 32, 64]), k=rng.randint(4, 8))
    if kind == "circuit_mixed":
        return dict(kind="circuit", form="mixed_tc", n=rng.randint(20, 100), p=rng.randint(1, 3),
                    chi=rng.choice([64, 128, 256]), k=rng.randint(8, 16))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 16), n_min=20, n_max=rng.randint(40, 100),
                    p=2, chi=128, k=rng.randint(4, 8))
    if kind == "vmpo":
        return dict(kind="vmpo", n=rng.randint(5, 8), layers=rng.randint(2, 4),
                    chi=rng.randint(6, 16), ppt=rng.random() < 0.5)
    if kind == "sample":
        return dict(kind="sample", n=rng.randint(8, 40), p=rng.randint(1, 2),
                    chi=rng.choice([16, 32, 64]), k=rng.randint(4, 8), shots=_log(rng, 10, 256))
    if kind == "second_order":
        return dict(kind="second_order", n=rng.randint(6, 24), p=rng.randint(1, 2),
                    chi=rng.randint(8, 16), k=rng.randint(4, 8))
    if kind == "train":
        return dict(kind="train", batch=_log(rng, 33, 2048), p=rng.randint(1, 3),
                    bf16=rng.random() < 0.5)
    if kind == "input_grad":
        return dict(kind="input_grad", batch=_log(rng, 8, 512), p=rng.randint(1, 3),
                    bf16=rng.random() < 0.5)
    if kind == "eig":
        return dict(kind="eig", n=_log(rng, 63, 1350))
    if kind == "gram":
        return dict(kind="gram", n=_log(rng, 33, 768), rows=_log(rng, 129, 4096))
    return dict(kind="product", m=_log(rng, 129, 2304), n=_log(rng, 65, 2304), k=_log(rng, 99, 768))


# ------------------------------------------------------------------ inputs
def _angles(rng, p):
    return rng.uniform(0, math.pi, p), rng.uniform(0, math.pi, p)


NOISE = dict(gamma_diss=0.005, gamma_deph=0.005, xtalk=0.01, pp=0.01)


def _qaoa_params(case, seed):
    """Angles of one chain; the noise is that of the 40- and 100-atom workloads."""
    a, b = _angles(np.random.default_rng(seed), case["p"])
    return dict(n=case["n"], alpha=a, beta=b, **NOISE)


def _batch_params(case, seed):
    """Ragged chains: sizes, depths, caps and log-uniform rates as in the batched workload."""
    rng, out = np.random.default_rng(seed), []
    for _ in range(case["count"]):
        n = int(rng.integers(case["n_min"], case["n_max"] + 1))
        p = int(rng.integers(1, case["p"] + 1))
        chi = min(case["chi"], int(rng.choice([32, 64, 128])))
        gd, gp = 10.0 ** rng.uniform(-4, -2, 2)
        a, b = _angles(rng, p)
        out.append(dict(n=n, alpha=a, beta=b, gamma_diss=float(gd), gamma_deph=float(gp),
                        xtalk=0.0, pp=0.01, chi=chi))
    return out


def _layers(q):
    return [lib.build_qaoa_layer(q["n"], k, float(a), float(b), gamma_diss=q["gamma_diss"],
                                 gamma_deph=q["gamma_deph"], xtalk_phase=q["xtalk"],
                                 delta_pp=q["pp"])
            for k, (a, b) in enumerate(zip(q["alpha"], q["beta"]))]


def _haar(case, seed):
    rng = np.random.default_rng(seed)
    z = rng.standard_normal((case["layers"], case["n"], 2, 2, 2)) @ np.array([1.0, 1j])
    q, r = np.linalg.qr(z)
    d = np.diagonal(r, axis1=-2, axis2=-1)
    return q * (d / np.abs(d))[..., None, :]


RCS = dict(gamma_diss=0.1, pp=0.01)


def _net(case, seed):
    """The surrogate's network (4 layers, width 256) and a batch in its feature range."""
    rng = np.random.default_rng(seed)
    widths = [4 + 10 * case["p"], 256, 256, 256, 2]
    w = [(rng.standard_normal((a, b)) / math.sqrt(a)).astype(np.float32)
         for a, b in zip(widths[:-1], widths[1:])]
    c = [(0.1 * rng.standard_normal(b)).astype(np.float32) for b in widths[1:]]
    x = rng.uniform(-1, 1, (case["batch"], widths[0])).astype(np.float32)
    t = rng.standard_normal((case["batch"], 2)).astype(np.float32)
    return widths, w, c, x, t


WOUT = np.array([1.0, -0.5], dtype=np.float32)


def _psd(n, seed):
    """A Hermitian matrix with the graded spectrum of a bond Gram (14 decades)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    z = torch.randn((n, n), dtype=torch.complex128, device="cuda", generator=g)
    q, _ = torch.linalg.qr(z)
    lam = 10.0 ** (-torch.linspace(0, 14, n, dtype=torch.float64, device="cuda"))
    a = (q * lam) @ q.conj().T
    return 0.5 * (a + a.conj().T)


def _matrix(rows, cols, seed):
    """A complex64 site tensor as a matrix, its columns' norms falling over four decades."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    z = torch.randn((rows, cols), dtype=torch.complex64, device="cuda", generator=g)
    return (z * 10.0 ** (-torch.linspace(0, 4, cols, device="cuda"))).contiguous()


def _handle(case, form, **more):
    kw = dict(FORMS[form], **more)
    return lib.Mpdo(case["n"], case["chi"], case["k"], m_max=M_MAX, own_stream=True, **kw)


def prepare(case, seed):
    kind, s = case["kind"], dict(case)
    if kind == "circuit":
        s["m"] = _handle(case, case["form"])
        s["layers"] = [s["m"].upload_layer(ops) for ops in _layers(_qaoa_params(case, seed))]
    elif kind == "batch":
        s["pool"] = [lib.Mpdo(case["n_max"], case["chi"], case["k"], m_max=M_MAX, own_stream=True,
                              **FORMS["mixed_tc"]) for _ in range(8)]
        s["circuits"] = [dict(n_sites=q["n"], chi_max=q["chi"], k_max=case["k"],
                              layers=[s["pool"][0].upload_layer(ops) for ops in _layers(q)])
                         for q in _batch_params(case, seed)]
    elif kind == "vmpo":
        s["layers"] = [lib.build_rcs_layer(case["n"], k, h, RCS["gamma_diss"], 0.0, 0.0, RCS["pp"])
                       for k, h in enumerate(_haar(case, seed))]
    elif kind in ("sample", "second_order"):
        s["m"] = _handle(case, "fp64", sv_cutoff=1e-6)
        for ops in _layers(_qaoa_params(case, seed)):
            s["m"].apply_layer(ops)
        s["seed"] = seed
    elif kind in ("train", "input_grad"):
        widths, w, c, x, t = _net(case, seed)
        s["net"] = lib.Mlp(widths, max_batch=case["batch"], bf16=case["bf16"])
        s["net"].set_params(lib.mlp_flat(list(zip(w, c))))
        s["x"], s["t"] = torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda")
        s["gx"] = torch.zeros_like(s["x"])
    elif kind == "eig":
        n = case["n"]
        s["a"] = _psd(n, seed)
        s["v"] = torch.zeros_like(s["a"])
        s["w"] = torch.zeros(n, dtype=torch.float64, device="cuda")
        g = torch.Generator(device="cuda").manual_seed(seed + 1)
        s["probe"] = torch.randn((1, n), dtype=torch.complex128, device="cuda", generator=g)
    elif kind == "gram":
        s["a"] = _matrix(case["rows"], case["n"], seed)
        s["c"] = torch.zeros((case["n"], case["n"]), dtype=torch.complex128, device="cuda")
    else:
        s["a"] = _matrix(case["m"], case["k"], seed)
        s["b"] = _matrix(case["k"], case["n"], seed + 1)
        s["c"] = torch.zeros((case["m"], case["n"]), dtype=torch.complex64, device="cuda")
    return s


# ------------------------------------------------------------------ one pass
KEYS = ("e_raw", "e_succ", "p_succ", "trace")


def _rows32(es, n):
    """Energies per site (as the surrogate takes them), success probability and trace."""
    return (np.array([[e[k] for k in KEYS] for e in es]) / [n, n, 1, 1]).astype(np.float32)


def _phased(v, w, probe):
    """Eigenvectors are given up to a phase: each column is turned so that its overlap with
    `probe` is real and positive, and weighted with the root of its eigenvalue.  The solver
    promises them to ~1e-8, so they are returned in 32 bits."""
    o = probe @ v
    return (v * (o.abs() / o) * w.clamp_min(0).sqrt()).to(torch.complex64)


def run(s):
    kind = s["kind"]
    if kind == "circuit":
        m = s["m"]
        m.reset()
        out = []
        for layer in s["layers"]:
            m.apply_uploaded(layer)
            out.append(m.expect_energy())
        return out if s["form"] == "fp64" else _rows32(out, s["n"])
    if kind == "batch":
        out = lib.batch_run(s["pool"], s["circuits"])
        return (out / [[c["n_sites"], c["n_sites"], 1, 1] for c in s["circuits"]]).astype(np.float32)
    if kind == "vmpo":
        v = lib.Vmpo(s["n"], s["chi"], ppt=s["ppt"], sv_cutoff=1e-7, init_vec=[1, 0, 0])
        for ops in s["layers"]:
            v.apply_layer(ops)
        out = dict(v.expect_energy(), purity=v.purity(), collision=v.collision())
        v.close()
        return out
    if kind == "sample":
        bits, probs = s["m"].sample_probs(s["shots"], s["seed"])
        # a probability is promised to 2e-6 (the floor of the bond cut), so 32 bits hold it
        return dict(bits=bits, probs=probs.astype(np.float32), energy=s["m"].expect_energy())
    if kind == "second_order":
        return s["m"].second_order(s["n"] // 2)
    if kind == "train":
        loss, grads = s["net"].loss_grad(s["x"], s["t"], want_grad=True)
        s["net"].adam_step(2e-4)
        return dict(loss=loss, grads=grads)
    if kind == "input_grad":
        s["net"].input_grad(s["x"], WOUT, s["gx"])
        return s["gx"]
    if kind == "eig":
        lib.kernel_heig(3, s["n"], s["a"], s["v"], s["w"])
        return dict(w=s["w"], v=_phased(s["v"], s["w"], s["probe"]))
    if kind == "gram":
        n, r = s["n"], s["rows"]
        lib.kernel_tcgemm_exact(2, 0, n, n, r, s["a"], n, 0, s["a"], n, 0, s["c"], n, 0, 1)
        return s["c"]
    lib.kernel_tcgemm("tf32x3", 0, 0, s["m"], s["n"], s["k"], s["a"], s["k"], 0, s["b"], s["n"], 0,
                      s["c"], s["n"], 0, 1)
    return s["c"]


# ------------------------------------------------------------------ the least work of a pass
def _bonds(n, p, chi):
    """Bond dimensions that noisy QAOA layers of random angles reach at the numerical floor
    of the cuts: 7, 18 and 33 after one, two and three layers, less at the chain's ends."""
    top = min(chi, (1, 7, 18, 33)[p])
    return [min(top, 3 ** min(i, n - i, 8)) for i in range(n + 1)]


def _chain_work(n, p, chi, k, word, energies):
    """Flops: the contractions of each update (two Grams, the bond matrix, the split, the new
    centre, its inner Gram and isometry) at the bonds of the layer; bytes: every site tensor
    read and written once per layer, its channel read, and read once per energy."""
    flops = moved = 0.0
    for layer in range(1, p + 1):
        d, kk = _bonds(n, layer, chi), k
        for i in range(n - 1):
            dl, dm, dr = d[i], d[i + 1], d[i + 2]
            mk = min(M_MAX * kk, 3 * dm * dr)
            macs = (dl * kk * (3 * dm) ** 2 + (3 * dm) ** 2 * kk * dr + 2 * (3 * dm) ** 2 * 9 * dm
                    + 2 * dl * kk * 9 * dm * dm + 3 * dm * M_MAX * 3 * dm * kk * dr
                    + mk ** 2 * 3 * dm * dr + kk * mk * 3 * dm * dr)
            flops += 8.0 * macs
            moved += word * (2 * 3 * kk * (dl * dm + dm * dr) / 2 + M_MAX * 81)
        if energies == "layer" or layer == p:
            f, b = _energy_work(d, kk, word)
            flops, moved = flops + f, moved + b
    return flops, moved


def _energy_work(d, k, word):
    flops = sum(8.0 * 4 * 3 * k * (dl * dl * dr + dl * dr * dr) for dl, dr in zip(d, d[1:]))
    return flops, sum(word * 3.0 * k * dl * dr for dl, dr in zip(d, d[1:]))


def work(case):
    kind = case["kind"]
    if kind == "circuit":
        f, b = _chain_work(case["n"], case["p"], case["chi"], case["k"],
                           16 if case["form"] == "fp64" else 8, "layer")
    elif kind == "batch":   # expected over the draws: mean size, half of each depth
        n = (case["n_min"] + case["n_max"]) // 2
        f = b = 0.0
        for p in range(1, case["p"] + 1):
            x, y = _chain_work(n, p, case["chi"], case["k"], 8, "end")
            f, b = f + x * case["count"] / case["p"], b + y * case["count"] / case["p"]
    elif kind == "vmpo":
        f = b = 0.0
        for layer in range(case["layers"]):
            for i in range(case["n"] - 1):
                d = min(case["chi"], 9 ** min(i + 1, case["n"] - 1 - i, 1 + layer))
                f += 8.0 * (81 * d ** 3 + 81 * 81 * d * d + 2 * 81 * d ** 2 * 9 * d)
                b += 16.0 * (4 * 9 * d * d + 81 * 81)
    elif kind == "sample":
        d = _bonds(case["n"], case["p"], case["chi"])
        f, b = _energy_work(d, case["k"], 16)
        f += case["shots"] * sum(8.0 * 3 * case["k"] * (dl * dl * dr + dl * dr * dr)
                                 for dl, dr in zip(d, d[1:]))
    elif kind == "second_order":
        d = _bonds(case["n"], case["p"], case["chi"])
        f = sum(8.0 * 9 * 3 * (dl ** 4 * dr ** 2 + dl ** 2 * dr ** 4) for dl, dr in zip(d, d[1:]))
        b = sum(8.0 * 3 * case["k"] * dl * dr for dl, dr in zip(d, d[1:]))
    elif kind in ("train", "input_grad"):
        widths = [4 + 10 * case["p"], 256, 256, 256, 2]
        macs = sum(x * y for x, y in zip(widths, widths[1:]))
        n = macs + sum(widths[1:])
        train = kind == "train"
        f = 2.0 * case["batch"] * macs * (3 if train else 2)
        # weights, batch, gradients on the device and host, Adam's two moments in and out
        b = 4.0 * (n * (8 if train else 1) + case["batch"] * (widths[0] * 2 + 4))
    elif kind == "eig":      # reduction, eigenvalues and eigenvectors of a dense matrix
        f, b = 8.0 * 9 * case["n"] ** 3, 16.0 * 2 * case["n"] ** 2
    elif kind == "gram":
        f = 8.0 * case["n"] ** 2 * case["rows"]
        b = 8.0 * case["n"] * case["rows"] + 16.0 * case["n"] ** 2
    else:
        m, n, k = case["m"], case["n"], case["k"]
        f, b = 8.0 * m * n * k, 8.0 * (m * k + k * n + m * n)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the same in 64 bits
X2 = np.array([[0, 1, 0], [1, 0, 0], [0, 0, 0]], dtype=complex)
Z2 = np.diag([1.0, -1.0, 0.0]).astype(complex)
PQ = np.diag([1.0, 1.0, 0.0]).astype(complex)
CZ = np.diag([1, 1, 1, 1, -1, 1, 1, 1, 1]).astype(complex)


def _expm(t, h):
    w, v = np.linalg.eigh(h)
    return (v * np.exp(-1j * t * w)) @ v.conj().T


def _noise1(gd, gp):
    """One atom's decay (1/16 into each qubit level, the rest lost) and dephasing, on vec(rho)."""
    f = np.exp(np.array([[0, -gp, -gd / 2 - gp / 4], [-gp, 0, -gd / 2 - gp / 4],
                         [-gd / 2 - gp / 4, -gd / 2 - gp / 4, -gd]])).reshape(-1)
    s = np.diag(f).astype(complex)
    s[0, 8] = s[4, 8] = (1 - math.exp(-gd)) / 16
    return s


def _kraus(u, gd, gp, post=None):
    """Kraus set of the unitary u, then the noise of both atoms, then the unitary post."""
    s1 = _noise1(gd, gp).reshape(3, 3, 3, 3)
    s2 = np.einsum("abcd,efgh->aebfcgdh", s1, s1).reshape(81, 81)
    s = s2 @ np.kron(u, u.conj())
    if post is not None:
        s = np.kron(post, post.conj()) @ s
    c = s.reshape(9, 9, 9, 9).transpose(0, 2, 1, 3).reshape(81, 81)
    w, v = np.linalg.eigh(0.5 * (c + c.conj().T))
    return np.stack([math.sqrt(x) * v[:, i].reshape(9, 9)
                     for i, x in enumerate(w) if x > 1e-15 * w[-1]])


def _promotion(pp):
    g = np.zeros((3, 3), dtype=complex)
    g[1, 2] = g[2, 1] = 1
    p = _expm(pp, g)
    return np.kron(p, p)


def _qaoa_ops(q):
    had = np.array([[1, 1, 0], [1, -1, 0], [0, 0, math.sqrt(2)]], dtype=complex) / math.sqrt(2)
    h2, eye, n = np.kron(np.eye(3), had), np.eye(3), q["n"]
    xt = np.diag(np.exp(-1j * q["xtalk"] * (np.arange(9) == 8)))
    for k, (a, b) in enumerate(zip(q["alpha"], q["beta"])):
        cnot = h2 @ CZ @ h2
        u = _promotion(q["pp"]) @ cnot @ np.kron(eye, _expm(a, Z2)) @ cnot @ xt
        v = _expm(b, X2)
        both = _kraus(u, q["gamma_diss"], q["gamma_deph"], np.kron(v, v))
        mid = _kraus(u, q["gamma_diss"], q["gamma_deph"],
                     np.kron(v, eye) if k % 2 == 0 else np.kron(eye, v))
        order = range(n - 1) if k % 2 == 0 else range(n - 2, -1, -1)
        last = n - 2 if k % 2 == 0 else 0
        yield [(i, both if i == last else mid) for i in order]


def _rcs_ops(case, seed):
    eye, n = np.eye(3, dtype=complex), case["n"]
    for k, haar in enumerate(_haar(case, seed)):
        order = range(n - 1) if k % 2 == 0 else range(n - 2, -1, -1)
        done, ops = set(), []
        for i in order:
            g = []
            for s in (i, i + 1):
                u = eye.copy()
                if s not in done:
                    u[:2, :2] = haar[s]
                done.add(s)
                g.append(u)
            pre = np.kron(*g)
            ops.append((i, _kraus(_promotion(RCS["pp"]) @ CZ @ pre, RCS["gamma_diss"], 0.0)
                        if i % 2 == k % 2 else pre[None]))
        yield ops


def _swap(e):
    return e.reshape(-1, 3, 3, 3, 3).transpose(0, 2, 1, 4, 3).reshape(-1, 9, 9)


def _ppt(lam, keep, t):
    """Purity-preserving values of the kept entries: a point of the plane of the kept values
    and trace weights at the angle that keeps the trace and the purity."""
    lp, tp = lam[:keep], t[:keep]
    nlp, ntp = np.linalg.norm(lp), np.linalg.norm(tp)
    ratio = (lam @ t) / np.linalg.norm(lam) / ntp
    theta = 0.0 if ratio > 1 else math.acos(ratio)
    cs = min(1.0, (lp @ tp) / (nlp * ntp))
    sigma = math.acos(cs)
    out = lp.copy()
    if sigma > 0:
        out = lp + (math.tan(theta) / math.tan(sigma) - 1) * (lp - nlp * cs * tp / ntp)
    out = np.maximum(out, 0) if np.all(t == 1) else np.where(out < 0, 0, out)
    return out * (lam @ t) / (out @ tp)


def _mpdo_step(a, b, e, chi, kmax, cut, inner):
    """One update of a pair with the centre on the left site; it moves to the right one."""
    dl, _, ka, dm = a.shape
    _, _, kb, dr = b.shape
    q, r = np.linalg.qr(a.transpose(0, 2, 1, 3).reshape(dl * ka, 3 * dm))
    qb, rb = np.linalg.qr(b.reshape(dm * 3, kb * dr).conj().T)
    lb = rb.conj().T.reshape(dm, 3, -1)
    core = np.einsum("csb,bte->cste", r.reshape(-1, 3, dm), lb)
    z = np.einsum("mSTst,cste->cSTme", e.reshape(-1, 3, 3, 3, 3), core)
    c, m, x = z.shape[0], z.shape[3], z.shape[4]
    u, s, vh = np.linalg.svd(z.reshape(c * 3, -1), full_matrices=False)
    keep = max(1, min(chi, int(np.sum(s > cut * s[0]))))
    s2 = s[:keep] * math.sqrt((s @ s) / (s[:keep] @ s[:keep]))
    na = np.einsum("xc,cSb->xSb", q, u[:, :keep].reshape(c, 3, keep))
    na = na.reshape(dl, ka, 3, keep).transpose(0, 2, 1, 3)
    nb = (s2[:, None] * vh[:keep]).reshape(keep, 3, m, x)
    # the inner Gram is unchanged by the isometry qb: cut in its small basis, kb kept whole
    full = np.einsum("bTmx,yx->bTmy", nb, qb.conj()).reshape(keep, 3, m * kb, dr)
    mat = full.transpose(2, 0, 1, 3).reshape(m * kb, -1)
    big = mat.shape[0] < mat.shape[1]
    g = np.linalg.qr(mat.conj().T, mode="reduced") if big else (None, None)
    us, sv, vv = np.linalg.svd(g[1].conj().T if big else mat, full_matrices=False)
    vv = vv @ g[0].conj().T if big else vv
    w = sv * sv
    kk = max(1, min(kmax, int(np.sum(sv > inner * sv[0]))))
    lt = _ppt(w, kk, np.ones_like(w))
    new = (np.sqrt(lt)[:, None] * vv[:kk]).reshape(kk, keep, 3, dr).transpose(1, 2, 0, 3)
    return na, new


class _Chain:
    def __init__(self, n, chi, k, cut, inner):
        self.a = [np.array([1, 1, 0], dtype=complex).reshape(1, 3, 1, 1) / math.sqrt(2)] * n
        self.centre, self.lim = 0, (chi, k, cut, inner)

    def apply(self, i, e):
        if self.centre == i:
            self.a[i], self.a[i + 1] = _mpdo_step(self.a[i], self.a[i + 1], e, *self.lim)
            self.centre = i + 1
        else:
            m = lambda x: x.transpose(3, 1, 2, 0)  # noqa: E731
            y, x = _mpdo_step(m(self.a[i + 1]), m(self.a[i]), _swap(e), *self.lim)
            self.a[i], self.a[i + 1], self.centre = m(x), m(y), i

    def energy(self):
        out = {}
        for tag, p in (("raw", np.eye(3)), ("succ", PQ)):
            f = lambda env, a, o: np.einsum("ab,askr,ts,btkq->rq", env, a, o, a.conj(),  # noqa: E731
                                            optimize=True)
            e0, ez, e1 = (np.array([[x]], dtype=complex) for x in (1, 0, 0))
            for a in self.a:
                e0, ez, e1 = (f(e0, a, p), f(e0, a, Z2),
                              f(e1, a, p) + f(e0, a, -X2) - f(ez, a, Z2))
            out[tag] = (e1[0, 0].real, e0[0, 0].real)
        tr, ps = out["raw"][1], out["succ"][1]
        return dict(e_raw=out["raw"][0] / tr, e_succ=out["succ"][0] / ps, p_succ=ps, trace=tr)

    def second_order(self, cut):
        left = _pairs([x for x in self.a[:cut]])
        right = _pairs([x.transpose(3, 1, 2, 0) for x in self.a[cut:][::-1]])
        d = left[0].shape[0]
        pur = np.einsum("abcd,abcd->", left[0], right[0]).real
        tl, tr = left[2], right[2]
        t = np.einsum("ab,ab->", tl, tr).real
        pl = np.einsum("abcd,ab,cd->", left[0], tr, tr).real
        pr = np.einsum("abcd,ab,cd->", right[0], tl, tl).real
        coll = np.einsum("abcd,abcd->", left[1], right[1]).real
        assert d == right[0].shape[0]
        s2, sl, sr = (-math.log(x / t ** 2) for x in (pur, pl, pr))
        return dict(xi=pur / t ** 2, collision=coll / t ** 2, s2_left=sl, s2_right=sr,
                    i2=sl + sr - s2)


def _pairs(sites):
    """Two-copy environments of a run of sites: crossed (tr rho^2), diagonal, and one copy's
    trace; the crossed one pairs copy 1's (s, s') with copy 2's (s', s)."""
    x = np.ones((1, 1, 1, 1), dtype=complex)
    d, t = x.copy(), np.ones((1, 1), dtype=complex)
    for a in sites:
        r = np.einsum("askr,btkq->abstrq", a, a.conj(), optimize=True)
        nx = nd = 0
        for s in range(3):
            for u in range(3):
                y = np.einsum("abcd,abrq->cdrq", x, r[:, :, s, u], optimize=True)
                nx = nx + np.einsum("cdrq,cdvw->rqvw", y, r[:, :, u, s], optimize=True)
            y = np.einsum("abcd,abrq->cdrq", d, r[:, :, s, s], optimize=True)
            nd = nd + np.einsum("cdrq,cdvw->rqvw", y, r[:, :, s, s], optimize=True)
        x, d = nx, nd
        t = np.einsum("ab,abssrq->rq", t, r)
    return x, d, t


def _vmpo(case, seed):
    n, chi, one = case["n"], case["chi"], np.ones(1, dtype=complex)
    tau = np.eye(3).reshape(9)
    st = [np.eye(9)[0].astype(complex).reshape(1, 9, 1)] * n

    def trace(sites):
        v = one
        for a in sites:
            v = np.einsum("l,e,ler->r", v, tau, a)
        return v

    def step(st, i, sup):
        a, b = st[i], st[i + 1]
        th = np.einsum("abcd,lcm,mdr->labr", sup, a, b, optimize=True)
        dl, dr = th.shape[0], th.shape[3]
        u, s, vh = np.linalg.svd(th.reshape(dl * 9, 9 * dr), full_matrices=False)
        nz = int(np.sum(s > 1e-7 * s[0]))
        keep = min(nz, chi)
        s = s[:nz]
        left = np.kron(trace(st[:i]), tau) @ u[:, :nz]
        right = vh[:nz] @ np.kron(tau, trace([x.transpose(2, 1, 0) for x in st[:i + 1:-1]]))
        sk = _ppt(s, keep, (left * right).real) if case["ppt"] else s[:keep]
        st[i], st[i + 1] = u[:, :keep].reshape(dl, 9, keep), (sk[:, None] * vh[:keep]).reshape(keep, 9, dr)

    centre = 0
    for ops in _rcs_ops(case, seed):
        for i, e in ops:
            rev = centre != i
            e5 = (_swap(e) if rev else e).reshape(-1, 3, 3, 3, 3)
            sup = np.einsum("mSTst,mUVuv->SUTVsutv", e5, e5.conj()).reshape(9, 9, 9, 9)
            m = [x.transpose(2, 1, 0) for x in st[::-1]] if rev else st
            step(m, n - 2 - i if rev else i, sup)
            st = [x.transpose(2, 1, 0) for x in m[::-1]] if rev else m
            centre = i if rev else i + 1
    out = {}
    for tag, p in (("raw", np.eye(3)), ("succ", PQ)):
        f = lambda v, a, o: np.einsum("l,e,ler->r", v, o.T.reshape(9), a)  # noqa: E731
        e0, ez, e1 = one, 0 * one, 0 * one
        for a in st:
            e0, ez, e1 = f(e0, a, p), f(e0, a, Z2), f(e1, a, p) + f(e0, a, -X2) - f(ez, a, Z2)
        out[tag] = (e1[0].real, e0[0].real)
    tr, ps = out["raw"][1], out["succ"][1]
    c2, t2 = np.ones((1, 1), dtype=complex), np.ones((1, 1), dtype=complex)
    for a in st:
        g = a[:, [0, 4, 8]]
        c2 = np.einsum("ab,asr,bsq->rq", c2, g, g, optimize=True)
        t2 = np.einsum("ab,aer,beq->rq", t2, a, a.conj(), optimize=True)
    return dict(e_raw=out["raw"][0] / tr, e_succ=out["succ"][0] / ps, p_succ=ps, trace=tr,
                purity=float(t2[0, 0].real), collision=float(c2[0, 0].real) / tr ** 2)


def _mlp(case, seed):
    _, w, c, x, t = _net(case, seed)
    w, c, x, t = [v.astype(float) for v in w], [v.astype(float) for v in c], x.astype(float), t.astype(float)
    acts = [x]
    for i in range(4):
        z = acts[-1] @ w[i] + c[i]
        acts.append(np.tanh(z) if i < 3 else z)
    train = case["kind"] == "train"
    g = 2 * (acts[-1] - t) / t.size if train else np.tile(WOUT.astype(float), (len(x), 1))
    grads = []
    for i in range(3, -1, -1):
        grads[:0] = [(acts[i].T @ g).reshape(-1), g.sum(axis=0)]
        g = g @ w[i].T
        if i:
            g = g * (1 - acts[i] ** 2)
    if not train:
        return g
    return dict(loss=float(np.mean((acts[-1] - t) ** 2)), grads=np.concatenate(grads))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("train", "input_grad"):
        return _mlp(case, seed)
    if kind == "vmpo":
        return _vmpo(case, seed)
    if kind == "eig":
        a = _psd(case["n"], seed)
        g = torch.Generator(device="cuda").manual_seed(seed + 1)
        probe = torch.randn((1, case["n"]), dtype=torch.complex128, device="cuda", generator=g)
        w, v = (torch.tensor(np.ascontiguousarray(x), device="cuda")
                for x in np.linalg.eigh(a.cpu().numpy()))
        return dict(w=w.flip(0), v=_phased(v.flip(1), w.flip(0), probe))
    if kind == "gram":
        a = _matrix(case["rows"], case["n"], seed).to(torch.complex128)
        return a.conj().T @ a
    if kind == "product":
        return (_matrix(case["m"], case["k"], seed).to(torch.complex128)
                @ _matrix(case["k"], case["n"], seed + 1).to(torch.complex128))
    # the plain update takes up to a second at the bonds of a third layer: a three-layer chain
    # or a batch of chains would take most of a minute
    if kind == "batch" or case["p"] > 2:
        return None
    fp64 = kind != "circuit" or case["form"] == "fp64"
    floor = math.sqrt(10 * (1e-16 if fp64 else 1e-14))
    c = _Chain(case["n"], case["chi"], case["k"], floor if kind == "circuit" else 1e-6, floor)
    out = []
    for ops in _qaoa_ops(_qaoa_params(case, seed)):
        for i, e in ops:
            c.apply(i, e)
        out.append(c.energy())
    if kind == "second_order":
        return c.second_order(case["n"] // 2)
    if kind == "sample":   # the outcomes follow the library's generator
        return dict(bits=None, probs=None, energy=out[-1])
    return out if fp64 else _rows32(out, case["n"]).astype(np.float64)
