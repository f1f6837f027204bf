"""FNO surrogate kernels against the FP64 oracle (oracle/fno.py), through the
C ABI: forward outputs and every parameter gradient, in the FP32-weight
checking mode (tight) and with BF16 spectral weights (BF16-level), plus the
Adam training loop, the library-side normalisation and pair training, and
the judge of pf_surrogate_step."""
import numpy as np
import pytest

import synth
from oracle import fno as ofno

pytestmark = pytest.mark.gpu

SHAPE = (16, 16, 16)
DIMS = dict(C=8, modes=4, H=16, L=2)


@pytest.fixture(scope="module")
def pfg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_36100_gb300 as m
    m.build()
    return m


def odims():
    return ofno.Dims(SHAPE, C=DIMS["C"], m=DIMS["modes"], H=DIMS["H"], L=DIMS["L"])


def data(seed=1):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((4,) + SHAPE)
    t = rng.standard_normal((4,) + SHAPE) * 0.1
    return x, t


def per_tensor(d, a, b):
    out = {}
    o = 0
    for name, s in ofno.layout(d):
        k = int(np.prod(s))
        da, db = a[o:o + k], b[o:o + k]
        out[name] = np.linalg.norm(da - db) / max(np.linalg.norm(db), 1e-30)
        o += k
    return out


@pytest.mark.parametrize("bf16,tol_out,tol_g", [(False, 1e-5, 1e-4), (True, 2e-2, 2e-2)])
def test_forward_and_gradients_vs_oracle(pfg, bf16, tol_out, tol_g):
    import torch
    d = odims()
    theta = ofno.init_params(d, 5)
    # spectral weights large enough that the spectral path matters
    P = ofno.unpack(d, theta)
    for l in range(d.L):
        P["W%d" % l][...] *= 20.0
    x, tgt = data()
    out_ref, acts = ofno.forward(d, theta, x, cache=True)
    g_ref = ofno.backward(d, theta, acts, out_ref, tgt)
    net = pfg.FNO(SHAPE, bf16=bf16, **DIMS)
    try:
        assert net.n == theta.size
        net.set_params(theta.astype(np.float32))
        xt = torch.from_numpy(x.astype(np.float32)).cuda()
        tt = torch.from_numpy(tgt.astype(np.float32)).cuda()
        out = net.forward(xt).cpu().numpy()
        rel = np.linalg.norm(out - out_ref) / np.linalg.norm(out_ref)
        assert rel <= tol_out, rel
        loss = net.backward(tt)
        assert loss == pytest.approx(ofno.loss(out_ref, tgt), rel=max(tol_out, 1e-6))
        errs = per_tensor(d, net.grads().astype(np.float64), g_ref)
        bad = {k: v for k, v in errs.items() if v > tol_g}
        assert not bad, bad
    finally:
        net.close()


@pytest.mark.parametrize("C", [5, 6])
@pytest.mark.parametrize("bf16", [False, True])
def test_mix_of_odd_and_even_channels(pfg, C, bf16):
    """Spectral weights that start on a pair of floats (even C) and between two (odd C), in the kernels of one operation
    each: FP32 sums throughout, spectral weights that BF16 holds exactly."""
    import torch
    shape = (8, 8, 12)
    d = ofno.Dims(shape, C=C, m=3, H=16, L=2)
    theta = ofno.init_params(d, 3).astype(np.float32)
    P = ofno.unpack(d, theta)
    for l in range(d.L):
        w = torch.from_numpy(P["W%d" % l] * np.float32(20.0))
        P["W%d" % l][...] = w.bfloat16().float().numpy()
    rng = np.random.default_rng(2)
    x, tgt = rng.standard_normal((4,) + shape), rng.standard_normal((4,) + shape) * 0.1
    x, tgt = x.astype(np.float32).astype(np.float64), tgt.astype(np.float32).astype(np.float64)
    out_ref, acts = ofno.forward(d, theta.astype(np.float64), x, cache=True)
    g_ref = ofno.backward(d, theta.astype(np.float64), acts, out_ref, tgt)
    net = pfg.FNO(shape, C=C, modes=3, H=16, L=2, bf16=bf16)
    try:
        net.set_params(theta)
        out = net.forward(torch.from_numpy(x.astype(np.float32)).cuda()).cpu().numpy()
        tol = 7 * 2.0 ** -16 if bf16 else 1e-5  # 2 L + 3 split products, or FP32 sums
        assert np.linalg.norm(out - out_ref) <= tol * np.linalg.norm(out_ref)
        net.backward(torch.from_numpy(tgt.astype(np.float32)).cuda())
        errs = per_tensor(d, net.grads().astype(np.float64), g_ref)
        bad = {k: v for k, v in errs.items() if k[0] == "W" and v > 10 * tol}
        assert not bad, bad
    finally:
        net.close()


# the fused layers' edges: the shortest and longest rows, odd rows and sides, padded channels, modes and hidden widths,
# one mode, one layer, modes up to the Nyquist plane of an axis
@pytest.mark.parametrize("shape,dims", [
    ((8, 6, 32), dict(C=32, modes=3, H=128, L=2)),
    ((18, 19, 36), dict(C=4, modes=9, H=128, L=2)),
    ((9, 11, 33), dict(C=18, modes=4, H=100, L=2)),
    ((4, 4, 256), dict(C=8, modes=1, H=16, L=2)),
    ((26, 27, 63), dict(C=2, modes=13, H=64, L=1)),
    ((8, 9, 150), dict(C=30, modes=4, H=65, L=2)),
    ((7, 9, 40), dict(C=5, modes=3, H=20, L=2)),  # odd channel counts run the unfused kernels
    # more rows than one sweep of the row kernels' teams (152 blocks of ten forward, eight backward; four or five of long
    # rows), more tiles than the projection has blocks (304), more rows than the lift's warps (4864)
    ((40, 42, 36), dict(C=32, modes=4, H=128, L=2)),
    ((28, 30, 256), dict(C=32, modes=13, H=64, L=2)),
    ((72, 70, 32), dict(C=8, modes=2, H=100, L=2)),
])
def test_fused_layers_vs_oracle(pfg, shape, dims):
    """Spectral weights that BF16 holds exactly, so that only the products' split (about 2^-16 relative for each of the
    contractions in a row: at most 2 L + 3 of them forward and as many back) and FP32 rounding separate the two."""
    import torch
    d = ofno.Dims(shape, C=dims["C"], m=dims["modes"], H=dims["H"], L=dims["L"])
    theta = ofno.init_params(d, 7).astype(np.float32)
    P = ofno.unpack(d, theta)
    for l in range(d.L):
        w = torch.from_numpy(P["W%d" % l] * np.float32(20.0))
        P["W%d" % l][...] = w.bfloat16().float().numpy()
    rng = np.random.default_rng(3)
    x, tgt = rng.standard_normal((4,) + shape), rng.standard_normal((4,) + shape) * 0.1
    x, tgt = x.astype(np.float32).astype(np.float64), tgt.astype(np.float32).astype(np.float64)
    out_ref, acts = ofno.forward(d, theta.astype(np.float64), x, cache=True)
    g_ref = ofno.backward(d, theta.astype(np.float64), acts, out_ref, tgt)
    net = pfg.FNO(shape, bf16=True, **dims)
    try:
        net.set_params(theta)
        xt, tt = torch.from_numpy(x.astype(np.float32)).cuda(), torch.from_numpy(tgt.astype(np.float32)).cuda()
        bound = (2 * d.L + 3) * 2.0 ** -16
        out = net.forward(xt).cpu().numpy()
        assert np.linalg.norm(out - out_ref) <= bound * np.linalg.norm(out_ref)
        loss = net.backward(tt)
        assert loss == pytest.approx(ofno.loss(out_ref, tgt), rel=bound)
        # A bias gradient is a plain sum over the points of values of both signs: its error scales with the terms and
        # not with what is left of them.  The gradient of the matrix beside the bias sums the same terms times inputs
        # of about unit size, so its norm says how large they are.
        o, bad = 0, {}
        got = net.grads().astype(np.float64)
        ref = ofno.unpack(d, g_ref)
        for name, s in ofno.layout(d):
            k = int(np.prod(s))
            size = np.linalg.norm(ref[name])
            if name[0] in "pvq":
                size = max(size, np.linalg.norm(ref[name[0].upper() + name[1:]]))
            e = np.linalg.norm(got[o:o + k] - g_ref[o:o + k]) / max(size, 1e-30)
            if not e <= 2 * bound:
                bad[name] = e
            o += k
        assert not bad, bad
        # a training step leaves the same gradients without computing the output
        assert net.train_step(xt, tt, 0.0) == loss
        assert np.array_equal(net.grads().astype(np.float64), got)
    finally:
        net.close()


@pytest.mark.parametrize("C,H", [(32, 40), (16, 48), (32, 65), (18, 80), (32, 100), (8, 112)])
def test_hidden_product_in_fp32(pfg, C, H):
    """Hidden widths whose row tiles are no power of two form Q1 a in FP32 (BF16 mode).  Pre-activations are small
    differences of a large product and a large bias, of factors close to 1 + 2^-8, which BF16 rounds most: the product of
    the two remainders, 2^-16 of every term, is what the split form leaves out.  FP32 sums lose at most (C + 2) 2^-24 of
    the terms' sum."""
    import torch
    shape = (8, 10, 36)
    d = ofno.Dims(shape, C=C, m=2, H=H, L=1)
    rng = np.random.default_rng(H)
    theta = ofno.init_params(d, 11)
    P = ofno.unpack(d, theta)
    P["W0"][...] = 0.0
    P["P"][...] = np.eye(4)[np.arange(C) % 4]  # a_1 = the inputs copied into the channels, exact also in BF16 parts
    P["V0"][...] = np.eye(C)
    P["Q1"][...] = 64.0 * (1 + 2.0 ** -8 - rng.integers(1, 64, (H, C)) * 2.0 ** -22)
    P["q1"][...] = -P["Q1"].sum(1) * (1 + 2.0 ** -8 - 4 * 2.0 ** -14)
    P["Q2"][...] = rng.uniform(0.5, 1.0, (4, H)) / H
    theta = theta.astype(np.float32).astype(np.float64)
    x = 1 + 2.0 ** -8 - rng.integers(1, 8, (4,) + shape) * 2.0 ** -14
    out_ref = ofno.forward(d, theta, x)
    net = pfg.FNO(shape, C=C, modes=2, H=H, L=1, bf16=True)
    try:
        net.set_params(theta.astype(np.float32))
        out = net.forward(torch.from_numpy(x.astype(np.float32)).cuda()).cpu().numpy().astype(np.float64)
    finally:
        net.close()
    # GELU' is at most 1.13, the weights of Q2 sum to less than 1, and the output product is the split one
    bound = 1.13 * (C + 2) * 2.0 ** -24 * 64.3 * C + 2.0 ** -16
    assert np.abs(out - out_ref).max() <= bound, (np.abs(out - out_ref).max(), bound)


def test_gelu_derivative(pfg):
    """GELU' through the gradient of q1: Q1 = 0, so that the hidden biases are the arguments, and one point whose output
    error is a power of two and outweighs the others', which are zero.  As exact as the formula with the CUDA library's
    erff and expf, which was measured at 1.5e-7 at most and 3.0e-8 rms for arguments within 3."""
    import math

    import torch
    shape, H = (4, 4, 32), 128
    net = pfg.FNO(shape, C=2, modes=1, H=H, L=1, bf16=True)
    d = ofno.Dims(shape, C=2, m=1, H=H, L=1)
    rng = np.random.default_rng(8)
    err = []
    try:
        x = torch.zeros((4,) + shape, device="cuda")
        for _ in range(24):
            theta = np.zeros(ofno.n_params(d))
            P = ofno.unpack(d, theta)
            z = rng.uniform(-3.0, 3.0, H).astype(np.float32)
            P["q1"][...] = z
            P["Q2"][0] = 1.0
            P["q2"][0] = -sum(float(v) * 0.5 * math.erfc(-float(v) / math.sqrt(2.0)) for v in z)
            net.set_params(theta.astype(np.float32))
            tgt = net.forward(x)
            tgt[0, 1, 2, 3] = -2.0 ** 30
            net.backward(tgt)
            g = net.grads().astype(np.float64)
            o = 0
            for name, s in ofno.layout(d):
                k = int(np.prod(s))
                if name == "q1":
                    got = g[o:o + k] / 2.0 ** 30 * (2 * 512)  # d = 2 (out - target) / (4 N)
                o += k
            ref = np.array([0.5 * math.erfc(-v / math.sqrt(2.0)) + v * math.exp(-0.5 * v * v) / math.sqrt(2 * math.pi)
                            for v in z.astype(np.float64)])
            err.append(got - ref)
    finally:
        net.close()
    err = np.array(err)
    assert np.abs(err).max() <= 1.5e-7, np.abs(err).max()
    assert np.sqrt((err ** 2).mean()) <= 3.0e-8, np.sqrt((err ** 2).mean())


def test_adam_training_reduces_loss(pfg):
    import torch
    d = odims()
    theta = ofno.init_params(d, 6)
    x, _ = data(2)
    tgt = 0.5 * x[::-1].copy()  # a learnable map: scaled channel permutation
    net = pfg.FNO(SHAPE, bf16=True, **DIMS)
    try:
        net.set_params(theta.astype(np.float32))
        xt = torch.from_numpy(x.astype(np.float32)).cuda()
        tt = torch.from_numpy(tgt.astype(np.float32)).cuda()
        first = net.train_step(xt, tt, 3e-3)
        for _ in range(100):
            last = net.train_step(xt, tt, 3e-3)
        assert last < 0.3 * first
        # one GPU Adam step equals the oracle's update from the same gradient
        net.set_params(theta.astype(np.float32))
        net.forward(xt)
        net.backward(tt)
        g = net.grads().astype(np.float64)
        lib = pfg.lib()
        assert lib.pf_fno_adam(net.f, 1e-3, 0.9, 0.999, 1e-8) == 0
        want = ofno.adam_step(theta.astype(np.float32).astype(np.float64), g, np.zeros_like(g), np.zeros_like(g), 1,
                              1e-3)
        assert np.max(np.abs(net.params() - want)) < 1e-6
    finally:
        net.close()


def test_fit_norm_and_train_pair(pfg, params):
    """The library's normalisation statistics equal numpy's over all
    consecutive snapshot pairs, and a training step on a raw pair equals a
    training step on the pair normalised by hand."""
    import torch
    rng = np.random.default_rng(9)
    snaps = rng.standard_normal((2, 3, 4) + SHAPE).astype(np.float32) * np.array([0.01, 0.3, 0.2, 0.1],
                                                                              dtype=np.float32)[None, None, :, None,
                                                                                                 None, None]
    snaps += np.array([0.05, 0.2, 0.1, 0.0], dtype=np.float32)[None, None, :, None, None, None]
    x = snaps[:, :-1].transpose(2, 0, 1, 3, 4, 5).reshape(4, -1).astype(np.float64)
    d = (snaps[:, 1:] - snaps[:, :-1]).transpose(2, 0, 1, 3, 4, 5).reshape(4, -1).astype(np.float64)
    mean, sd, dsd = x.mean(axis=1), x.std(axis=1), d.std(axis=1)
    dev = torch.from_numpy(snaps).to("cuda").contiguous()
    a = pfg.FNO(SHAPE, bf16=False, **DIMS)
    b = pfg.FNO(SHAPE, bf16=False, **DIMS)
    try:
        th = (np.random.default_rng(4).standard_normal(a.n) * 0.05).astype(np.float32)
        a.set_params(th)
        b.set_params(th)
        a.fit_norm(dev)
        la = a.train_pair(dev[0, 0], dev[0, 1], 1e-3)
        b.set_norm(mean, sd, dsd)
        xin = torch.from_numpy(((snaps[0, 0] - mean[:, None, None, None]) / sd[:, None, None, None])
                               .astype(np.float32)).to("cuda").contiguous()
        tgt = torch.from_numpy(((snaps[0, 1] - snaps[0, 0]) / dsd[:, None, None, None])
                               .astype(np.float32)).to("cuda").contiguous()
        lb = b.train_step(xin, tgt, 1e-3)
        assert la == pytest.approx(lb, rel=1e-4)
        assert np.max(np.abs(a.params() - b.params())) <= 1e-6
    finally:
        a.close()
        b.close()


def test_surrogate_step_judged_by_verified_integration(pfg, params):
    """The judge integrates the proposal's interval with the method itself:
    the call ends at the state and time of a plain adaptive integration of
    the same interval (bitwise), and reports the proposal's WRMS distance to
    it (weights from the verified state), accepting only within 1."""
    import torch  # noqa: F401
    p = params
    y0 = synth.ic_spheres(16, 2, 3.0, 4.0, 3, p)
    tau, h, rtol, atol = 8.0, 0.5, 1e-4, 1e-8
    with pfg.Simulation(SHAPE, p, "ark4", "fp64") as ref:
        ref.set_state(y0)
        ref.set_time(0.0, h)
        ref.advance(tau, rtol, atol)
        y_tau = ref.get_state()
        yh_tau = ref.state_hat().cpu().numpy()
    net = pfg.FNO(SHAPE, bf16=True, **DIMS)
    sim = pfg.Simulation(SHAPE, p, "ark4", "fp64")
    try:
        net.set_norm([0.05, 0.0, 0.0, 0.0], [0.05, 1.0, 1.0, 1.0], [1e-3, 1e-2, 1e-2, 1e-2])
        # zero network: the proposal is y(t) itself
        net.set_params(np.zeros(net.n, dtype=np.float32))
        sim.set_state(y0)
        ok, dist = net.surrogate_step(sim, tau, h, rtol, atol)
        want = np.sqrt(np.mean(((y0 - y_tau) / (rtol * np.abs(y_tau) + atol)) ** 2))
        assert dist == pytest.approx(want, rel=1e-9)
        assert ok == (want <= 1.0)
        assert sim.time()[0] == pytest.approx(tau, rel=1e-14)
        assert np.array_equal(sim.state_hat().cpu().numpy(), yh_tau)
        # a noisy network: far outside the tolerance, rejected; the state is
        # still the verified integration
        rng = np.random.default_rng(3)
        net.set_params((rng.standard_normal(net.n) * 3.0).astype(np.float32))
        sim.set_state(y0)
        sim.set_time(0.0, h)
        ok, dist = net.surrogate_step(sim, tau, h, rtol, atol)
        assert not ok and not (dist <= 1.0)
        assert np.array_equal(sim.state_hat().cpu().numpy(), yh_tau)
    finally:
        sim.close()
        net.close()
