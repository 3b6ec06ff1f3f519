"""Closure network on the tensor cores (pic_mlp_*) against the FP64 oracle network
(oracle.mlp) with the same bfloat16 roundings of weights and matrix inputs.

Tolerances: the two sides differ in FP32 accumulation order and in the sigmoid, which the
kernels take from tanh.approx (relative error ~2^-11).  That error can move a hidden activation
across a bfloat16 rounding boundary; one such flip changes the output by about
|w3| |W2| 2^-8 h1, ~1e-3 of the output scale, in a few samples.  So, relative to the output
scale: median error <= 1e-5 and mean <= 2e-4 (without flips the error is ~1e-7; any real error
in the products or the layout breaks both), maximum <= 5e-3 (the bar for the forward pass is
1e-2); gradients (recovered from the first Adam moment, m = (1 - beta1) g
at t = 1) to cosine >= 0.999 and 2e-2 relative.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pic():
    import __graft_entry__ as ge
    ge.build()
    import paper_0808_4078_gb300 as pic
    return pic


def _data(n, seed=4, nin=9):
    rng = np.random.default_rng(seed)
    x = rng.normal(0, 1, (n, 9)) * np.linspace(0.5, 3, 9) + np.linspace(-1, 1, 9)
    t = np.tanh(x[:, 0] - 0.5 * x[:, 2]) + 0.2 * x[:, 4] ** 2 / 9
    x = x.astype(np.float32).astype(np.float64)
    if nin < 9:
        x[:, nin:] = 0.0
    return x, t.astype(np.float32).astype(np.float64)


def _close(y, yo):
    scale = np.abs(yo).max() + 1e-6
    err = np.abs(y - yo) / scale
    assert np.median(err) <= 1e-5, np.median(err)
    assert err.mean() <= 2e-4, err.mean()
    assert err.max() <= 5e-3, err.max()


def _net(pic, p, x, nin=9):
    from oracle import mlp
    mu, sd = mlp.feature_norm(x[:, :nin])
    mu = np.concatenate([mu, np.zeros(9 - nin)]).astype(np.float32).astype(np.float64)
    sd = np.concatenate([sd, np.ones(9 - nin)]).astype(np.float32).astype(np.float64)
    return pic.ClosureNet(p, mu, sd, nin=nin), mu, sd


def _dev(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float32), device="cuda")


@pytest.mark.parametrize("n", [1, 127, 128, 1000, 70_001, 1 << 20])
def test_forward_matches_oracle(pic, n):
    from oracle import mlp
    x, _ = _data(n)
    p = mlp.init_params(1)
    net, mu, sd = _net(pic, p, x)
    y = net.forward(_dev(x.T)).cpu().numpy().astype(np.float64)
    yo, _ = mlp.forward(p, x, mu, sd, bf16_path=True)
    _close(y, yo)


def test_forward_eight_inputs(pic):
    from oracle import mlp
    x, _ = _data(3000, seed=5, nin=8)
    p = mlp.init_params(2, nin=8)
    net, mu, sd = _net(pic, p, x, nin=8)
    xg = x.copy()
    xg[:, 8] = 123.0              # ignored when nin = 8
    y = net.forward(_dev(xg.T)).cpu().numpy().astype(np.float64)
    yo, _ = mlp.forward(p, x, mu, sd, bf16_path=True)
    _close(y, yo)


def test_gradient_and_loss_match_oracle(pic):
    from oracle import mlp
    n = 5000
    x, t = _data(n, seed=6)
    p = mlp.init_params(3)
    net, mu, sd = _net(pic, p, x)
    loss = net.train_step(_dev(x.T), _dev(t), lr=1e-3)
    g = net.m.cpu().numpy().astype(np.float64) / 0.1          # m = (1 - beta1) g at t = 1
    Lo, go = mlp.loss_and_grad(p, x, t, mu, sd, bf16_path=True)
    assert loss == pytest.approx(Lo, rel=2e-3)
    cos = g @ go / (np.linalg.norm(g) * np.linalg.norm(go))
    assert cos >= 0.999, cos
    assert np.linalg.norm(g - go) <= 2e-2 * np.linalg.norm(go)
    # the Adam update itself: p1 = p - lr m_hat / (sqrt(v_hat) + eps)
    p1 = net.params.cpu().numpy().astype(np.float64)
    pe, _, _ = mlp.adam_step(p.astype(np.float32).astype(np.float64), g, np.zeros_like(g), np.zeros_like(g), 1, 1e-3)
    assert np.abs(p1 - pe).max() <= 1e-6


def test_training_is_deterministic_and_converges(pic):
    from oracle import mlp
    n = 20_000
    x, t = _data(n, seed=8)
    p = mlp.init_params(4)
    runs = []
    for _ in range(2):
        net, _, _ = _net(pic, p, x)
        xd, td = _dev(x.T), _dev(t)
        losses = [net.train_step(xd, td, lr=3e-3) for _ in range(150)]
        runs.append((losses, net.params.cpu().numpy()))
    assert runs[0][0] == runs[1][0]
    assert np.array_equal(runs[0][1], runs[1][1])
    assert runs[0][0][-1] < 0.2 * runs[0][0][0]


def test_forward_on_recorded_moments(pic):
    """The recorder's feature rows feed the network without a copy (ldx = ncoarse)."""
    import pic_inputs as pi
    from oracle import mlp
    wl = pi.weibel_load(ndim=2, nx=64, ny=64, ppc=8, T_perp_beam=0.2, T_bg=0.01, nu=0.1, seed=71)
    eng = pic.Engine.from_workload(wl)
    eng.step(2)
    rows = eng.record_moments(4, 4)                     # (12, 256)
    feats = rows[:9]
    xf = feats.cpu().numpy().T.astype(np.float64)
    p = mlp.init_params(5)
    mu, sd = mlp.feature_norm(xf)
    mu, sd = mu.astype(np.float32).astype(np.float64), sd.astype(np.float32).astype(np.float64)
    net = pic.ClosureNet(p, mu, sd)
    y = net.forward(feats).cpu().numpy().astype(np.float64)
    yo, _ = mlp.forward(p, xf, mu, sd, bf16_path=True)
    _close(y, yo)
    eng.close()


class _Gradient:
    """Gradient (times 1 - beta1) of a network that is left as it is (lr = 0)."""

    def __init__(self, pic, seed=5):
        from oracle import mlp
        self.net = pic.ClosureNet(mlp.init_params(seed, nin=9), np.zeros(9), np.ones(9), nin=9)

    def __call__(self, x, t):
        self.net.m.zero_()
        self.net.train_step(_dev(x), _dev(t), lr=0.0)
        g = self.net.m.cpu().numpy().astype(np.float64)
        return dict(W2=g[640:4736].reshape(64, 64), b2=g[4736:4800], b3=g[4864])


def test_gradient_keeps_fp32_factors(pic):
    """One sample: db2 / db3 = w3 silu'(z2), whatever the residual, to two roundings of delta2 and one
    of each Adam moment (4 x 2^-24, so 2^-21 between two residuals).  Without the third bfloat16 part
    of delta2 it varies by up to 2^-17, without the second by 2^-8."""
    grad, ratio = _Gradient(pic), []
    for target in (-3.1, -0.77, 0.0, 1.3, 2.9):
        g = grad(np.linspace(-1.2, 1.4, 9)[:, None], [target])
        ratio.append(g["b2"] / g["b3"])
    ratio = np.array(ratio)
    assert (np.ptp(ratio, axis=0) <= 2.0 ** -21 * np.abs(ratio[0])).all()


def test_gradient_sums_as_accurate_as_fp32(pic):
    """dW2 of 1024 samples against the FP64 sum over the samples of db2 (of each alone) times its
    bfloat16 h1: an error of at most 1e-7 in norm, what FP32 sums rounded to nearest, one sample after
    the other, have at best; sums of a tile in one go on the tensor cores exceed it."""
    grad, n = _Gradient(pic), 1024
    rng = np.random.default_rng(3)
    x, t = rng.standard_normal((9, n)), rng.normal(0.2, 1.0, n)
    want = np.zeros((64, 64))
    for i in range(n):
        g = grad(x[:, i:i + 1], t[i:i + 1])
        k = np.abs(g["b2"]).argmax()
        h1 = (g["W2"][k] / g["b2"][k]).astype(np.float32)
        h1 = ((h1.view(np.uint32) + np.uint32(0x8000)) & np.uint32(0xffff0000)).view(np.float32).astype(np.float64)
        want += g["b2"][:, None] * h1 / n
    r = grad(x, t)["W2"] - want
    assert np.linalg.norm(r) <= 1e-7 * np.linalg.norm(want)
