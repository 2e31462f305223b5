"""The training kernels where they can go wrong: hidden widths that do not
fill a 32-unit slice or a 64-wide chunk, minibatches around the 128-row tile,
one to eight members.
"""
import numpy as np
import pytest

from oracle import mlp_oracle as M

pytestmark = pytest.mark.gpu

CASES = [(1, 16, 16), (2, 48, 112), (3, 80, 144), (2, 144, 128), (8, 208, 272), (5, 256, 256),
         (1, 256, 1040)]


@pytest.fixture(scope="module")
def S():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1702_04487_gb300 import surrogate
    return surrogate


def _data(n, seed):
    from paper_1702_04487_gb300 import surrogate as S
    rng = np.random.default_rng(seed)
    x = S.sample_inputs(n, seed).astype(np.float32)
    y = np.stack([3000 * np.exp(0.2 * rng.standard_normal(n)), 0.05 + 0.01 * rng.random(n),
                  400 * np.exp(0.3 * rng.standard_normal(n)), 1 + rng.random(n)], 1)
    return x, y.astype(np.float32)


def _transformed(sg, x, y):
    im, isc, om, osc = sg.transform()
    xv, yv = x.copy(), y.copy()
    for d in range(7):
        if (sg.config["log_inputs"] >> d) & 1:
            xv[:, d] = np.log(xv[:, d])
    for d in range(4):
        if (sg.config["log_outputs"] >> d) & 1:
            yv[:, d] = np.log(yv[:, d])
    return ((xv - im) / isc).astype(np.float64), ((yv - om) / osc).astype(np.float64)


@pytest.mark.parametrize("members,H,rows", CASES)
def test_gradients(S, members, H, rows):
    """Every layer against the oracle's backward pass with BF16 rounding at the
    same points, within the bounds of the H = 32 gradient test (2 % of the
    largest entry, 1 % in the Frobenius norm)."""
    sg = S.Surrogate(members=members, hidden=H, batch=max(rows, 16), seed=H + rows)
    x, y = _data(rows + 20, 5)
    sg.set_data(x, y)
    g, loss = sg.gradients(x[:rows], y[:rows])
    xt, yt = _transformed(sg, x[:rows], y[:rows])
    w = np.array(sg.config["out_weight"])
    for m in range(members):
        Wt, b = S.unpack(sg.get_params(m).astype(np.float64), H)
        Wt[0], Wt[4], b[4] = Wt[0][:, :7], Wt[4][:4], b[4][:4]
        out, cache = M.forward(Wt, b, xt, bf16=True)
        gW, gb = M.backward(Wt, b, cache, out, yt, weight=w, bf16=True)
        Wg, bg = S.unpack(g[m].astype(np.float64), H)
        assert not Wg[0][:, 7:].any() and not Wg[4][4:].any() and not bg[4][4:].any()
        Wg[0], Wg[4], bg[4] = Wg[0][:, :7], Wg[4][:4], bg[4][:4]
        assert abs(loss[m] - M.mse_loss(out, yt, weight=w)) < 1e-3 * loss[m]
        for l in range(5):
            for got, ref in ((Wg[l], gW[l]), (bg[l], gb[l])):
                scale = np.abs(ref).max() + 1e-30
                assert np.abs(got - ref).max() < 2e-2 * scale, (m, l)
                assert np.linalg.norm(got - ref) < 1e-2 * np.linalg.norm(ref) + 1e-30, (m, l)


def _mix64(z):
    mask = (1 << 64) - 1
    z = (z + 0x9E3779B97F4A7C15) & mask
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
    return z ^ (z >> 31)


@pytest.mark.parametrize("members,H,rows", CASES)
def test_first_steps(S, members, H, rows):
    """The first Adam step from zero moments moves every parameter by lr g /
    (|g| + eps) of its own minibatch's gradient: the update of an entry is lr
    times a number in [-1, 1] computed in a few FP32 operations, and is added
    with one rounding (2^-24 of at most 1), so 1e-6 lr + 2^-23 bounds the
    difference.  The BF16 copies that the step leaves (forward and transposed)
    are those of the parameters: a fresh ensemble given the same parameters
    has the same gradients bit for bit; and a two-step call equals two
    one-step calls."""
    cfg = dict(members=members, hidden=H, batch=max(rows, 16), lr=1e-3, lr_cosine=0)
    x, y = _data(1100, 9)
    sg, twin, two = [S.Surrogate(seed=4, **cfg) for _ in range(3)]
    for s in (sg, twin, two):
        s.set_data(x, y)
    p0 = [sg.get_params(m).astype(np.float64) for m in range(members)]
    grads = []
    for m in range(members):
        r = [_mix64((4 ^ 0x5EED) ^ _mix64((m << 56) ^ i)) % len(x) for i in range(rows)]
        grads.append(sg.gradients(x[r], y[r])[0][m].astype(np.float64))
    sg.train(1)
    for m in range(members):
        want = p0[m] - 1e-3 * grads[m] / (np.abs(grads[m]) + 1e-8)
        assert np.abs(sg.get_params(m) - want).max() <= 1e-9 + 2.0 ** -23
        twin.set_params(m, sg.get_params(m))
    a, b = sg.gradients(x[:rows], y[:rows]), twin.gradients(x[:rows], y[:rows])
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    sg.train(1)
    two.train(2)
    for m in range(members):
        assert np.array_equal(sg.get_params(m), two.get_params(m))
