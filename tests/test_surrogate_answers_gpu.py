"""The fused prediction kernels at the sizes where they can go wrong: partial
and whole 128-row tiles, one tile per SM and several, hidden widths that do
not fill a 64-wide slice or a 128-unit chunk, and the gate's search at counts
of training points around its groups.
"""
import numpy as np
import pytest

from oracle import mlp_oracle as M

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1702_04487_gb300 import surrogate
    return surrogate


def _set_up(S, members, H, nt, seed):
    rng = np.random.default_rng(seed)
    sg = S.Surrogate(members=members, hidden=H, batch=32, seed=seed)
    x = S.sample_inputs(nt, seed).astype(np.float32)
    y = np.stack([3000 * np.exp(0.2 * rng.standard_normal(nt)), 0.05 + 0.01 * rng.random(nt),
                  400 * np.exp(0.3 * rng.standard_normal(nt)), rng.random(nt)], 1)
    sg.set_data(x, y)
    for m in range(members):
        p = sg.get_params(m)
        for b in S.unpack(p, H)[1]:  # biases (views into p) that matter
            b[:4] = rng.uniform(-0.2, 0.2, 4)
        sg.set_params(m, p)
    return sg, x


def _outputs(S, sg, x, H):
    """Inverse-transformed outcomes of every member, from the oracle's network
    with BF16 rounding at the kernel's rounding points."""
    im, isc, om, osc = [a.astype(np.float64) for a in sg.transform()]
    xt = x.astype(np.float64).copy()
    for d in range(7):
        if (sg.config["log_inputs"] >> d) & 1:
            xt[:, d] = np.log(xt[:, d])
    xt = (xt - im) / isc
    out = []
    for m in range(sg.members):
        Wt, b = S.unpack(sg.get_params(m).astype(np.float64), H)
        Wt[0], Wt[4], b[4] = Wt[0][:, :7], Wt[4][:4], b[4][:4]
        o = M.forward(Wt, b, xt, bf16=True)[0] * osc + om
        for d in range(4):
            if (sg.config["log_outputs"] >> d) & 1:
                o[:, d] = np.exp(o[:, d])
        out.append(o)
    return np.stack(out), osc


@pytest.mark.parametrize("members,H,n", [
    (1, 16, 1), (2, 48, 129), (3, 80, 127), (5, 128, 300), (2, 144, 1000), (8, 208, 257),
    (5, 256, 128), (5, 256, 384),
    (5, 256, 385), (5, 256, 5000), (1, 256, 20000)])
def test_forward_tiles(S, members, H, n):
    """Every row against the oracle.  A hidden value whose FP32 sum lands on
    the other side of a BF16 rounding point moves by 2^-8 of itself; with H of
    them averaged in, 2e-2 of an outcome's scale (the bound of the gradient
    test) is far above what a handful of such moves gives and far below what
    a misplaced tile, chunk or bias gives."""
    sg, _ = _set_up(S, members, H, 300, 3 + H)
    x = S.sample_inputs(n, 77).astype(np.float32)
    mean, sd, _ = sg.predict(x, gate=False)
    o, osc = _outputs(S, sg, x, H)
    scale = np.abs(o).max(axis=(0, 1))
    assert (np.abs(mean - o.mean(0)) <= 2e-2 * scale).all()
    assert (np.abs(sd - o.std(0)) <= 2e-2 * scale).all()
    for r in {0, n // 2, n - 1}:  # a row's answer does not depend on its batch
        one = sg.predict(x[r:r + 1], gate=False)
        assert np.array_equal(one[0][0], mean[r]) and np.array_equal(one[1][0], sd[r])


@pytest.mark.parametrize("nt", [2, 31, 128, 129, 1000])
@pytest.mark.parametrize("n", [1, 9, 456, 457, 4200])
def test_gate_search(S, nt, n):
    """accept against box, spread and nearest distance computed on the host
    (distances in FP64: queries within 1e-5 of the cut or of a spread bound
    are left out, FP32 rounding being 1e-6 of them)."""
    sg, xt = _set_up(S, 3, 32, nt, 5)
    cut = 0.8
    sg.set_gate(0.6, 0.4, cut)
    rng = np.random.default_rng(n)
    x = xt[rng.integers(0, nt, n)].astype(np.float64)
    x[:, :5] *= np.exp(rng.normal(0, 0.15, (n, 5)))
    x = x.astype(np.float32)
    mean, sd, acc = sg.predict(x)
    im, isc, _, _ = [a.astype(np.float64) for a in sg.transform()]

    def tr(a):
        a = a.astype(np.float64).copy()
        for d in range(7):
            if (sg.config["log_inputs"] >> d) & 1:
                a[:, d] = np.log(a[:, d])
        return (a - im) / isc

    q, t = tr(x), tr(xt)
    near = np.array([np.sqrt(((t - v) ** 2).sum(1).min()) for v in q])
    inside = ((x >= xt.min(0)) & (x <= xt.max(0))).all(1)
    rel = sd[:, :2].astype(np.float64) / np.abs(mean[:, :2])
    lim = np.array([0.6, 0.4])
    want = inside & (near <= cut) & (rel <= lim).all(1)
    clear = (np.abs(near - cut) > 1e-5 * cut) & (np.abs(rel - lim) > 1e-5 * lim).all(1)
    assert clear.sum() >= n - 2
    assert np.array_equal(acc.astype(bool)[clear], want[clear])
