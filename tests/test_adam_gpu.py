"""Adam on the device against the oracle's, step by step over two calls of
sg_train, with moments that are not zero and the learning rate decaying.

Each step starts from the library's own parameters (those after t steps of an
ensemble that stopped there) and takes the library's own gradient of the step's
minibatch, so that only the moments, the bias corrections, the schedule and the
update are compared.  A call of two steps has learning rates lr and lr / 2 (half
cosine), and its first step equals that of a call of one.

Bound, in units of 2^-24: betas 0.5 and 0.75 have exact powers, so that the bias
corrections carry powf's error alone (4 units, CUDA's documented bound; 4 of
1 - 0.5, three times 4 of 1 - 0.75, halved by the root).  An update is about ten
FP32 operations on terms of at most 4 lr (|m| / sqrt(v) <= 1.23 for these betas,
more for the terms of a cancelling sum): (10 + 4 + 6) 2^-24 4 lr < 1e-5 lr, and
the sum with the parameter is rounded once.
"""
import numpy as np
import pytest

from oracle import mlp_oracle as M

pytestmark = pytest.mark.gpu

LR, BETA1, BETA2, EPS, SEED, ROWS = 0.05, 0.5, 0.75, 1e-8, 4, 48


def _mix64(z):
    mask = (1 << 64) - 1
    z = (z + 0x9E3779B97F4A7C15) & mask
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
    return z ^ (z >> 31)


@pytest.mark.parametrize("members,H", [(2, 48), (1, 256)])
def test_steps_of_two_calls(members, H):
    import torch
    from paper_1702_04487_gb300 import surrogate as S
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    rng = np.random.default_rng(3)
    x = S.sample_inputs(500, 7).astype(np.float32)
    y = np.stack([3000 * np.exp(0.2 * rng.standard_normal(500)), 0.05 + 0.01 * rng.random(500),
                  400 * np.exp(0.3 * rng.standard_normal(500)), 1 + rng.random(500)], 1)
    sg = []
    for calls in ((), (1,), (2,), (2, 1), (2, 2)):  # after 0 .. 4 steps
        s = S.Surrogate(members=members, hidden=H, batch=ROWS, seed=SEED, lr=LR, beta1=BETA1,
                        beta2=BETA2, eps=EPS, lr_cosine=1)
        s.set_data(x, y)
        for m in range(members):  # small parameters, next to which an update is not lost
            s.set_params(m, 0.1 * s.get_params(m))
        for n in calls:
            s.train(n)
        sg.append(s)
    y = y.astype(np.float32)
    for m in range(members):
        mom, var = np.zeros(sg[0].param_count()), np.zeros(sg[0].param_count())
        for t in range(1, 5):
            r = [_mix64((SEED ^ 0x5EED) ^ _mix64((m << 56) ^ ((t - 1) << 24) ^ i)) % len(x)
                 for i in range(ROWS)]
            g = sg[t - 1].gradients(x[r], y[r])[0][m].astype(np.float64)
            p0 = sg[t - 1].get_params(m).astype(np.float64)
            lr = float(np.float32(LR)) * (1.0 if t % 2 else 0.5)
            want = M.adam_step(p0.copy(), g, mom, var, t, lr, BETA1, BETA2, float(np.float32(EPS)))
            got = sg[t].get_params(m).astype(np.float64)
            assert np.abs(got - p0).max() > 0.1 * lr
            assert (np.abs(got - want) <= 1e-5 * lr + 2.0 ** -24 * np.abs(want)).all(), (m, t)
