"""A device allocation that fails leaves a handle as it was: the call reports
IJ_ERR_OOM, and later calls that fit give what they gave before.

The failure is made on the host: the allocator callback returns NULL for its
k-th request.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


class Allocator:
    """torch's caching allocator, refusing every request from the `left`-th on."""

    def __init__(self, alloc):
        self.alloc, self.left = alloc, None

    def __call__(self, *args):
        if self.left is not None:
            if self.left == 0:
                return 0
            self.left -= 1
        return self.alloc(*args)


@pytest.fixture
def allocator(monkeypatch):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    a = Allocator(torch.cuda.caching_allocator_alloc)
    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", a)
    return a


def _refused(allocator, left, call):
    from paper_1702_04487_gb300 import inkjet as ij
    allocator.left = left
    try:
        with pytest.raises(ij.InkjetError) as e:
            call()
    finally:
        allocator.left = None
    assert e.value.status == ij.IJ_ERR_OOM


def _data(n, seed):
    from paper_1702_04487_gb300 import surrogate as S
    rng = np.random.default_rng(seed)
    y = np.stack([3000 * np.exp(0.2 * rng.standard_normal(n)), 0.05 + 0.01 * rng.random(n),
                  400 * np.exp(0.3 * rng.standard_normal(n)), 1 + rng.random(n)], 1)
    return S.sample_inputs(n, seed).astype(np.float32), y.astype(np.float32)


@pytest.mark.parametrize("left", [0, 1, 2, 3])
def test_queries_that_do_not_fit(allocator, left):
    from paper_1702_04487_gb300 import surrogate as S
    sg = S.Surrogate(members=2, hidden=32, batch=2048, seed=3)
    x, y = _data(300, 1)
    sg.set_data(x, y)
    sg.set_gate(1e9, 1e9, 1e9)
    many, targets = _data(2048, 2)
    want, grads = sg.predict(x[:50]), sg.gradients(x[:48], y[:48])
    _refused(allocator, left, lambda: sg.predict(many))
    _refused(allocator, left, lambda: sg.gradients(many, targets))
    for a, b in zip(sg.predict(x[:50]) + sg.gradients(x[:48], y[:48]), want + grads):
        assert np.array_equal(a, b)
    assert np.isfinite(sg.predict(many)[0]).all()  # it fits again


@pytest.mark.parametrize("left", range(7))
def test_training_data_that_do_not_fit(allocator, left):
    from paper_1702_04487_gb300 import surrogate as S
    sg, twin = [S.Surrogate(members=2, hidden=32, batch=64, seed=3) for _ in range(2)]
    x, y = _data(300, 1)
    more = _data(1000, 2)
    for s in (sg, twin):
        s.set_data(x, y)
        s.set_gate(1e9, 1e9, -1.0)
    _refused(allocator, left, lambda: sg.set_data(*more))
    for a, b in zip(sg.transform(), twin.transform()):
        assert np.array_equal(a, b)
    sg.train(3)
    twin.train(3)
    for a, b in zip(sg.predict(x), twin.predict(x)):
        assert np.array_equal(a, b)
    sg.set_data(*more)  # it fits again
    assert np.isfinite(sg.predict(more[0])[0]).all()


def _states(ij, h, n):
    return [u for k in range(n) for u in ij.ij_get_state(h, k)]


@pytest.mark.parametrize("dim", [2, 3])
def test_work_lists_that_do_not_fit(allocator, dim):
    """A longer work list that cannot be uploaded leaves the list in use."""
    from paper_1702_04487_gb300 import inkjet as ij, workloads as W
    p = W.small_nozzle(nx=70, ny=4000) if dim == 2 else W.small_nozzle3(nx=64, ny=64, nz=160)
    h, twin = ij.ij_create(p), ij.ij_create(p)
    for s in (h, twin):
        ij.ij_tune(s, 0, 64, 1)
    before = ij.ij_get_tuning(h)
    _refused(allocator, 0, lambda: ij.ij_tune(h, 0, 1, 1))
    assert ij.ij_get_tuning(h) == before
    _refused(allocator, 0, lambda: ij.ij_autotune(h, 1))
    assert ij.ij_get_tuning(h) == before
    for s in (h, twin):
        ij.ij_step(s, 25)
    for a, b in zip(_states(ij, h, 1), _states(ij, twin, 1)):
        assert np.array_equal(a, b)
    ij.ij_tune(h, 0, 1, 1)  # it fits again
    ij.ij_step(h, 1)


def test_states_that_do_not_fit(allocator):
    """The FP32 staging buffer of FP16 and 3-D states grows with the lattice."""
    from paper_1702_04487_gb300 import inkjet as ij, workloads as W
    for ps in ([W.small_nozzle(precision=1), W.small_nozzle(nx=96, ny=160, precision=1)],
               [W.small_nozzle3(), W.small_nozzle3(nx=30, ny=30)]):
        h = ij.ij_create(ps)
        want = ij.ij_get_state(h, 0)
        _refused(allocator, 0, lambda: ij.ij_get_state(h, 1))
        for a, b in zip(ij.ij_get_state(h, 0), want):
            assert np.array_equal(a, b)
        assert all(np.isfinite(u).all() for u in ij.ij_get_state(h, 1))
