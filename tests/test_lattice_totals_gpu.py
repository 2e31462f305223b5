"""The lattice totals of a diagnostics record are FP64 sums of the cells' FP32
values, however long the work items are.

phi of every cell is a multiple of 2^-51 with 24 significant bits and below
2^-6, so that every partial sum of a few thousand of them stays below 4 and is
exact in FP64 in any order: the record must hold the exact sum, whatever the
work list.  (Sums that keep fewer than 53 bits do not: emulated on one lane's
chain below.)
"""
import numpy as np
import pytest

NX, NY, GRAIN = 60, 200, 2.0 ** -51


def _values():
    rng = np.random.default_rng(5)
    e = rng.integers(-27, -5, (NY, NX))
    m = rng.integers(1 << 23, 1 << 24, (NY, NX))
    v = rng.choice([-1.0, 1.0], (NY, NX)) * np.ldexp(m.astype(np.float64), e - 24)
    k = v / GRAIN
    assert np.array_equal(v, v.astype(np.float32)) and np.array_equal(k, np.round(k))
    return v


def _exact(v):
    return sum(int(k) for k in (v / GRAIN).ravel()) * GRAIN


def test_a_pair_of_floats_loses_these_sums():
    """The values tell FP64 from an FP32 pair (TwoSum with an FP32 correction)."""
    lost = 0
    v = _values()
    for lane in range(30):
        chain = v[:, 2 * lane:2 * lane + 2].ravel()
        hi = lo = np.float32(0)
        for x in chain.astype(np.float32):
            s = hi + x
            b = s - hi
            lo = lo + ((hi - (s - b)) + (x - b))
            hi = s
        assert np.cumsum(chain)[-1] == _exact(chain)
        lost += float(hi) + float(lo) != _exact(chain)
    assert lost >= 20


@pytest.mark.gpu
@pytest.mark.parametrize("chunk", [8, 37, NY, 0])
def test_totals_are_exact(chunk):
    import torch
    from paper_1702_04487_gb300 import inkjet as ij, workloads as W
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    v = _values()
    p = dict(W.small_nozzle(nx=NX, ny=NY), geometry=0, axial_bc=1, init_kind=3, init_r=0.0,
             F0=0.0, F_neg=0.0, jitter=0.0, diag_every=1)
    h = ij.ij_create(p)
    ij.ij_tune(h, 0, chunk, 1)
    f, g = ij.ij_get_state(h, 0)
    g[:] = 0
    g[0] = v
    ij.ij_set_state(h, 0, f, g, 0)
    ij.ij_step(h, 1)
    assert ij.ij_history(h, 0)[0, 2] == _exact(v)
