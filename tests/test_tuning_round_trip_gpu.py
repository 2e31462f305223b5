"""What ij_get_tuning reports, given to ij_tune, makes another handle run the
same kernels, and ij_autotune times every kernel that a handle can run.
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ij():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1702_04487_gb300 import inkjet
    return inkjet


def _copy(ij, h, to):
    for b in ij.ij_get_tuning(h):
        ij.ij_tune(to, b["block_size"], b["chunk"], b["prefetch"])


def _step_us(ij, h):
    """Least time of a step without diagnostics, over graph replays of 16."""
    import torch
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    us = []
    for _ in range(6):
        e[0].record()
        ij.ij_step(h, 160)
        e[1].record()
        torch.cuda.synchronize()
        us.append(1e3 * e[0].elapsed_time(e[1]) / 160)
    return min(us)


@pytest.mark.parametrize("nx,ny,precision", [(64, 256, 0), (64, 256, 1), (400, 600, 0)])
def test_round_trip(ij, nx, ny, precision):
    """A 64 x 256 lattice takes about 4 us a step in tiles and 10 in strips."""
    from paper_1702_04487_gb300 import workloads as W
    p = W.small_nozzle(nx=nx, ny=ny, F0=1e-4, F_neg=5e-5, precision=precision, diag_every=0)
    a, b = ij.ij_create(p), ij.ij_create(p)
    _copy(ij, a, b)
    assert ij.ij_get_tuning(b) == ij.ij_get_tuning(a)
    if nx == 64:
        assert _step_us(ij, b) < 1.5 * _step_us(ij, a)
    ij.ij_tune(a, 0, 24, 2)  # the list ...
    _copy(ij, a, b)
    (t,) = ij.ij_get_tuning(b)
    assert (t["block_size"], t["chunk"], t["prefetch"]) == (32, 24, 2)
    ij.ij_tune(a, 192, 24, 2)  # ... and the tiles again
    ij.ij_tune(a, 192, 24, 2)
    _copy(ij, a, b)
    (t,) = ij.ij_get_tuning(b)
    assert (t["block_size"], t["chunk"], t["prefetch"]) == (192, 24, 2)
    if nx == 64:
        assert _step_us(ij, b) < 1.5 * _step_us(ij, a)


def test_tiles_are_refused_where_an_untuned_handle_does_not_take_them(ij):
    from paper_1702_04487_gb300 import workloads as W
    h = ij.ij_create(W.small_nozzle(nx=401, ny=600))
    before = ij.ij_get_tuning(h)
    assert before[0]["block_size"] == 32
    for size in (192, 64):
        with pytest.raises(ij.InkjetError) as e:
            ij.ij_tune(h, size, 24, 1)
        assert e.value.status == ij.IJ_ERR_PARAM
    assert ij.ij_get_tuning(h) == before


@pytest.mark.parametrize("nx,ny", [(2000, 3), (64, 1), (64, 5), (64, 256)])
def test_autotune_times_the_tiles_of_every_small_lattice(ij, nx, ny):
    """Four prefetch depths of each list, and the tiles once, however few the
    rows (a candidate is a warm-up and one timed launch)."""
    from paper_1702_04487_gb300 import workloads as W
    h = ij.ij_create(dict(W.small_nozzle(nx=nx, ny=ny, F0=1e-4, F_neg=5e-5), geometry=0))
    n = ij.ij_launch_count(h)
    ij.ij_autotune(h, 1)
    candidates = (ij.ij_launch_count(h) - n) // 2
    assert candidates % 4 == 1
