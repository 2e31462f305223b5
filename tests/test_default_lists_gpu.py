"""The work list of an untuned handle where row chunks are the slower choice
(many strips side by side, FP16 storage, short lattices): the balanced list is
taken, and the state after some steps equals that of a row-chunk list bit for bit.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _lattices(count, nx, ny, precision, uneven=0):
    from paper_1702_04487_gb300 import workloads as W
    out = []
    for k in range(count):
        a, b = nx + 2 * uneven * (k % 3), ny + uneven * (k % 5)
        w = max(4, a // 4)
        out.append(W.small_nozzle(nx=a, ny=b, nozzle_width=w, nozzle_length=max(2, b // 6), seed=k,
                                  theta_deg=40.0 + k % 90, precision=precision, diag_every=4))
    return out


@pytest.mark.parametrize("count,nx,ny,precision,uneven,chunk", [
    (3, 1700, 600, 0, 0, -1),    # 29 strips: the line at 40 rows a slot
    (5, 901, 300, 0, 0, -1),     # 16 strips, odd width: at 30
    (6, 1950, 366, 1, 0, -1),    # FP16: at 60
    (80, 382, 66, 0, 0, -1),     # fewer than 100 rows, a narrow strip
    (130, 334, 61, 0, 0, 0),     # the same, from 20 rows a slot on
    (150, 80, 150, 0, 1, -1),    # uneven, narrow strips, fewer than 200 rows
    (6, 342, 1092, 0, 0, None)])  # 6 strips, tall: row chunks stay
def test_choice(count, nx, ny, precision, uneven, chunk):
    import torch
    from paper_1702_04487_gb300 import inkjet as ij
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    ps = _lattices(count, nx, ny, precision, uneven)
    a, b = ij.ij_create(ps), ij.ij_create(ps)
    (t,) = ij.ij_get_tuning(a)
    assert t["chunk"] == chunk if chunk is not None else t["chunk"] > 0
    ij.ij_tune(b, 0, 37, 1)
    ij.ij_step(a, 5)
    ij.ij_step(b, 5)
    for k in sorted({0, count // 2, count - 1}):
        for u, v in zip(ij.ij_get_state(a, k), ij.ij_get_state(b, k)):
            assert np.array_equal(u, v), k
