"""The z chunk of an untuned 3-D handle: the one whose busiest CTA has the fewest
planes, an item counting four beside those it writes.  The sets are some whose
chunk was chosen too short when an item counted three.
"""
import pytest

pytestmark = pytest.mark.gpu

CHUNKS = list(range(1, 17)) + [18, 20, 22, 24, 26, 28, 30, 32, 36, 40, 44, 48, 56, 64, 72, 80, 96, 128]


def _busiest(count, nx, ny, nz, chunk, ctas):
    tiles = -(-nx // 28) * -(-ny // 12)
    load, k = [0] * ctas, 0
    for z0 in range(0, nz, chunk):
        for _ in range(count * tiles):
            load[k % ctas] += min(chunk, nz - z0) + 4
            k += 1
    return max(load)


@pytest.mark.parametrize("count,nx,ny,nz,precision", [
    (2, 54, 137, 246, 0), (3, 44, 116, 200, 0), (8, 48, 193, 102, 1), (1, 32, 32, 160, 0),
    (1, 20, 20, 1, 0), (2, 30, 26, 33, 0)])
def test_choice(count, nx, ny, nz, precision):
    import torch
    from paper_1702_04487_gb300 import inkjet as ij, workloads as W
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    h = ij.ij_create([W.small_nozzle3(nx=nx, ny=ny, nz=nz, nozzle_length=max(1, nz // 4), seed=k,
                                      precision=precision) for k in range(count)])
    (t,) = ij.ij_get_tuning(h)
    ctas = torch.cuda.get_device_properties(0).multi_processor_count
    cost = {c: _busiest(count, nx, ny, nz, c, ctas) for c in CHUNKS}
    assert t["chunk"] == min(CHUNKS, key=lambda c: (cost[c], c))
