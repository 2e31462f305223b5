"""The launch shapes an untuned handle and the allocation-free step choose by
size: every choice covers each cell exactly once, so the state after some
steps equals that of a plain row-chunk (or z-chunk) list, bit for bit.
"""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ij():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1702_04487_gb300 import inkjet
    return inkjet


def _lat2(nx, ny, **kw):
    from paper_1702_04487_gb300 import workloads as W
    w = max(4, nx // 4)
    return W.small_nozzle(nx=nx, ny=ny, nozzle_width=w, nozzle_length=max(4, ny // 6), **kw)


@pytest.mark.parametrize("count,nx,ny,chunk,precision", [
    (1, 33, 40, -1, 0), (1, 61, 130, -1, 0),          # a few rows per slot
    (4, 200, 1600, 16, 0), (4, 201, 1601, 16, 0),     # row chunks, a narrow last strip
    (6, 120, 1700, -1, 0), (6, 88, 2600, 12, 1),      # equal pieces; FP16 row chunks
    (300, 64, 480, None, 0)])                          # beyond: at most 56 rows
def test_untuned_2d_list(ij, count, nx, ny, chunk, precision):
    ps = [_lat2(nx, ny, seed=k, theta_deg=40.0 + k % 90, precision=precision)
          for k in range(count)]
    a, b = ij.ij_create(ps), ij.ij_create(ps)
    (t,) = ij.ij_get_tuning(a)
    if chunk is None:
        assert 8 <= t["chunk"] <= 56
    elif chunk == -1:
        assert t["chunk"] == -1
    else:
        assert t["chunk"] > 0
    ij.ij_tune(b, 0, 37, 1)
    ij.ij_step(a, 4)
    ij.ij_step(b, 4)
    for k in sorted({0, count // 2, count - 1}):
        for u, v in zip(ij.ij_get_state(a, k), ij.ij_get_state(b, k)):
            assert np.array_equal(u, v), k


@pytest.mark.parametrize("nx,ny,nz", [(16, 16, 1), (17, 29, 40), (30, 26, 161), (64, 40, 200)])
def test_untuned_3d_chunk(ij, nx, ny, nz):
    from paper_1702_04487_gb300 import workloads as W
    p = W.small_nozzle3(nx=nx, ny=ny, nz=nz, nozzle_width=4, nozzle_length=min(12, max(1, nz // 3)))
    a, b = ij.ij_create(p), ij.ij_create(p)
    ij.ij_tune(b, 0, 80, 1)
    ij.ij_step(a, 3)
    ij.ij_step(b, 3)
    for u, v in zip(ij.ij_get_state(a, 0), ij.ij_get_state(b, 0)):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("nx,ny", [(20, 3), (64, 256), (301, 257), (60, 8192), (1500, 2100)])
def test_noalloc_list(ij, nx, ny):
    """One allocation-free step equals one step of a handle, bit for bit, from
    the same stored state: the handle keeps f - w n0 rounded once (a fused
    multiply-add), which FP64 reproduces (24-bit factors, one rounding)."""
    import torch
    p = dict(_lat2(nx, ny), nozzle_length=max(1, ny // 6), wall_thickness=2, diag_every=0)
    h = ij.ij_create(p)
    ij.ij_step(h, 2)
    f, g = ij.ij_get_state(h, 0)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, np.float32).astype(np.float64)
    fluid = f[0] != 0
    rest = (w * 5.5)[:, None, None] * fluid
    fin = torch.from_numpy((f.astype(np.float64) - rest).astype(np.float32)).cuda()
    gin = torch.from_numpy(g).cuda()
    fo, go = torch.full_like(fin, 7.0), torch.full_like(gin, 7.0)
    st = torch.ones(1, dtype=torch.int32, device="cuda")
    lib = C.CDLL(ij.library_path())
    prm = ij.make_params(p)
    ptr = [C.c_void_p(t.data_ptr()) for t in (fin, gin, fo, go)]
    assert lib.ij_step_noalloc(C.byref(prm), C.c_longlong(2), *ptr, None,
                               C.c_void_p(st.data_ptr()), C.c_void_p(0)) == 0
    torch.cuda.synchronize()
    assert int(st) == 0
    ij.ij_set_state(h, 0, f, g, 2)
    ij.ij_step(h, 1)
    f1, g1 = ij.ij_get_state(h, 0)
    got = (fo.cpu().numpy().astype(np.float64) + rest).astype(np.float32)
    assert np.array_equal(got, f1) and np.array_equal(go.cpu().numpy(), g1)


@pytest.mark.parametrize("ps", [
    [dict(nx=64, ny=256)], [dict(nx=33, ny=41)], [dict(nx=17, ny=9, axial_bc=1)],
    [dict(nx=48, ny=96, axial_bc=2)], [dict(nx=50, ny=70, precision=1)],
    [dict(nx=30, ny=31), dict(nx=64, ny=20, theta_deg=140.0), dict(nx=18, ny=50)],
    [dict(nx=40, ny=40, plate=1)], [dict(nx=5, ny=7, free=1)], [dict(nx=1, ny=1, free=1)],
    [dict(nx=400, ny=600)]], ids=str)
def test_small_lattice_kernel(ij, ps):
    """The kernel of small lattices against the strip list: the same state bit
    for bit, through diagnostics steps (every third) and a moving front."""
    def params(p):
        q = dict(p)
        plate, free = q.pop("plate", 0), q.pop("free", 0)
        nx, ny = q.pop("nx"), q.pop("ny")
        if plate:
            return dict(q, nx=nx, ny=ny, geometry=2, wall_thickness=3, axial_bc=2, init_kind=1,
                        init_x=20.0, init_y=10.0, init_r=9.0, theta_deg=60.0, diag_every=3)
        if free:
            return dict(q, nx=nx, ny=ny, init_kind=2, init_y=ny / 2.0, F0=1e-4, T1=100, diag_every=3)
        w = max(4, nx // 4)
        return dict(_lat2(nx, ny, **q), nozzle_width=w, wall_thickness=max(1, min(3, (nx - w) // 2)),
                    diag_every=3)
    full = [params(p) for p in ps]
    a, b = ij.ij_create(full), ij.ij_create(full)
    ij.ij_tune(b, 0, 11, 1)
    for n in (1, 1, 4, 24):
        ij.ij_step(a, n)
        ij.ij_step(b, n)
    for k in range(len(full)):
        for u, v in zip(ij.ij_get_state(a, k), ij.ij_get_state(b, k)):
            assert np.array_equal(u, v), k
