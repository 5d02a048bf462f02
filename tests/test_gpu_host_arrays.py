"""State read into and set from arrays of unusual memory: what the kernels may
not reach goes through buffers and the driver's copies."""
import ctypes as C
import mmap
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

from helpers import make_scene

pytestmark = pytest.mark.gpu


def scene(nx, ny, seed=1):
    rng = np.random.default_rng(seed)
    sc = make_scene(nx, ny, dt=1e-3)
    sc.init_pos[:] = rng.normal(size=sc.init_pos.shape)
    sc.init_vel[:] = rng.normal(size=sc.init_vel.shape)
    return sc


@pytest.fixture
def two_ranges():
    """An array of 6,400 nodes whose ends lie in two page-locked ranges, with pageable memory in between."""
    import torch
    n, page = 6400, max(mmap.PAGESIZE, 65536)
    raw = np.frombuffer(mmap.mmap(-1, 4 * page), np.uint8)
    at = -raw.ctypes.data % page
    rt = torch.cuda.cudart()
    ends = [raw.ctypes.data + at, raw.ctypes.data + at + 2 * page]
    for p in ends:
        assert int(rt.cudaHostRegister(p, page, 0)) == 0
    yield raw[at + page - 4096:][:12 * n].view(np.float32).reshape(n, 3)
    for p in ends:
        assert int(rt.cudaHostUnregister(p)) == 0


def test_array_over_two_page_locked_ranges(cloth_lib, two_ranges):
    sc = scene(80, 80)
    with cloth_lib.Cloth(sc) as cl:
        for k in range(2):
            two_ranges[:] = 0.0
            p, _ = cl.read(vel=False, out_pos=two_ranges)
            assert p is two_ranges and np.array_equal(p, sc.init_pos)


@pytest.mark.parametrize("nx,ny", [(7, 5), (127, 87)])
@pytest.mark.parametrize("page_locked", [True, False])
def test_arrays_off_the_float_boundary(cloth_lib, nx, ny, page_locked):
    import torch
    n = nx * ny

    def array():
        raw = torch.empty(12 * n + 4, dtype=torch.uint8)
        raw = (raw.pin_memory() if page_locked else raw).numpy()
        a = raw[1:1 + 12 * n].view(np.float32).reshape(n, 3)
        assert a.ctypes.data % 4 == 1
        return a

    sc, p, v = scene(nx, ny), array(), array()
    with cloth_lib.Cloth(sc) as cl:
        cl.read(out_pos=p, out_vel=v)
        assert np.array_equal(p, sc.init_pos) and np.array_equal(v, sc.init_vel)
        cl.set_state(v, p)
        got = cl.read()
    assert np.array_equal(got[0], sc.init_vel) and np.array_equal(got[1], sc.init_pos)


@pytest.mark.parametrize("nx,ny", [(7, 5), (127, 87)])
def test_device_array_is_left_to_the_driver(cloth_lib, nx, ny):
    """cloth_read into device memory: an error code or the driver's copy, not a store by the host."""
    import torch
    sc, lib = scene(nx, ny), cloth_lib.capi.lib()
    out = torch.zeros((nx * ny, 3), device="cuda")
    torch.cuda.synchronize()
    with cloth_lib.Cloth(sc) as cl:
        rc = lib.cloth_read(cl.h, C.cast(out.data_ptr(), C.POINTER(C.c_float)), None)
        if rc == 0:
            assert np.array_equal(out.cpu().numpy(), sc.init_pos)
        else:
            assert rc == -3 and not out.any()  # CLOTH_ERR_CUDA


def test_reads_at_the_same_time(cloth_lib):
    """Reads share page-locked buffers, each taken for one read; twelve threads, more than are kept."""
    scs = [scene(20 + i, 30, seed=i) for i in range(24)]
    cls = [cloth_lib.Cloth(sc) for sc in scs]

    def work(t):
        for k in range(60):
            i = 2 * t + k % 2
            p, v = cls[i].read()
            assert np.array_equal(p, scs[i].init_pos) and np.array_equal(v, scs[i].init_vel)

    with ThreadPoolExecutor(12) as pool:
        list(pool.map(work, range(12)))
    for cl in cls:
        cl.close()
