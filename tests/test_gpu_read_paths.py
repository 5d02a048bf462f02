"""State in and out of host memory over its paths: page-locked arrays (written
and read by the kernels), small pageable ones (a page-locked buffer in between)
and large pageable ones (the driver's copies), each alone and mixed, around the
size where the pageable path changes (10,922 nodes), for cloths and batches."""
import numpy as np
import pytest

import cloth_scenes as cs
from helpers import make_scene

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (3, 5), (127, 86), (127, 87), (300, 41)]  # 10,922 and 11,049 nodes in the middle


def scene(nx, ny, seed=1):
    rng = np.random.default_rng(seed)
    sc = make_scene(nx, ny, dt=1e-3)
    sc.init_pos[:] = rng.normal(size=sc.init_pos.shape)
    sc.init_vel[:] = rng.normal(size=sc.init_vel.shape)
    return sc


def pinned(n):
    import torch
    return torch.empty((n, 3), dtype=torch.float32).pin_memory().numpy()


@pytest.mark.parametrize("nx,ny", SHAPES)
def test_cloth(cloth_lib, nx, ny):
    sc, n = scene(nx, ny), nx * ny
    with cloth_lib.Cloth(sc) as cl:
        for make in (lambda n: np.empty((n, 3), np.float32), pinned):
            for pos, vel in ((True, True), (True, False), (False, True)):
                p, v = cl.read(pos, vel, make(n) if pos else None, make(n) if vel else None)
                assert p is None or np.array_equal(p, sc.init_pos)
                assert v is None or np.array_equal(v, sc.init_vel)
        p, v = cl.read(out_pos=pinned(n))  # one of each
        assert np.array_equal(p, sc.init_pos) and np.array_equal(v, sc.init_vel)
        x, y = pinned(n), pinned(n)
        x[:], y[:] = sc.init_vel, sc.init_pos
        cl.set_state(x, y)
        assert np.array_equal(cl.read()[0], sc.init_vel) and np.array_equal(cl.read()[1], sc.init_pos)
        cl.set_state(sc.init_pos, None)
        cl.set_state(None, x)
        p, v = cl.read()
        assert np.array_equal(p, sc.init_pos) and np.array_equal(v, sc.init_vel)
        x[-1, 2] = np.nan  # the flags come with the state
        cl.set_state(x)
        cl.step(1)
        with pytest.raises(cloth_lib.ClothError):
            cl.read()


def test_batch(cloth_lib):
    scs = [scene(nx, ny, 5 + i) for i, (nx, ny) in enumerate(SHAPES)]
    b = cloth_lib.ClothBatch(scs)
    for i, sc in enumerate(scs):
        p, v = b.read(i)
        assert np.array_equal(p, sc.init_pos) and np.array_equal(v, sc.init_vel)
        x = pinned(sc.n)
        x[:] = sc.init_vel
        b.set_state(i, x)
        assert np.array_equal(b.read(i)[0], sc.init_vel)
    b.close()
