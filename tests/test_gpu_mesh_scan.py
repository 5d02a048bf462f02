"""Meshes on both sides of the size from which cloth_set_mesh looks them over
on the device (4,096 triangles): the grid bit for bit the oracle's, and bad
input refused with the same code and message, the previous mesh kept."""
import numpy as np
import pytest

import cloth_scenes as cs
from helpers import make_scene

pytestmark = pytest.mark.gpu


def mesh(nt, seed, scale=1.0, offset=0.0):
    rng = np.random.default_rng(seed)
    v = rng.uniform(-1, 1, (nt // 2 + 3, 3)) * scale + offset
    base = rng.integers(0, len(v) - 2, nt)
    t = np.stack([base, base + 1, base + 2], axis=1)
    # neighbouring vertices lie close together, so that triangles are small
    v = np.cumsum(rng.normal(0, 0.02 * scale, v.shape), axis=0) + offset
    return v.astype(np.float32), t.astype(np.int32)


@pytest.mark.parametrize("nt,scale,offset", [(4095, 1.0, 0.0), (4096, 1.0, 0.0), (4097, 1e-3, -7.0), (20001, 30.0, 5.0)])
def test_grid_is_the_oracles(cloth_lib, oracle_lib, nt, scale, offset):
    v, t = mesh(nt, nt, scale, offset)
    g = oracle_lib.Grid(v, t)
    with cloth_lib.Cloth(make_scene(3, 3)) as cl:
        cl.set_mesh(v, t)
        i = cl.info()
        start, ids = cl.grid()
    assert tuple(i.grid_dims) == tuple(g.params["dims"])
    assert i.grid_h == np.float32(g.params["h"]) and tuple(i.grid_origin) == tuple(np.float32(g.params["origin"]))
    assert np.array_equal(start, g.cell_start()) and np.array_equal(ids, g.tri_ids())


@pytest.mark.parametrize("nt", [4000, 9000])
def test_bad_meshes_are_refused(cloth_lib, nt):
    v, t = mesh(nt, 1)
    lib = cloth_lib.capi
    with cloth_lib.Cloth(make_scene(3, 3)) as cl:
        cl.set_mesh(*cs.sphere_mesh(2, 0.3))
        before = cl.grid()
        for place, value in (((nt - 1, 2), len(v)), ((17, 1), -1), ((0, 0), 2 ** 31 - 1)):
            bad = t.copy()
            bad[nt // 2, 0] = len(v) + 5  # the first bad position is the one reported
            bad[place] = value
            flat = bad.reshape(-1)
            first = int(np.nonzero((flat < 0) | (flat >= len(v)))[0][0])
            with pytest.raises(cloth_lib.ClothError) as e:
                cl.set_mesh(v, bad)
            assert e.value.code == lib.CLOTH_ERR_BAD_MESH
            assert f"triangle index {flat[first]} at {first} out of range [0, {len(v)})" in str(e.value)
        for x in (np.nan, np.inf, -np.inf):
            bad = v.copy()
            bad[-1, 2] = bad[5, 1] = x
            with pytest.raises(cloth_lib.ClothError) as e:
                cl.set_mesh(bad, t)
            assert e.value.code == lib.CLOTH_ERR_BAD_MESH and "non-finite vertex coordinate at 16" in str(e.value)
        after = cl.grid()
        assert np.array_equal(before[0], after[0]) and np.array_equal(before[1], after[1])
        cl.step(1)
        cl.sync()
