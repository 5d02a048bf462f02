"""The collision of a substep in its two places, the one-kernel substep
(cloth_step of a small cloth) and the list pass behind the walk
(cloth_profile_substeps, which always runs those two): against the FP64 oracle
and bit for bit against each other, over the scenes of test_gpu_collide_lists,
at the list lengths where the pass changes its lanes per node (152 SMs, 456 CTAs:
eight up to 14,592 nodes, two up to 58,368, one beyond), with crowded cells and
long paths in each, and over cells whose entries end just before, at and after
the filter's batches (8, 16, 32 and the 96 of one lane)."""
import numpy as np
import pytest

from helpers import make_scene
from test_gpu_collide_lists import CASES as SCENES
from test_gpu_collide_lists import crowded, wavy
from test_gpu_parity import TOL_1, _explained_by_rounding

pytestmark = pytest.mark.gpu

CASES = dict(SCENES)
CASES.update({
    "eight_lanes_last": (152, 96, lambda: wavy(40, 1.0, 0.01, 41), 3.0, 1e-3, 0.0),
    "two_lanes_from": (139, 105, lambda: wavy(40, 1.0, 0.01, 42), 3.0, 1e-3, 0.0),
    "two_lanes_last": (228, 256, lambda: wavy(60, 1.0, 0.01, 43), 3.0, 1e-3, 0.0),
    "one_lane_from": (278, 210, lambda: wavy(60, 1.0, 0.01, 44), 3.0, 1e-3, 0.0),
    "crowded_cell_two_lanes": (160, 120, lambda: crowded(45), 3.0, 1e-3, 0.0),
    "crowded_cell_last_fused": (300, 250, lambda: crowded(46), 3.0, 1e-3, 0.0),
    "long_paths_two_lanes": (160, 120, lambda: wavy(30, 1.0, 0.05, 47), 30.0, 1e-2, 0.0),
    "long_paths_one_lane": (270, 230, lambda: wavy(30, 1.0, 0.05, 48), 30.0, 1e-2, 0.0),
    "behind_the_start_two_lanes": (160, 120, lambda: wavy(30, 1.0, 0.01, 49), 3.0, 1e-3, -5e-3),
})


def both_forms(P, sc):
    got = []
    for run in ("step", "profile_substeps"):
        with P.Cloth(sc) as cl:
            getattr(cl, run)(1)
            got.append((*cl.read(), cl.collision_stats()))
    (p, v, s), (p2, v2, s2) = got
    np.testing.assert_array_equal(p, p2)
    np.testing.assert_array_equal(v, v2)
    assert s == s2
    return p, s


def check(P, oracle, sc):
    p, stats = both_forms(P, sc)
    grid, clo = oracle.Grid(sc.mesh_verts, sc.mesh_tris), oracle.Cloth(sc)
    x, _, hits = oracle.step(clo, sc.init_pos, sc.init_vel, 0, 1, grid, want_hits=True)
    err = np.abs(p.astype(np.float64) - x).max(axis=1)
    off = np.nonzero(err > TOL_1)[0]
    for i in off:
        assert _explained_by_rounding(oracle, clo, grid, sc.init_pos, sc.init_vel, i, p[i].astype(np.float64),
                                      TOL_1), (int(i), float(err[i]))
    assert len(off) <= 2 + sc.n // 500
    return hits, stats


@pytest.mark.parametrize("case", CASES)
def test_forms_match(cloth_lib, oracle_lib, case):
    nx, ny, mesh, speed, dt, t_min = CASES[case]
    v, t = mesh()
    lo, hi = v.min(0).astype(float), np.minimum(v.max(0), 1.0).astype(float)
    rng = np.random.default_rng(19)
    n = nx * ny
    pos = np.stack([rng.uniform(lo[0] + 0.1, hi[0] - 0.1, n), rng.uniform(lo[1], hi[1], n),
                    rng.uniform(lo[2] + 0.1, hi[2] - 0.1, n)], axis=1)
    if case.startswith("crowded"):  # many of them near the small triangles
        pos[::3] = np.array([0.5, 0.0, 0.5]) + rng.uniform(-0.012, 0.012, pos[::3].shape)
    d = rng.normal(size=(n, 3))
    vel = speed * d / np.linalg.norm(d, axis=1, keepdims=True)
    hits, stats = check(cloth_lib, oracle_lib, make_scene(nx, ny, pos=pos, vel=vel, mesh=(v, t), dt=dt, t_min=t_min))
    assert stats[0] == n
    if n > 100:
        assert (hits > 0).sum() > n // 200


@pytest.mark.parametrize("entries", [1, 3, 4, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33, 40, 64, 95, 96, 97])
@pytest.mark.parametrize("nx,ny", [(20, 16), (160, 120), (256, 220)])
def test_entries_of_a_cell(cloth_lib, oracle_lib, nx, ny, entries):
    """A stack of equal triangles in one cell, crossed by paths of all lengths: every entry of the
    cell is a candidate, and up to all of them are hits."""
    rng = np.random.default_rng(entries)
    y = 1e-3 * np.arange(entries)
    v = np.array([[[0.0, h, 0.0], [1.0, h, 0.0], [0.0, h, 1.0]] for h in y], np.float32).reshape(-1, 3)
    t = rng.permutation(3 * entries).reshape(-1, 3).astype(np.int32)
    v[t.reshape(-1)] = v.copy()  # triangles listed in another order than they are stacked
    n = nx * ny
    top = y[-1] + 1e-3
    pos = np.stack([rng.uniform(0.02, 0.45, n), rng.uniform(-1e-3, top, n), rng.uniform(0.02, 0.45, n)], axis=1)
    vel = np.stack([rng.uniform(-1, 1, n), rng.uniform(-1, 1, n) * top / 1e-3, rng.uniform(-1, 1, n)], axis=1)
    sc = make_scene(nx, ny, pos=pos, vel=vel, mesh=(v, t), dt=1e-3)
    if n < 10000:
        hits, stats = check(cloth_lib, oracle_lib, sc)
        assert hits.max() > entries // 2
    else:
        _, stats = both_forms(cloth_lib, sc)
    assert stats[1] >= entries * stats[0] // 2 and stats[2] > n // 10
