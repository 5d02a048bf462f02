"""The node collision pass at the edges of its forms: lists on either side of
every change of lanes per node, cells with more entries than one lane goes
through, paths over more cells than one lane goes through, hits behind the
path's start, and a grid whose coordinates leave the candidate filter less
than its full resolution.  One substep without spring forces over a wavy
surface, against the FP64 oracle: every node within 1e-5 m (the one-step
tolerance of the parity tests), or explained by float32 rounding of a
threshold as there."""
import numpy as np
import pytest

from helpers import make_scene
from test_gpu_parity import TOL_1, _explained_by_rounding

pytestmark = pytest.mark.gpu


def wavy(m, size, amp, seed):
    rng = np.random.default_rng(seed)
    g = np.linspace(0.0, size, m)
    x, z = np.meshgrid(g, g)
    v = np.stack([x, rng.uniform(-amp, amp, x.shape), z], axis=2).reshape(-1, 3)
    i = np.arange(m * m).reshape(m, m)
    t = np.concatenate([np.stack([i[:-1, :-1], i[1:, :-1], i[1:, 1:]], 2).reshape(-1, 3),
                        np.stack([i[:-1, :-1], i[1:, 1:], i[:-1, 1:]], 2).reshape(-1, 3)])
    return v.astype(np.float32), t.astype(np.int32)


def crowded(seed):
    """A wavy surface with 300 small triangles around one of its points."""
    v, t = wavy(12, 1.0, 0.02, seed)
    rng = np.random.default_rng(seed + 1)
    c = np.array([0.5, 0.0, 0.5]) + rng.uniform(-0.01, 0.01, (300, 1, 3))
    small = (c + rng.uniform(-2e-3, 2e-3, (300, 3, 3))).reshape(-1, 3).astype(np.float32)
    return np.concatenate([v, small]), np.concatenate([t, len(v) + np.arange(900, dtype=np.int32).reshape(-1, 3)])


def two_parts(seed):
    """A wavy surface and a copy 200 m away: 5,000 cells along x."""
    v, t = wavy(60, 1.0, 0.01, seed)
    return np.concatenate([v, v + np.float32([200.0, 0, 0])]), np.concatenate([t, t + len(v)]).astype(np.int32)


CASES = {
    # nx, ny, mesh, speed (m/s), dt, t_min
    "one_node": (1, 1, lambda: wavy(9, 1.0, 0.02, 0), 3.0, 1e-3, 0.0),
    "ragged": (7, 5, lambda: wavy(9, 1.0, 0.02, 1), 3.0, 1e-3, 0.0),
    # 152 SMs: 608 CTAs, eight lanes per node up to 19,456 nodes, two up to 77,824
    "eight_lanes_full": (152, 128, lambda: wavy(40, 1.0, 0.01, 2), 3.0, 1e-3, 0.0),
    "two_lanes_first": (139, 140, lambda: wavy(40, 1.0, 0.01, 3), 3.0, 1e-3, 0.0),
    "two_lanes_full": (304, 256, lambda: wavy(60, 1.0, 0.01, 4), 3.0, 1e-3, 0.0),
    "one_lane_first": (278, 281, lambda: wavy(60, 1.0, 0.01, 5), 3.0, 1e-3, 0.0),
    "crowded_cell": (61, 47, lambda: crowded(6), 3.0, 1e-3, 0.0),
    "crowded_cell_one_lane": (300, 270, lambda: crowded(7), 3.0, 1e-3, 0.0),
    "long_paths": (40, 31, lambda: wavy(30, 1.0, 0.05, 8), 30.0, 1e-2, 0.0),
    "behind_the_start": (60, 50, lambda: wavy(30, 1.0, 0.01, 9), 3.0, 1e-3, -5e-3),
    "long_grid": (60, 50, lambda: two_parts(10), 3.0, 1e-3, 0.0),
}


@pytest.mark.parametrize("case", CASES)
def test_one_substep_matches_oracle(cloth_lib, oracle_lib, case):
    nx, ny, mesh, speed, dt, t_min = CASES[case]
    v, t = mesh()
    lo, hi = v.min(0).astype(float), np.minimum(v.max(0), 1.0).astype(float)
    rng = np.random.default_rng(17)
    n = nx * ny
    pos = np.stack([rng.uniform(lo[0] + 0.1, hi[0] - 0.1, n), rng.uniform(lo[1], hi[1], n),
                    rng.uniform(lo[2] + 0.1, hi[2] - 0.1, n)], axis=1)
    if case.startswith("crowded"):  # many of them near the small triangles
        pos[::3] = np.array([0.5, 0.0, 0.5]) + rng.uniform(-0.012, 0.012, pos[::3].shape)
    d = rng.normal(size=(n, 3))
    vel = speed * d / np.linalg.norm(d, axis=1, keepdims=True)
    sc = make_scene(nx, ny, pos=pos, vel=vel, mesh=(v, t), dt=dt, t_min=t_min)
    grid = oracle_lib.Grid(v, t)
    clo = oracle_lib.Cloth(sc)
    x, _, hits = oracle_lib.step(clo, sc.init_pos, sc.init_vel, 0, 1, grid, want_hits=True)
    with cloth_lib.Cloth(sc) as cl:
        cl.step(1)
        p, _ = cl.read()
        listed, tested, hit = cl.collision_stats()
    assert listed == n
    err = np.abs(p.astype(np.float64) - x).max(axis=1)
    off = np.nonzero(err > TOL_1)[0]
    for i in off:
        assert _explained_by_rounding(oracle_lib, clo, grid, sc.init_pos, sc.init_vel, i, p[i].astype(np.float64),
                                      TOL_1), (int(i), float(err[i]))
    print(f"{case}: {n} nodes, {tested} candidates, {hit} hits, {len(off)} explained by rounding")
    assert len(off) <= 2 + n // 500
    if n > 100:
        assert (hits > 0).sum() > n // 200


# edge narrow phase: eight lanes per edge up to 6,485 listed nodes on 152 SMs, one beyond; a steep sheet
# whose edges span up to 12 cells, some more than one lane goes through
EDGE_CASES = {"eight_lanes": (81, 80, 60), "one_lane": (82, 80, 60), "long_edges": (30, 26, 90)}


@pytest.mark.parametrize("case", EDGE_CASES)
def test_edge_substep_matches_oracle(cloth_lib, oracle_lib, case):
    nx, ny, m = EDGE_CASES[case]
    v, t = wavy(m, 1.0, 0.01, 21)
    rng = np.random.default_rng(22)
    h = 0.8 / nx
    x, z = np.meshgrid(0.1 + h * np.arange(nx), 0.1 + h * np.arange(ny))
    pos = np.stack([x, rng.uniform(-0.03, 0.03, x.shape), z], axis=2)
    vel = rng.normal(size=(nx * ny, 3)) * 0.5
    sc = make_scene(nx, ny, pos=pos, vel=vel, mesh=(v, t), dt=1e-3)
    grid = oracle_lib.Grid(v, t)
    clo = oracle_lib.Cloth(sc)
    xo, _, hits = oracle_lib.step_edges(clo, sc.init_pos, sc.init_vel, 0, 1, grid, want_hits=True)
    with cloth_lib.Cloth(sc, flags=cloth_lib.capi.CLOTH_FLAG_EDGE_COLLISION) as cl:
        cl.step(1)
        p, _ = cl.read()
    S = sc.init_pos.astype(np.float64)
    err = np.abs(p.astype(np.float64) - xo).max(axis=1)
    # a hit decided within float32 rounding of its threshold may go either way (as in test_gpu_edges)
    bound = np.linalg.norm(xo - S, axis=1) + np.linalg.norm(p.astype(np.float64) - S, axis=1)
    print(f"{case}: {int((hits > 0).sum())} nodes affected, {int((err > 1e-5).sum())} beyond 1e-5")
    assert np.all(err <= np.maximum(1e-5, 1.01 * bound + 1e-7))
    assert (err > 1e-5).mean() <= 0.02
    assert (hits > 0).mean() > 0.3


@pytest.mark.parametrize("nx,ny", [(41, 37), (90, 85)])
def test_edge_statistics_count_every_edge(cloth_lib, nx, ny):
    # a flat sheet above the surface, inside its cells: nothing hits, so the
    # candidates of every edge follow from the final positions and the grid
    v, t = wavy(40, 1.0, 0.01, 31)
    h = 0.8 / nx
    x, z = np.meshgrid(0.1 + h * np.arange(nx), 0.1 + h * np.arange(ny))
    sc = make_scene(nx, ny, pos=np.stack([x, np.full_like(x, 0.0100), z], axis=2), mesh=(v, t), dt=1e-3)
    with cloth_lib.Cloth(sc, flags=cloth_lib.capi.CLOTH_FLAG_EDGE_COLLISION) as cl:
        cl.step(1)
        p, _ = cl.read()
        listed, tested, hits = cl.collision_stats()
        i = cl.info()
        start, _ = cl.grid()
    assert hits == 0 and listed == nx * ny
    dims = np.array(i.grid_dims)
    cell = np.floor((p - np.float32(i.grid_origin)) * np.float32(i.grid_inv)).astype(int).reshape(ny, nx, 3)
    count = np.diff(start).reshape(dims[::-1])
    total = 0
    for dr, dc in ((0, 1), (1, 0), (1, 1)):
        a, b = cell[:ny - dr, :nx - dc].reshape(-1, 3), cell[dr:, dc:].reshape(-1, 3)
        for lo, hi in zip(np.minimum(a, b), np.maximum(a, b)):
            total += int(count[lo[2]:hi[2] + 1, lo[1]:hi[1] + 1, lo[0]:hi[0] + 1].sum())
    assert tested == total
