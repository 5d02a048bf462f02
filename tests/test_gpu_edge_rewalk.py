"""An edge with more hits than the edge test stores points for is walked again by
the node's gather, which has to find the same hits.  Beside five small triangles
that the edge crosses lies a large tilted one: the edge is in its plane to within
1e-7 m, but 6 to 22 mm outside its box and in the same grid cell.  The float32 test
accepts it (its errors in u and v grow as 1 / a), the candidate filter does not,
and in exact arithmetic it is missed.  Checked against the FP64 oracle."""
import numpy as np
import pytest

from helpers import make_scene

pytestmark = pytest.mark.gpu


def floats(s):
    return np.array([float.fromhex(x) for x in s.split()], np.float32)


# large triangle's vertices, the edge's ends
EDGES = [tuple(map(floats, e)) for e in (
    ("0x1.92a0ap-3 0x1.9cb16ep-4 0x1.1320fep-3", "0x1.45725p+3 0x1.21c47p-2 0x1.825b48p-2",
     "0x1.35f266p-2 0x1.918f6p+2 0x1.0bb4e8p+3", "0x1.7c0346p-3 0x1.450e8p+0 0x1.b168aap+0",
     "0x1.64e42ep-3 0x1.446e94p+0 0x1.b0937p+0"),
    ("0x1.fab2ccp-2 0x1.957a1ap-3 0x1.0e517ep-2", "0x1.406e34p+3 0x1.3634f2p-5 0x1.9d9b04p-5",
     "0x1.dc6428p-3 0x1.865c82p+2 0x1.043daap+3", "0x1.d04608p-3 0x1.d50e46p+0 0x1.38b42ep+1",
     "0x1.b99a26p-3 0x1.d45824p+0 0x1.383ac2p+1"))]


@pytest.mark.parametrize("which", range(len(EDGES)))
def test_second_walk_finds_the_same_hits(cloth_lib, oracle_lib, which):
    v0, v1, v2, S, E = EDGES[which]
    d = (E - S).astype(float)
    L = np.linalg.norm(d)
    d /= L
    n = np.array([0.0, 0.8, -0.6])  # the large triangle's plane
    n -= (n @ d) * d
    n /= np.linalg.norm(n)
    b = np.cross(d, n)
    V = [v0, v1, v2]
    for t in (0.1, 0.2, 0.3, 0.4, 0.9):  # five small triangles across the edge
        V += [S + t * L * d + 1e-3 * (np.cos(2.1 * k + 0.3) * n + np.sin(2.1 * k + 0.3) * b) for k in range(3)]
    rng = np.random.default_rng(1)
    for _ in range(1200):  # small triangles far away, which set the cell size (0.056 m)
        c = rng.uniform([2, 0.5, 0.5], [9, 5, 7])
        V += [c, c + [0.02, 0, 0], c + [0, 0.02, 0]]
    V = np.array(V, np.float32)
    T = np.arange(len(V), dtype=np.int32).reshape(-1, 3)
    off = np.array([-0.03, 0.0, 0.0]) + 0.02 * n  # the cloth's other row: away from the triangles
    sc = make_scene(2, 2, pos=np.array([S, E, S + off, E + off]), mesh=(V, T), dt=1e-3)
    grid = oracle_lib.Grid(V, T)
    assert 0 in grid.candidates_f32(S, E)  # the large triangle shares a cell with the edge
    x, _, hits = oracle_lib.step_edges(oracle_lib.Cloth(sc), sc.init_pos, sc.init_vel, 0, 1, grid, want_hits=True)
    assert hits[0] == 5 and hits[1] == 5
    with cloth_lib.Cloth(sc, flags=cloth_lib.capi.CLOTH_FLAG_EDGE_COLLISION) as cl:
        cl.step(1)
        p, _ = cl.read()
    # hit points and their mean: a few roundings of coordinates up to 3 m, below 1e-5 m; a
    # point counted twice would move the mean by 5e-4 m
    assert np.abs(p.astype(np.float64) - x).max() < 1e-5
