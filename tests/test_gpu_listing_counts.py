"""Substeps that list nodes for the collision pass and substeps that do not, in
turn: the listing counts are per parity of the substep, and each substep starts
with an empty list whatever form the substeps before it had.  The list holds
exactly one entry per node, and here every node is listed, so one left-over
entry would not fit.  cloth_profile_substeps always lists; cloth_step of a small
cloth with a surface model does not, nor does one without a model."""
import numpy as np
import pytest

from helpers import floor_mesh, make_scene

pytestmark = pytest.mark.gpu


def scene(nx, ny):
    """A sheet lying on the floor: every node within the mesh's box, most of them in contact."""
    h = 0.9 / max(nx, ny)
    rng = np.random.default_rng(nx)
    sc = make_scene(nx, ny, origin=(0.05, 0.0, 0.05), du=(h, 0, 0), dv=(0, 0, h), total_mass=nx * ny / 1000,
                    ks=(100.0, 50.0, 20.0), kd=(0.1, 0.1, 0.1), gravity=(0.0, -9.81, 0.0), dt=1 / 2400)
    sc.init_pos[:, 1] = rng.uniform(1e-5, 2e-4, nx * ny)
    sc.init_vel[:] = rng.normal(0.0, 0.02, sc.init_vel.shape)
    v, t = floor_mesh()
    # a vertex above and one below the sheet, so that the mesh's box contains it
    sc.mesh_verts = np.concatenate([v, np.float32([[0.0, 0.5, 0.0], [0.0, -0.5, 0.0], [0.0, 0.5, 0.01]])])
    sc.mesh_tris = np.concatenate([t, np.int32([[4, 5, 6]])])
    return sc


# padded positions per 64: one CTA, one per SM, and the largest forms that do not list (152 SMs: 77,824 positions)
SIZES = [(5, 4), (96, 100), (256, 300)]


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("graph", [True, False])
def test_profile_and_step_in_turn(cloth_lib, nx, ny, graph):
    P, sc = cloth_lib, scene(nx, ny)
    flags = 0 if graph else P.capi.CLOTH_FLAG_NO_GRAPH
    with P.Cloth(sc, flags=flags) as a, P.Cloth(sc) as b:
        done = 0
        for steps in (1, 3, 1, 2, 1):  # an odd number of substeps between two listings, mostly
            a.profile_substeps(1)
            a.step(steps)
            done += 1 + steps
        a.profile_substeps(2)
        b.profile_substeps(done + 2)
        (pa, va), (pb, vb) = a.read(), b.read()
        sa, sb = a.collision_stats(), b.collision_stats()
    assert sa == sb
    assert sa[0] == nx * ny * (done + 2) and sa[2] > 0
    np.testing.assert_array_equal(pa, pb)
    np.testing.assert_array_equal(va, vb)


@pytest.mark.parametrize("edges,atomic", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("free", [1, 2])
def test_model_taken_away_and_set_again(cloth_lib, edges, atomic, free):
    """Listing substeps, `free` substeps without a model, listing substeps: as
    two cloths, the second created in the state that the first had."""
    P, sc = cloth_lib, scene(31, 23)
    flags = (P.capi.CLOTH_FLAG_EDGE_COLLISION if edges else 0) | (P.capi.CLOTH_FLAG_ATOMIC_SPRINGS if atomic else 0)
    with P.Cloth(sc, flags=flags) as a, P.Cloth(sc, flags=flags) as b:
        a.profile_substeps(1)
        a.set_mesh(None, None)
        a.step(free)
        a.set_mesh(sc.mesh_verts, sc.mesh_tris)
        p, v = a.read()
        before = a.collision_stats()
        a.profile_substeps(3)
        b.set_state(p, v)
        b.profile_substeps(3)
        (pa, va), (pb, vb) = a.read(), b.read()
        sa, sb = a.collision_stats(), b.collision_stats()
    listed = sa[0] - before[0]
    assert listed == sb[0] and sb[0] <= 3 * sc.n
    if not atomic:  # the atomic forces' order of summation is free
        assert tuple(x - y for x, y in zip(sa, before)) == sb
        np.testing.assert_array_equal(pa, pb)
        np.testing.assert_array_equal(va, vb)


@pytest.mark.parametrize("nx,ny", [(31, 23), (150, 131)])
def test_atomic_forces_with_edges(cloth_lib, nx, ny):
    """Both flags together: the edge narrow phase alone fills the list.  Without
    spring forces the two force paths round alike, so the results are those of
    the edge flag alone, bit for bit."""
    P, sc = cloth_lib, scene(nx, ny)
    sc.ks = sc.kd = (0.0, 0.0, 0.0)
    got = []
    for flags in (P.capi.CLOTH_FLAG_EDGE_COLLISION, P.capi.CLOTH_FLAG_EDGE_COLLISION | P.capi.CLOTH_FLAG_ATOMIC_SPRINGS):
        with P.Cloth(sc, flags=flags) as cl:
            cl.step(3)
            got.append((*cl.read(), cl.collision_stats()))
    (pa, va, sa), (pb, vb, sb) = got
    assert sa == sb and sa[0] == 3 * sc.n and sa[2] > 0
    np.testing.assert_array_equal(pa, pb)
    np.testing.assert_array_equal(va, vb)
