"""The one-kernel substep of small cloths (cloth_step) against the column walk
and the collision pass (cloth_profile_substeps, which always runs those two):
bit for bit, at grid shapes around its pairs, rows and CTAs, at the sizes where
its warps per CTA change (152 SMs: 9,728, 29,184, 77,824 and 116,736 padded
positions), with pins, wind, per-spring constants and contact, and with the edge
narrow phase.  The walk itself is held to the oracle by the parity tests."""
import numpy as np
import pytest

import cloth_scenes as cs
from helpers import make_scene

pytestmark = pytest.mark.gpu


def scene(nx, ny, mesh, wind, seed=3):
    rng = np.random.default_rng(seed)
    h = 0.9 / max(nx, ny, 2)
    sc = make_scene(nx, ny, origin=(-0.5 * (nx - 1) * h, 0.3, -0.5 * (ny - 1) * h), du=(h, 0, 0), dv=(0, 0, h), total_mass=1.0 * nx * ny / 1000,
                    ks=(400.0, 200.0, 80.0), kd=(0.4, 0.3, 0.2), gravity=(0.3, -9.81, 0.1), dt=1 / 2400, substeps=2)
    r = np.linalg.norm(sc.init_pos[:, [0, 2]], axis=1)
    top = np.where(r < 0.29, np.sqrt(np.maximum(0.09 - r * r, 0.0)), 0.0) + 2e-4  # just above a sphere of radius 0.3
    sc.init_pos[:, 1] = top + rng.uniform(0, 3e-4, len(r))
    sc.init_vel[:] = rng.normal(0, 0.05, sc.init_vel.shape)
    sc.init_vel[:, 1] -= 1.0
    if mesh:
        sc.mesh_verts, sc.mesh_tris = cs.sphere_mesh(4, 0.3)
    if wind:
        sc.wind = cs.Wind(3.0, (0.2, 0.1, 1.0), (0.6, 0.1, 0.8), 2.0, 9.0, 0.7)
    sc.pinned[rng.integers(0, nx * ny, 1 + nx * ny // 50)] = 1
    sc.pin_velocity = (0.1, 0.0, -0.2)
    return sc


def per_spring(sc, seed=4):
    rng = np.random.default_rng(seed)
    n = cs.spring_count(sc.nx, sc.ny)
    sc.ks_spring = rng.uniform(50, 400, n).astype(np.float32)
    sc.kd_spring = rng.uniform(0.05, 0.4, n).astype(np.float32)
    return sc


def compare(P, sc, steps, flags=0):
    with P.Cloth(sc, flags=flags) as a, P.Cloth(sc, flags=flags) as b:
        a.step(steps)
        b.profile_substeps(steps * sc.substeps)
        (pa, va), (pb, vb) = a.read(), b.read()
        sa, sb = a.collision_stats(), b.collision_stats()
    np.testing.assert_array_equal(pa, pb)
    np.testing.assert_array_equal(va, vb)
    assert sa == sb
    return sa


SHAPES = [(1, 1), (2, 1), (1, 3), (3, 2), (5, 5), (64, 1), (1, 70), (65, 2), (2, 65), (31, 33), (66, 7), (130, 5)]


@pytest.mark.parametrize("nx,ny", SHAPES)
@pytest.mark.parametrize("kind", ["plain", "springs", "wind"])
def test_shapes(cloth_lib, nx, ny, kind):
    sc = scene(nx, ny, mesh=False, wind=kind == "wind")
    if kind == "springs" and cs.spring_count(nx, ny):
        per_spring(sc)
    compare(cloth_lib, sc, 3)


# padded positions: 9,728 and 9,744; 29,184 and 29,216; 77,824 and 77,888; 116,736
SIZES = [(152, 64), (28, 348), (192, 152), (88, 332), (256, 304), (16, 4868), (304, 384)]


@pytest.mark.parametrize("nx,ny", [(29, 31), *SIZES])
@pytest.mark.parametrize("springs", [False, True])
def test_contact(cloth_lib, nx, ny, springs):
    sc = scene(nx, ny, mesh=True, wind=True)
    stats = compare(cloth_lib, per_spring(sc) if springs else sc, 4)
    assert stats[2] > 0


@pytest.mark.parametrize("nx,ny", [(29, 31), (91, 80)])
def test_edges(cloth_lib, nx, ny):
    sc = scene(nx, ny, mesh=True, wind=False)
    compare(cloth_lib, sc, 3, cloth_lib.capi.CLOTH_FLAG_EDGE_COLLISION)


@pytest.mark.parametrize("nx,ny", [(21, 26), (152, 70), (200, 170), (250, 236), (256, 306)])
def test_rollout_recompute(cloth_lib, nx, ny):
    """The reverse pass recomputes its segments with the recording form: its
    gradients do not depend on the checkpoint distance."""
    import torch
    from paper_2507_11794_gb300.rollout import Rollout
    sc = per_spring(scene(nx, ny, mesh=True, wind=False))
    got = []
    for every in (1, 4):
        with cloth_lib.Cloth(sc) as cl:
            ro = Rollout(cl, 4, every)
            args = [torch.tensor(a, device="cuda", requires_grad=True)
                    for a in (sc.ks_spring, sc.kd_spring, sc.init_vel)]
            pos, vel = ro(*args)
            got.append([pos.detach().cpu(), *[g.cpu() for g in torch.autograd.grad((pos ** 2).sum() + vel.sum(), args)]])
            ro.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)


# (sides, cloths): groups of 64 positions on 152 SMs: below one, three and eight CTAs per SM, and above (the walk)
BATCHES = {"few": ((5, 17, 31), 1), "eight_warps": ((16, 33, 40), 3), "four_warps": ((24, 61, 70), 4),
           "two_warps": ((40, 61, 90), 7), "walk": ((100, 120, 121), 5)}


@pytest.mark.parametrize("case", BATCHES)
@pytest.mark.parametrize("springs", [False, True])
@pytest.mark.parametrize("mesh", [False, True])
def test_batches(cloth_lib, case, springs, mesh):
    """Every cloth of a batch as stepped alone by the walk, over an odd number
    of substeps per step (both parities)."""
    sides, times = BATCHES[case]
    scs = [scene(n + i, n, mesh, True, seed=n + i) for i in range(times) for n in sides]
    for sc in scs:
        sc.substeps, sc.dt = 3, 3 / 4800
        if springs:
            per_spring(sc)
    b = cloth_lib.ClothBatch(scs)
    b.step(1)
    b.step(2)
    total = np.zeros(3, int)
    for i, sc in enumerate(scs):
        with cloth_lib.Cloth(sc) as cl:
            cl.profile_substeps(9)
            (pa, va), (pb, vb) = b.read(i), cl.read()
            total += cl.collision_stats()
        np.testing.assert_array_equal(pa, pb)
        np.testing.assert_array_equal(va, vb)
    assert tuple(total) == b.collision_stats()
    b.close()


def test_batch_changes_form(cloth_lib):
    """Meshes set and cleared between steps take a batch from one form of the
    substep to the other (one walk variant or mixed) and back."""
    scs = [scene(30, 28, True, False, seed=i) for i in range(3)]
    b = cloth_lib.ClothBatch(scs)
    cls = [cloth_lib.Cloth(sc) for sc in scs]
    for clear in (None, 1, 2, None):
        for i, (cl, sc) in enumerate(zip(cls, scs)):
            v, t = (None, None) if i == clear else (sc.mesh_verts, sc.mesh_tris)
            cl.set_mesh(v, t)
            cloth_lib.capi.cloth_batch_set_mesh(b.h, i, v, t)
        b.step(3)
        for i, cl in enumerate(cls):
            cl.step(3)
            (pa, va), (pb, vb) = b.read(i), cl.read()
            np.testing.assert_array_equal(pa, pb)
            np.testing.assert_array_equal(va, vb)
    b.close()
    for cl in cls:
        cl.close()


@pytest.mark.parametrize("steps,every", [(3, 1), (3, 2), (4, 2), (5, 2), (6, 6)])
@pytest.mark.parametrize("graph", [True, False])
def test_rollout_reverse_twice(cloth_lib, steps, every, graph):
    """The forward pass records the last two segments; a second reverse pass
    (with more than two, of recomputed ones) and one after another forward
    pass with other inputs in between give the same gradients."""
    import torch
    from paper_2507_11794_gb300.rollout import Rollout
    sc = per_spring(scene(23, 19, mesh=True, wind=False))
    with cloth_lib.Cloth(sc, flags=0 if graph else cloth_lib.capi.CLOTH_FLAG_NO_GRAPH) as cl:
        ro = Rollout(cl, steps, every)
        args = [torch.tensor(a, device="cuda", requires_grad=True) for a in (sc.ks_spring, sc.kd_spring, sc.init_vel)]

        def loss():
            pos, vel = ro(*args)
            return (pos ** 2).sum() + vel.sum()

        L = loss()
        first = torch.autograd.grad(L, args, retain_graph=True)
        again = torch.autograd.grad(L, args)
        state = cl.read()
        with torch.no_grad():
            ro(args[0] * 1.1, args[1], args[2])
        third = torch.autograd.grad(loss(), args)
        after = cl.read()
        ro.close()
    for a, b, c in zip(first, again, third):
        assert torch.equal(a, b) and torch.equal(a, c)
    assert np.array_equal(state[0], after[0]) and np.array_equal(state[1], after[1])
