"""Infinite output adjoints: a spring that does not exist, or whose ends
coincide, has no terms in the reverse pass whatever its ends' adjoints are, so
what its nodes have that is finite stays finite."""
import numpy as np
import pytest
import torch

from helpers import make_scene

pytestmark = pytest.mark.gpu


def grads(P, sc, gpos):
    capi = P.capi
    n = sc.n
    from cloth_scenes import spring_count
    S = max(spring_count(sc.nx, sc.ny), 1)
    gks, gkd, gv0 = (torch.full(s, 7.0, device="cuda") for s in ((S,), (S,), (n, 3)))
    g = torch.tensor(gpos, dtype=torch.float32, device="cuda").contiguous()
    with P.Cloth(sc) as cl:
        r = capi.cloth_rollout_create(cl.h, 3, 2)
        capi.cloth_rollout_forward(r, 0, 0, 0, 0, 0)
        capi.cloth_rollout_backward(r, g.data_ptr(), 0, gks.data_ptr(), gkd.data_ptr(), gv0.data_ptr())
        capi.cloth_rollout_destroy(r)
    return gks.cpu().numpy(), gkd.cpu().numpy(), gv0.cpu().numpy()


def test_node_without_springs(cloth_lib):
    sc = make_scene(1, 1, dt=1e-3, gravity=(0.0, -9.81, 0.0))
    _, _, gv = grads(cloth_lib, sc, [[np.inf, 1.0, -2.0]])
    assert gv[0, 0] == np.inf
    np.testing.assert_allclose(gv[0, 1:], [3e-3, -6e-3], rtol=1e-6)


def test_coincident_nodes(cloth_lib):
    # two nodes in one place, at rest relative to each other: the only spring is degenerate in every substep
    sc = make_scene(2, 1, dt=1e-3, gravity=(0.0, -9.81, 0.0), ks=(5.0, 5.0, 5.0), kd=(0.1, 0.1, 0.1),
                    pos=np.zeros((2, 3)))
    gks, gkd, gv = grads(cloth_lib, sc, [[np.inf, 1.0, -2.0], [1.0, 2.0, 3.0]])
    assert gks[0] == 0.0 and gkd[0] == 0.0
    assert gv[0, 0] == np.inf
    np.testing.assert_allclose(gv[0, 1:], [3e-3, -6e-3], rtol=1e-6)
    np.testing.assert_allclose(gv[1], [3e-3, 6e-3, 9e-3], rtol=1e-6)
