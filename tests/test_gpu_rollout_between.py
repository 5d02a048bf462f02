"""What happens to a cloth between a rollout's forward and reverse pass: the
reverse pass takes the segments that the forward pass recorded only while the
cloth's surface model and constants are the ones they were recorded with.  Over
more than two segments a second reverse pass recomputes all of them, so it shows
what the first should have used."""
import numpy as np
import pytest
import torch

import cloth_scenes as cs
from test_gpu_node_kernel import per_spring, scene

pytestmark = pytest.mark.gpu


def tensors(sc, scale=1.0):
    return [torch.tensor(a * np.float32(s), device="cuda", requires_grad=True)
            for a, s in ((sc.ks_spring, scale), (sc.kd_spring, 1.0), (sc.init_vel, 1.0))]


@pytest.mark.parametrize("graph", [True, False])
@pytest.mark.parametrize("change", ["model", "constants"])
def test_change_before_the_reverse_pass(cloth_lib, graph, change):
    from paper_2507_11794_gb300.rollout import Rollout
    sc = per_spring(scene(23, 19, mesh=True, wind=False))
    with cloth_lib.Cloth(sc, flags=0 if graph else cloth_lib.capi.CLOTH_FLAG_NO_GRAPH) as cl:
        ro, other = Rollout(cl, 4, 1), Rollout(cl, 2, 1)
        args = tensors(sc)

        def loss():
            pos, vel = ro(*args)
            return (pos ** 2).sum() + vel.sum()

        plain = torch.autograd.grad(loss(), args)
        L = loss()
        if change == "model":
            cl.set_mesh(*cs.sphere_mesh(3, 0.3005))
        else:
            with torch.no_grad():
                other(*[a.detach() for a in tensors(sc, 1.3)])
        first = torch.autograd.grad(L, args, retain_graph=True)
        again = torch.autograd.grad(L, args)
        ro.close()
        other.close()
    for a, b in zip(first, again):
        assert torch.equal(a, b)
    assert not torch.equal(first[2], plain[2])  # the change matters


@pytest.mark.parametrize("steps,every", [(1, 1), (3, 3), (4, 2), (5, 2), (7, 3)])
@pytest.mark.parametrize("substeps", [1, 2])
@pytest.mark.parametrize("graph", [True, False])
def test_forward_with_and_without_recording(cloth_lib, steps, every, substeps, graph):
    """Both forward passes leave the same state, and the reverse pass gives the
    same gradients after either, also in turn on one rollout."""
    capi = cloth_lib.capi
    sc = per_spring(scene(23, 19, mesh=True, wind=True))
    sc.substeps = substeps
    ks, kd, v0 = (t.detach() for t in tensors(sc))
    seed = torch.randn((sc.n, 3), device="cuda", generator=torch.Generator("cuda").manual_seed(0))
    runs = []
    with cloth_lib.Cloth(sc, flags=0 if graph else capi.CLOTH_FLAG_NO_GRAPH) as cl:
        r = capi.cloth_rollout_create(cl.h, steps, every)
        for record in (False, True, True, False):
            forward = capi.cloth_rollout_forward_record if record else capi.cloth_rollout_forward
            pos, vel = torch.empty_like(v0), torch.empty_like(v0)
            grads = [torch.empty_like(t) for t in (ks, kd, v0)]
            forward(r, ks.data_ptr(), kd.data_ptr(), v0.data_ptr(), pos.data_ptr(), vel.data_ptr())
            held = cl.read()
            capi.cloth_rollout_backward(r, seed.data_ptr(), seed.data_ptr(), *(g.data_ptr() for g in grads))
            after = cl.read()
            runs.append([pos, vel, *grads, *(torch.from_numpy(a).cuda() for a in (*held, *after))])
        capi.cloth_rollout_destroy(r)
    assert torch.equal(runs[0][0], runs[0][5]) and torch.equal(runs[0][0], runs[0][7])
    for other in runs[1:]:
        for a, b in zip(runs[0], other):
            assert torch.equal(a, b)


def test_null_rollout(cloth_lib):
    capi = cloth_lib.capi
    assert capi.lib().cloth_rollout_forward_record(None, None, None, None, None, None) == capi.CLOTH_ERR_INVALID_ARG
