"""cloth_batch_tune and the two forms of a batch's substep: its settings belong
to the persistent walk, so a batch of small cloths keeps the ones it has and says
that it timed one form; the state is as before in either."""
import numpy as np
import pytest

import cloth_scenes as cs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("small", [True, False])
def test_tuning(cloth_lib, small):
    sides = (24, 31) if small else (300, 310)  # 310 x 310 padded positions alone are beyond the one-launch form
    scs = [cs.small_collision_scene(n, level=2, gap=0.004, seed=n) for n in sides]
    b = cloth_lib.ClothBatch(scs)
    ref = cloth_lib.ClothBatch(scs)
    b.set_tuning(5, 3)
    b.step(1)
    t = b.tune(4)
    assert t.us_per_substep > 0.0
    if small:
        assert (t.rows_per_warp, t.walk_ctas_per_sm, t.candidates) == (5, 3, 1)
    else:
        assert t.candidates > 7
    now = b.tuning()
    assert (now.rows_per_warp, now.walk_ctas_per_sm) == (t.rows_per_warp, t.walk_ctas_per_sm)
    b.step(2)
    ref.step(3)
    for i in range(len(scs)):
        for x, y in zip(b.read(i), ref.read(i)):
            np.testing.assert_array_equal(x, y)
    assert b.collision_stats() == ref.collision_stats()
    b.close()
    ref.close()
