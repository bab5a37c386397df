"""LR steps of small sets, all passes in one launch by a cluster of blocks,
against the persistent solver's grid (other lanes per particle and another
barrier): the same bits, at the edges of a warp's, a block's and the cluster's
particles, one above, without stabilization or solver passes, with grain
materials, and in a batch."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


def _scene(n, seed):
    sc = scenes.stir(scenes.column(seed=scenes.SEED_BASE + 90 + seed, n_low=n, ratio=2, z0=0.012), seed=seed, v_scale=0.2)
    return sc


def _steps(gs, sc, solver, iters, materials=False, **kw):
    ctx = gs.Context(sc, **kw)
    if materials:
        ctx.set_materials(*scenes.materials(sc, 5, "random"))
    ctx.set_lr_solver(solver)
    for _ in range(4):
        ctx.step_low(1.0 / 240.0, iters)
    ctx.frame(1.0 / 60.0, 3, iters)      # steps that begin the next one's binning
    out = [ctx.read(f) for f in (gs.GS_FIELD_LR_POS, gs.GS_FIELD_LR_VEL, gs.GS_FIELD_HR_POS)]
    ctx.close()
    return out


@pytest.mark.parametrize("n, n_stab, iters, materials", [
    (1, 2, 4, False), (4, 2, 4, False), (5, 0, 3, False), (64, 2, 0, False), (65, 1, 1, True), (700, 2, 4, True),
    (1023, 2, 5, False), (1024, 2, 4, False), (1025, 2, 4, False)])
def test_small_sets_equal_the_solver(n, n_stab, iters, materials):
    import paper_2308_01629_gb300 as gs
    sc = _scene(n, 1)
    a, b = (_steps(gs, sc, s, iters, materials, n_stab=n_stab) for s in (0, 1))
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x.view(np.uint32), y.view(np.uint32))


def test_a_small_batch_equals_the_solver():
    import paper_2308_01629_gb300 as gs
    batch = [_scene(n, k) for k, n in enumerate((130, 1, 400, 333))]
    a, b = (_steps(gs, batch, s, 4) for s in (0, 1))
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x.view(np.uint32), y.view(np.uint32))
