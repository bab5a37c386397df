"""The library's rollout (gs_rollout_forward / gs_rollout_backward): what its
arguments may be."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu
DT = 1.0 / 120.0


def _ins(sc):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(sc[k])).cuda() for k in ("lr_pos", "lr_vel", "hr_pos", "hr_vel")]


def test_step_lengths_that_the_steps_refuse_are_refused():
    # as gs_step_low_forward and gs_upsample_forward refuse them; nothing runs
    import torch

    import paper_2308_01629_gb300 as gs
    sc = scenes.column(n_low=400, ratio=8)
    g = gs.Context(sc, stream="torch")
    ins = _ins(sc)
    outs = [torch.full_like(t, -7.0) for t in ins]
    ptrs = [t.data_ptr() for t in ins]
    lr0 = g.read(gs.GS_FIELD_LR_POS)

    def forward(dt, frames, n_sub):
        return gs.gs_rollout_forward(g.ctx, *ptrs, dt, frames, n_sub, 4, 2, *[t.data_ptr() for t in outs])

    for dt, n_sub in ((float("inf"), 1), (float("nan"), 1), (-1.0, 1), (0.0, 1), (1e-45, 4)):
        assert forward(dt, 2, n_sub) == gs.GS_ERR_ARG
    torch.cuda.synchronize()
    for o in outs:
        assert bool((o == -7.0).all())
    assert gs.gs_rollout_backward(g.ctx, *ptrs, *[t.data_ptr() for t in outs]) == gs.GS_ERR_STATE
    np.testing.assert_array_equal(g.read(gs.GS_FIELD_LR_POS), lr0)
    # a rollout of no frames takes no step
    assert forward(float("inf"), 0, 1) == gs.GS_OK
    assert all(torch.equal(a, b) for a, b in zip(ins, outs))
    assert forward(DT, 2, 1) == gs.GS_OK
    g.sync()
    assert all(bool(torch.isfinite(o).all()) for o in outs)
    g.close()
