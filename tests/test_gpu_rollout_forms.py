"""The library's rollout (gs_rollout_forward / gs_rollout_backward): what its
arguments may be, and rollouts of several lengths in one context."""
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


def test_rollouts_of_several_lengths_in_one_context_equal_fresh_ones():
    # a longer one moves the checkpoints, more steps per segment move the work
    # buffers, and other callers free the step tapes: captured sequences must
    # not outlive the buffers that they hold
    import torch

    import paper_2308_01629_gb300 as gs
    sc = scenes.column(n_low=400, ratio=8)
    ins = _ins(sc)
    gen = torch.Generator(device="cpu").manual_seed(5)
    cot = [torch.randn(t.shape, generator=gen).cuda() for t in ins]

    def run(g, frames, every):
        outs, grads = [torch.empty_like(t) for t in ins], [torch.empty_like(t) for t in ins]
        assert gs.gs_rollout_forward(g.ctx, *[t.data_ptr() for t in ins], DT, frames, 1, 4, every,
                                     *[t.data_ptr() for t in outs]) == gs.GS_OK
        assert gs.gs_rollout_backward(g.ctx, *[t.data_ptr() for t in cot], *[t.data_ptr() for t in grads]) == gs.GS_OK
        torch.cuda.current_stream().synchronize()
        return [t.cpu().numpy() for t in outs + grads]

    def context():
        g = gs.Context(sc, stream="torch")
        g.set_graphs(True)
        g.set_deterministic_backward(True)      # the same bits on every run
        return g

    with torch.cuda.stream(torch.cuda.Stream()):
        torch.cuda.synchronize()
        ref = {}
        for c in ((2, 1), (12, 1), (12, 6), (3, 3)):
            g = context()
            ref[c] = run(g, *c)
            g.close()
        g = context()
        for k, c in enumerate([(2, 1), (2, 1), (3, 3), (3, 3), (12, 1), (2, 1), (2, 1), (12, 6), (2, 1), (3, 3), (12, 1),
                               (12, 1), (12, 6), (2, 1), (3, 3), (2, 1)]):
            if k in (7, 13):
                g.set_step_tapes(0)
            for a, b in zip(run(g, *c), ref[c]):
                np.testing.assert_array_equal(a, b, err_msg=f"call {k}: {c}")
        g.close()
