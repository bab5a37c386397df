"""The functional HR frame's routes against one another and against the
context's own frame: on the caller's buffers directly (large sets), as a graph
between copies (small sets, graphs on), and with buffers that are not 16-byte
aligned; in place and out of place.  The same bits every way."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu
DT = 1.0 / 60.0


def _frame_of_the_context(gs, sc):
    ctx = gs.Context(sc)
    ctx.upsample(DT)
    out = ctx.read(gs.GS_FIELD_HR_POS), ctx.read(gs.GS_FIELD_HR_VEL)
    ctx.close()
    return out


@pytest.mark.parametrize("graphs", [False, True])
@pytest.mark.parametrize("form", ["plain", "in_place", "misaligned"])
@pytest.mark.parametrize("n_low, ratio", [(1000, 7), (10486, 25)])     # 7,000 HR; 262,150: the direct route
def test_functional_frame_routes(n_low, ratio, form, graphs):
    import torch

    import paper_2308_01629_gb300 as gs
    sc = scenes.stir(scenes.funnel(n_low=n_low, ratio=ratio), seed=4)
    ref = _frame_of_the_context(gs, sc)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = gs.Context(sc, stream="torch")
        ctx.set_graphs(graphs)

        def place(a):    # a device copy, 4 bytes off a 16-byte boundary where asked
            if form != "misaligned":
                return torch.from_numpy(a).cuda()
            t = torch.zeros(a.size + 1, dtype=torch.float32, device="cuda")[1:]
            t.copy_(torch.from_numpy(a).cuda().reshape(-1))
            return t
        for _ in range(3):      # the third call replays what the second captured, in the other buffer parity
            ins = [place(sc[k]) for k in ("lr_pos", "lr_vel", "hr_pos", "hr_vel")]
            outs = ins[2:] if form == "in_place" else [place(np.zeros_like(sc["hr_pos"])) for _ in range(2)]
            rc = gs.gs_upsample_forward(ctx.ctx, *[t.data_ptr() for t in ins + outs], DT)
            assert rc == gs.GS_OK
            ctx.sync()
            for t, r in zip(outs, ref):
                np.testing.assert_array_equal(t.cpu().numpy().reshape(-1, 4).view(np.uint32), r.view(np.uint32))
        # the context's state is the frame's result too
        np.testing.assert_array_equal(ctx.read(gs.GS_FIELD_HR_POS)[:, :3], ref[0][:, :3])
        np.testing.assert_array_equal(ctx.read(gs.GS_FIELD_LR_POS), sc["lr_pos"])
    ctx.close()


@pytest.mark.parametrize("graphs", [False, True])
@pytest.mark.parametrize("form", ["plain", "in_place", "misaligned"])
def test_functional_frame_routes_at_the_direct_route(form, graphs):
    test_functional_frame_routes(16000, 25, form, graphs)      # 400,000 HR


@pytest.mark.parametrize("n_low, copies", [(10486, 2), (15999, 2), (16000, 1)])
def test_functional_frame_is_direct_only_above_its_line(n_low, copies):
    # the route between copies has one launch more, that of the results
    import torch

    import paper_2308_01629_gb300 as gs
    sc = scenes.funnel(n_low=n_low, ratio=25)
    with torch.cuda.stream(torch.cuda.Stream()):
        ctx = gs.Context(sc, stream="torch")
        ctx.set_graphs(True)
        ins = [torch.from_numpy(sc[k]).cuda() for k in ("lr_pos", "lr_vel", "hr_pos", "hr_vel")]
        outs = [torch.zeros_like(t) for t in ins[2:]]
        n = []
        for off in (0, 1):      # misaligned buffers go between copies, by the driver's
            bufs = [t if not off else torch.zeros(t.numel() + 1, device="cuda")[1:].copy_(t.reshape(-1)) for t in ins + outs]
            k0 = ctx.launches()
            assert gs.gs_upsample_forward(ctx.ctx, *[t.data_ptr() for t in bufs], DT) == gs.GS_OK
            ctx.sync()
            n.append(ctx.launches() - k0)
        ctx.close()
    assert n[0] - n[1] == copies


def test_functional_frame_is_direct_without_graphs():
    import torch

    import paper_2308_01629_gb300 as gs
    sc = scenes.funnel(n_low=1000, ratio=7)
    with torch.cuda.stream(torch.cuda.Stream()):
        ctx = gs.Context(sc, stream="torch")
        ins = [torch.from_numpy(sc[k]).cuda() for k in ("lr_pos", "lr_vel", "hr_pos", "hr_vel")]
        outs = [torch.zeros_like(t) for t in ins[2:]]
        n = []
        for graphs in (False, True):
            ctx.set_graphs(graphs)
            k0 = ctx.launches()
            assert gs.gs_upsample_forward(ctx.ctx, *[t.data_ptr() for t in ins + outs], DT) == gs.GS_OK
            ctx.sync()
            n.append(ctx.launches() - k0)
        ctx.close()
    assert n[1] - n[0] == 1      # the copy of the results


@pytest.mark.parametrize("graphs", [False, True])
@pytest.mark.parametrize("n_low, ratio", [(1000, 7), (10486, 25), (16000, 25)])
def test_functional_frame_in_a_capture_of_the_caller(n_low, ratio, graphs):
    import torch

    import paper_2308_01629_gb300 as gs
    sc = scenes.stir(scenes.funnel(n_low=n_low, ratio=ratio), seed=4)
    ref = _frame_of_the_context(gs, sc)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = gs.Context(sc, stream="torch")
        ctx.set_graphs(graphs)
        ins = [torch.from_numpy(sc[k]).cuda() for k in ("lr_pos", "lr_vel", "hr_pos", "hr_vel")]
        outs = [torch.zeros_like(t) for t in ins[2:]]
        ctx.sync()
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin(capture_error_mode="global")
        rc = gs.gs_upsample_forward(ctx.ctx, *[t.data_ptr() for t in ins + outs], DT)
        graph.capture_end()
        assert rc == gs.GS_OK
        for _ in range(2):
            for t in outs:
                t.zero_()
            graph.replay()
            stream.synchronize()
            for t, r in zip(outs, ref):
                np.testing.assert_array_equal(t.cpu().numpy().view(np.uint32), r.view(np.uint32))
        ctx.close()


@pytest.mark.parametrize("iters", [0, 4])
@pytest.mark.parametrize("n_stab", [0, 2])
def test_taped_step_and_its_reverse_equal_the_recording_ones(n_stab, iters):
    # with and without solver passes: the last pass writes the step's end
    # itself only when it is a solver pass; no pass at all leaves the prediction
    import torch

    import paper_2308_01629_gb300 as gs
    sc = scenes.stir(scenes.column(n_low=700, ratio=2, z0=0.02), seed=6, v_scale=0.2)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = gs.Context(sc, stream="torch", n_stab=n_stab)
        x, v = torch.from_numpy(sc["lr_pos"]).cuda(), torch.from_numpy(sc["lr_vel"]).cuda()
        g = [torch.randn(x.shape, generator=torch.Generator().manual_seed(k)).cuda() for k in (1, 2)]
        new = lambda: [torch.zeros_like(x), torch.zeros_like(x)]  # noqa: E731
        o1, o2, b1, b2 = new(), new(), new(), new()
        p = lambda ts: [t.data_ptr() for t in ts]  # noqa: E731
        assert gs.gs_step_low_forward(ctx.ctx, *p([x, v]), *p(o1), 1 / 240, iters) == gs.GS_OK
        assert gs.gs_step_low_backward(ctx.ctx, *p([x, v]), *p(g), *p(b1), 1 / 240, iters) == gs.GS_OK
        ctx.set_step_tapes(2)
        assert gs.gs_step_low_forward_taped(ctx.ctx, *p([x, v]), *p(o2), 1 / 240, iters, 5) == gs.GS_OK
        assert gs.gs_step_low_backward_taped(ctx.ctx, 5, *p(g), *p(b2)) == gs.GS_OK
        ctx.sync()
        for a, b in zip(o1 + b1, o2 + b2):
            np.testing.assert_array_equal(a.cpu().numpy(), b.cpu().numpy())
    ctx.close()
