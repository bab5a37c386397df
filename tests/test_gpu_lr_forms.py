"""The forms of the LR step's kernels against one another: eight or two lanes
per particle in a pass, four or one in the candidate search, one-scene
parameters or a scene table, and the binning by buckets or by the general
counting sort.  Which form runs depends on the sizes only, and all give the
same bits, so the same scene is stepped alone and among copies of itself."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


def _small(kind):
    sc = scenes.cube(n_side=12, ratio=1)
    if kind == "packed":     # over 64 candidates per particle and cells of over 16: windows and spilled buckets
        c = sc["lr_pos"][:, :3].mean(0)
        sc["lr_pos"][:, :3] = c + (sc["lr_pos"][:, :3] - c) * np.float32(0.45)
    rng = np.random.default_rng(5)
    sc["lr_vel"][:, :3] = rng.normal(0.0, 0.4, (len(sc["lr_vel"]), 3))
    return sc


def _states(gs, sl, frames=2, mat=None, dt=1.0 / 60.0):
    ctx = gs.Context(sl if len(sl) > 1 else sl[0], max_neighbors=512)
    if mat is not None:
        ctx.set_materials(scenes.MATERIALS, np.concatenate([mat] * len(sl)))
    for _ in range(frames):
        ctx.frame(dt, 2, 5)
    out = [ctx.read(f)[ctx.scene_slice(k, f)] for k in range(len(sl)) for f in (gs.GS_FIELD_LR_POS, gs.GS_FIELD_LR_VEL)]
    ctx.close()
    return out


@pytest.mark.parametrize("copies", [3, 10, 39])     # 5,184 / 17,280 / 67,392 LR: on each side of both lines
@pytest.mark.parametrize("kind", ["cube", "packed", "materials"])
def test_lane_forms_give_the_same_bits(kind, copies):
    import paper_2308_01629_gb300 as gs
    sc = _small(kind)
    mat = np.random.default_rng(6).integers(0, 3, len(sc["lr_pos"])).astype(np.uint32) if kind == "materials" else None
    ref = _states(gs, [sc], mat=mat)
    got = _states(gs, [sc] * copies, mat=mat)
    for k in range(copies):
        np.testing.assert_array_equal(got[2 * k], ref[0])
        np.testing.assert_array_equal(got[2 * k + 1], ref[1])


@pytest.mark.parametrize("size", [0.66, 1.17])      # 22,000 / 69,000 LR
def test_one_scene_equals_a_scene_among_others(size):
    import paper_2308_01629_gb300 as gs
    sc = scenes.digging(ratio=1, size=size)
    sc["lr_vel"][:, :3] = np.random.default_rng(7).normal(0.0, 0.2, (len(sc["lr_vel"]), 3))
    ref = _states(gs, [sc], frames=1)
    got = _states(gs, [sc, scenes.cube(ratio=1)], frames=1)
    np.testing.assert_array_equal(got[0], ref[0])
    np.testing.assert_array_equal(got[1], ref[1])


@pytest.mark.parametrize("pile", [0, 15, 16, 17, 33, 700])
@pytest.mark.parametrize("n_cells_x", [1, 63, 64, 65])    # with 8 x 8 more: one cell row up to past a tile of 4,096
def test_bucket_binning_order(orc, pile, n_cells_x):
    import paper_2308_01629_gb300 as gs
    sc = dict(scenes.cube(ratio=1))
    h = float(np.float32(3.0 * sc["r_low"] * (1.0 + 1.0 / 1024.0)))
    sc["box_lo"], sc["box_hi"] = (0.0, 0.0, 0.0), (h * (n_cells_x - 0.5), 7.5 * h, 7.5 * h)
    rng = np.random.default_rng(pile + n_cells_x)
    ctx = None
    for round_ in range(2):      # the second binning meets what the first one left of its counts
        p = sc["lr_pos"].copy()
        p[:, :3] = rng.uniform(-0.5 * h, np.asarray(sc["box_hi"]) + 0.5 * h, (len(p), 3))
        p[rng.choice(len(p), pile, replace=False), :3] = np.asarray(sc["box_hi"]) - 0.3 * h
        if ctx is None:
            ctx = gs.Context(dict(sc, lr_pos=p))
        else:
            ctx.write(gs.GS_FIELD_LR_POS, p)
        ctx.bin_low()
        o, _, ih, dims = orc.grid(float(np.float32(sc["r_low"])), np.float32(sc["box_lo"]).astype(float),
                                  np.float32(sc["box_hi"]).astype(float))
        nc = int(np.prod(dims))
        ref_idx, ref_start = orc.counting_sort(orc.cell_keys(p, o, ih, dims), nc)
        np.testing.assert_array_equal(ctx.read(gs.GS_FIELD_LR_SORTED_INDEX), ref_idx)
        np.testing.assert_array_equal(ctx.read(gs.GS_FIELD_LR_CELL_START)[:nc + 1], ref_start)
    ctx.close()


def test_a_grid_too_large_for_buckets_gives_the_same_steps():
    # over four million cells take the general counting sort; the cell order
    # of the particles is that of the small grid with the same origin
    import paper_2308_01629_gb300 as gs
    sc = _small("cube")
    sc["sdfs"] = [scenes.box_interior((0, 0, 0), (0.5, 0.5, 0.5))]
    ref = _states(gs, [sc])
    big = dict(sc, box_hi=(5.0, 5.0, 5.0))
    got = _states(gs, [big])
    np.testing.assert_array_equal(got[0], ref[0])
    np.testing.assert_array_equal(got[1], ref[1])


@pytest.mark.parametrize("solid", [False, True])
@pytest.mark.parametrize("ratio", [3, 12])      # 4,700 / 18,900 warp items: on each side of the persistent grid's line
def test_gather_shapes_and_scene_forms_give_the_same_bits(ratio, solid):
    import paper_2308_01629_gb300 as gs
    sc = scenes.stir(scenes.digging(ratio=ratio), seed=9)
    if solid:
        sc["lr_pos"][::97, 3] = 0.0

    def run(sl, shape):
        ctx = gs.Context(sl if len(sl) > 1 else sl[0])
        if shape:
            ctx.set_tuning(*shape)
        for _ in range(2):
            ctx.upsample(1.0 / 60.0)
        out = [ctx.read(f)[ctx.scene_slice(0, f)] for f in (gs.GS_FIELD_HR_POS, gs.GS_FIELD_HR_VEL)]
        ctx.close()
        return out

    ref = run([sc], (8, 0))
    for sl, shape in (([sc], None), ([sc], (4, 7)), ([sc], (16, 0)), ([sc, scenes.cube()], None)):
        for a, b in zip(run(sl, shape), ref):
            np.testing.assert_array_equal(a.view(np.uint32), b.view(np.uint32))


@pytest.mark.parametrize("kind", ["cube", "bed", "solids", "body", "materials", "batch"])
def test_steps_that_begin_the_next_binning_give_the_same_bits(kind):
    # within a frame a step's last pass begins the next binning; with the
    # timers on every phase keeps its own launches
    import paper_2308_01629_gb300 as gs
    sc = {"cube": scenes.cube, "bed": lambda: scenes.digging(ratio=2, size=0.7), "solids": scenes.cube_on_particle_floor,
          "body": scenes.cube_with_block, "materials": scenes.cube,
          "batch": lambda: scenes.batch(n_scenes=3, lo_count=300, hi_count=900)}[kind]()
    out = []
    for timing in (False, True):
        ctx = gs.Context(sc)
        if kind == "materials":
            ctx.set_materials(*scenes.materials(sc, 3))
        ctx.set_timing(timing)
        for _ in range(3):
            ctx.frame(1.0 / 60.0, 3, 4)
        out.append([ctx.read(f).view(np.uint32) for f in (gs.GS_FIELD_LR_POS, gs.GS_FIELD_LR_VEL, gs.GS_FIELD_HR_POS,
                                                           gs.GS_FIELD_HR_VEL)])
        ctx.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


def _crowds(sc, kind, rng):
    """LR positions whose cells hold far more particles than a bucket."""
    p = sc["lr_pos"].copy()
    n, hi = len(p), np.asarray(sc["box_hi"])
    h = float(np.float32(3.0 * sc["r_low"] * (1.0 + 1.0 / 1024.0)))
    if kind == "bed":            # 24 in most cells
        side = h * (n / 24.0) ** (1.0 / 3.0)
        p[:, :3] = 0.1 + rng.uniform(0.0, side, (n, 3))
    elif kind == "pile":         # all in one cell
        p[:, :3] = 10.5 * h + rng.uniform(0.0, 1e-3, (n, 3))
    elif kind == "piles":        # over a thousand in each of some cells, the particles of a cell far apart in the set
        c = rng.uniform(0.1, 0.9, (40, 3)) * hi
        p[:, :3] = c[rng.integers(0, len(c), n)] + rng.uniform(0.0, 1e-4, (n, 3))
    elif kind == "line":         # on each side of the line between the two ways of counting
        p[:, :3] = rng.uniform(0.0, 1.0, (n, 3)) * hi
        at = rng.permutation(n)
        p[at[:2048], :3] = h * np.array([20.5, 5.5, 5.5])
        p[at[2048:4097], :3] = h * np.array([25.5, 5.5, 5.5])
        p[at[4097:], 0] = np.where(np.abs(p[at[4097:], 0] - 23.0 * h) < 4.0 * h, 0.1, p[at[4097:], 0])
    else:                        # outside the grid: clamped into its edge cells
        p[:, :3] = hi * rng.uniform(0.0, 1.0, (n, 3)) + (0.0, 0.0, 10.0)
        p[: n // 3, :3] += 10.0
    return p


@pytest.mark.parametrize("kind", ["bed", "pile", "piles", "line", "outside"])
def test_crowded_cells_are_ordered_and_cost_no_more_than_the_general_sort(orc, kind):
    # the same particles in a grid of a few cells and in one of over four
    # million, which takes the general counting sort (linear in the crowd);
    # the bound on the time is twice that
    import torch

    import paper_2308_01629_gb300 as gs
    base = scenes.digging(ratio=1)
    p = _crowds(base, kind, np.random.default_rng(17))
    ms = []
    for box_hi in (base["box_hi"], tuple(np.asarray(base["box_hi"]) * 5.1)):
        sc = dict(base, box_hi=box_hi)
        q = p.copy()
        if kind == "outside":    # beyond this grid too
            q[:, 2] += box_hi[2]
        with torch.cuda.stream(torch.cuda.Stream()):
            ctx = gs.Context(dict(sc, lr_pos=q), stream="torch")
            ctx.set_graphs(False)
            best = 1e9
            for _ in range(4):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                ctx.bin_low()
                b.record()
                b.synchronize()
                best = min(best, a.elapsed_time(b))
            ms.append(best)
            o, _, ih, dims = orc.grid(float(np.float32(sc["r_low"])), np.float32(sc["box_lo"]).astype(float),
                                      np.float32(box_hi).astype(float))
            nc = int(np.prod(dims))
            ref_idx, ref_start = orc.counting_sort(orc.cell_keys(q, o, ih, dims), nc)
            np.testing.assert_array_equal(ctx.read(gs.GS_FIELD_LR_SORTED_INDEX), ref_idx)
            np.testing.assert_array_equal(ctx.read(gs.GS_FIELD_LR_CELL_START)[:nc + 1], ref_start)
            ctx.close()
    print(f"{kind}: buckets {ms[0]:.3f} ms, general sort {ms[1]:.3f} ms, {len(p)} LR, largest cell "
          f"{np.diff(ref_start).max()}")
    assert ms[0] < 2.0 * ms[1]


@pytest.mark.parametrize("kind", ["body", "depth_friction", "solids"])
def test_lane_forms_among_bystanders_give_the_same_bits(kind):
    # the same grains with few and with many others far away in the same
    # scene: on each side of both lines
    import paper_2308_01629_gb300 as gs
    base = scenes.cube_on_particle_floor() if kind == "solids" else scenes.cube_with_block()
    n, r = len(base["lr_pos"]), base["r_low"]
    hi = np.array([4.0, 1.0, 1.0])
    side = np.arange(0.05, 0.95, 2.5 * r)
    room = np.stack(np.meshgrid(np.arange(1.5, 3.9, 2.5 * r), side, side, indexing="ij"), -1).reshape(-1, 3)
    states = []
    for others in (64, 17000, 68000):
        assert others <= len(room) and base["lr_pos"][:, 0].max() < 1.4
        p = np.zeros((others, 4), np.float32)
        p[:, :3], p[:, 3] = room[:others], base["lr_pos"][:, 3].max()
        v = np.random.default_rng(23).normal(0.0, 0.5, (others, 4)).astype(np.float32)
        v[:, 3] = 0.0
        sc = dict(base, box_lo=(0.0, 0.0, 0.0), box_hi=tuple(hi), sdfs=[scenes.box_interior((0, 0, 0), tuple(hi))],
                  lr_pos=np.concatenate([base["lr_pos"], p]), lr_vel=np.concatenate([base["lr_vel"], v]))
        sc.pop("lr_body", None)
        if kind == "body":
            sc["lr_body"] = np.concatenate([base["lr_body"], np.zeros(others, np.uint32)])
        ctx = gs.Context(sc, friction_mode=int(kind == "depth_friction"))
        for _ in range(4):
            ctx.frame(1.0 / 60.0, 2, 5)
        states.append([ctx.read(f)[:n].view(np.uint32) for f in (gs.GS_FIELD_LR_POS, gs.GS_FIELD_LR_VEL)])
        ctx.close()
    for s in states[1:]:
        for a, b in zip(s, states[0]):
            np.testing.assert_array_equal(a, b)
