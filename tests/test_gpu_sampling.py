"""The library's volume sampler (Sec. 4 initial sampling, gs_sample_volume)
against the oracle's: the same inside decisions and the same chosen
candidates in the same order, bit for bit, on a sphere, the castle union
at the LR and the HR radius, and edge cases; then a castle scene seeded by
it (LR and HR particles, and a rigid boulder sampled from an icosphere)
runs frames."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


def _both(orc, V, T, cand, r):
    import paper_2308_01629_gb300 as gs
    rc, sel, inside = gs.gs_sample_volume(V, T, cand, r)
    assert rc == gs.GS_OK
    ref_sel, ref_inside = orc.sample_volume(V, T, cand, r)
    np.testing.assert_array_equal(inside, ref_inside)
    np.testing.assert_array_equal(sel, ref_sel)
    return sel


@pytest.mark.parametrize("r, per_cell", [(0.012, 5.0), (0.004, 4.0)])
def test_sphere_samples_equal_the_oracle(orc, r, per_cell):
    V, T = scenes.icosphere((0.3, 0.2, 0.1), 0.15, 2)
    cand = scenes.volume_candidates(V, r, per_cell=per_cell, seed=21)
    sel = _both(orc, V, T, cand, r)
    assert len(sel) > 100


@pytest.mark.parametrize("r", [0.02, 0.0075])
def test_castle_samples_equal_the_oracle(orc, r):
    orc.set_threads(orc.max_threads())
    V, T = scenes.castle_mesh()
    cand = scenes.volume_candidates(V, r, per_cell=3.0, seed=22)
    sel = _both(orc, V, T, cand, r)
    orc.set_threads(1)
    P = cand[sel]
    # spot check of the spacing on a random subset (the oracle's pins cover the rest)
    rng = np.random.default_rng(0)
    sub = P[rng.choice(len(P), size=min(len(P), 1500), replace=False)]
    d2 = ((sub[:, None] - sub[None]) ** 2).sum(-1)
    np.fill_diagonal(d2, np.inf)
    assert d2.min() >= 4 * r * r


def test_sampler_edge_cases_on_the_gpu(orc):
    import paper_2308_01629_gb300 as gs
    V, T = scenes.box_mesh((0, 0, 0), (0.1, 0.1, 0.1))
    for cand in (np.zeros((0, 3)), [[0.05, 0.05, 0.05]], [[0.5, 0.5, 0.5], [-1, 0, 0]],
                 [[0.05, 0.05, 0.05], [0.0501, 0.05, 0.05]]):
        _both(orc, V, T, np.asarray(cand, float).reshape(-1, 3), 0.01)
    cand = scenes.volume_candidates(V, 0.01, seed=3)
    rc, sel, _ = gs.gs_sample_volume(V, T, cand, 0.01, capacity=3)
    assert rc == gs.GS_ERR_CAPACITY and len(sel) == 3
    rc, sel, inside = gs.gs_sample_volume(V, np.zeros((0, 3), np.int32), cand, 0.01)   # no triangles: nothing inside
    assert rc == gs.GS_OK and len(sel) == 0 and not inside.any()


def test_castle_scene_seeded_by_the_sampler_runs():
    import paper_2308_01629_gb300 as gs
    sc = scenes.castle_scene(gs.sample_volume, size=0.6, height=0.2, r_low=0.02, r_high=0.0075)
    assert sc["ratio"] >= 15 and len(sc["hr_pos"]) > 10 * len(sc["lr_pos"])
    ctx = gs.Context(sc)
    x0 = ctx.read(gs.GS_FIELD_HR_POS)
    for _ in range(6):
        ctx.frame(1.0 / 60.0, 4, sc["iters"])
    x1 = ctx.read(gs.GS_FIELD_HR_POS)
    lr = ctx.read(gs.GS_FIELD_LR_POS)
    assert np.isfinite(x1).all() and np.isfinite(lr).all()
    body = sc["lr_body"] > 0
    assert np.abs(lr[body, :3] - sc["lr_pos"][body, :3]).max() > 0.05    # the boulder flew
    assert np.abs(x1[:, :3] - x0[:, :3]).max() > 0.0
    ctx.close()


def test_surface_samples_equal_the_oracle_and_the_mesh_bucket_runs(orc):
    import paper_2308_01629_gb300 as gs
    for V, T, r in [(*scenes.box_mesh((0.1, 0.2, 0.05), (0.35, 0.3, 0.2)), 0.01),
                    (*scenes.icosphere((0.0, 0.0, 0.0), 0.2, 3), 0.006)]:
        cand = scenes.surface_candidates(V, T, r, seed=9)
        rc, sel = gs.gs_sample_surface(V, cand, r)
        assert rc == gs.GS_OK
        np.testing.assert_array_equal(sel, orc.sample_surface(V, cand, r))
    sc = scenes.digging_mesh_bucket(gs.sample_surface, size=0.5)
    ctx = gs.Context(sc)
    n_g = len(sc["lr_pos"]) - sc["n_solid"]
    x0 = ctx.read(gs.GS_FIELD_LR_POS)
    for _ in range(4):
        ctx.frame(1.0 / 60.0, 4, sc["iters"])
    x1 = ctx.read(gs.GS_FIELD_LR_POS)
    assert np.isfinite(x1).all() and np.isfinite(ctx.read(gs.GS_FIELD_HR_POS)).all()
    # the boundary particles move with their prescribed velocity
    u = sc["lr_vel"][n_g:, :3]
    np.testing.assert_allclose(x1[n_g:, :3] - x0[n_g:, :3], 4 / 60.0 * u, atol=1e-5)
    ctx.close()


def _near_surface(V, T, rng, n):
    """Candidates at 1e-2 .. 1e-10 of the mesh's size from its faces, edges and vertices, and some far away."""
    size = float((V.max(0) - V.min(0)).max())
    t = rng.integers(0, len(T), n)
    bary = rng.dirichlet((1.0, 1.0, 1.0), n)
    bary[: n // 3, 2] = 0.0                     # on an edge
    bary[: n // 9] = (1.0, 0.0, 0.0)            # on a vertex
    bary /= bary.sum(1, keepdims=True)
    p = (V[T[t]] * bary[:, :, None]).sum(1)
    d = rng.normal(size=(n, 3))
    d *= size * 10.0 ** rng.uniform(-10, -2, (n, 1)) / np.linalg.norm(d, axis=1, keepdims=True)
    far = V.mean(0) + size * rng.uniform(-50.0, 50.0, (16, 3))
    return np.concatenate([p + d, far])


@pytest.mark.parametrize("scale, shift", [(1.0, 0.0), (1e-12, 0.0), (1e9, 0.0), (1.0, 1e3)])
@pytest.mark.parametrize("mesh", ["castle", "sphere", "open_box"])
def test_inside_decisions_near_the_surface_equal_the_oracle(orc, mesh, scale, shift):
    # the single-precision evaluation may decide only what double precision
    # decides too: equality, no tolerance (offsets stay far above the double
    # evaluation's own rounding, also after a shift by 1e3)
    rng = np.random.default_rng(31)
    if mesh == "castle":
        V, T = scenes.castle_mesh()
    elif mesh == "sphere":
        V, T = scenes.icosphere((0.1, 0.2, 0.3), 0.15, 3)     # 1280 triangles: several staging rounds, a remainder
        T = T[: len(T) - 77]                                   # and not closed
    else:
        V, T = scenes.box_mesh((0, 0, 0), (1, 0.5, 0.25))
        T = T[2:]
    V = V * scale + shift
    cand = _near_surface(V, T, rng, 20000)
    if shift:
        cand = cand[: 20000][np.linalg.norm(cand[: 20000] - shift, axis=1) > 0]
    import paper_2308_01629_gb300 as gs
    orc.set_threads(orc.max_threads())
    r = 0.02 * float((V.max(0) - V.min(0)).max())
    rc, sel, inside = gs.gs_sample_volume(V, T, cand, r)
    ref_sel, ref_inside = orc.sample_volume(V, T, cand, r)
    orc.set_threads(1)
    assert rc == gs.GS_OK
    np.testing.assert_array_equal(inside, ref_inside)
    np.testing.assert_array_equal(sel, ref_sel)


def _symmetric_meshes():
    """Convex meshes whose centres and lattice points see their triangles under round angles, with the centre."""
    rng = np.random.default_rng(41)
    out = [(*scenes.box_mesh((0, 0, 0), (1, 1, 1)), np.full(3, 0.5)),
           (*scenes.box_mesh((-1, -2, -3), (1, 2, 3)), np.zeros(3)),
           (*scenes.box_mesh((0.125, 0.25, 0.5), (0.375, 0.75, 0.625)), np.array([0.25, 0.5, 0.5625]))]
    tet = np.array([(1, 1, 1), (1, -1, -1), (-1, 1, -1), (-1, -1, 1)], float)
    out.append((tet, np.array([(0, 1, 2), (0, 2, 3), (0, 3, 1), (1, 3, 2)], np.int32), np.zeros(3)))
    for axes in (np.eye(3), np.array([(1, 2, 2), (1, -2, -2), (-1, 2, -2)], float)):   # the latter: den exactly 0
        V = np.concatenate([axes, -axes])
        T = np.array([(a, 1 + b, 2 + c) for a in (0, 3) for b in (0, 3) for c in (0, 3)], np.int32)
        for t in T:
            if np.linalg.det(V[t]) < 0.0:
                t[1:] = t[2:0:-1]
        out.append((V, T, np.zeros(3)))
    # scaled and shifted cubes, whose coordinates round
    out += [(V0 * s + c, T0, c + 0.5 * s) for V0, T0, _ in out[:1]
            for s, c in [(rng.uniform(0.1, 10.0), rng.uniform(-1.0, 1.0, 3)) for _ in range(4)]]
    return out


@pytest.mark.parametrize("mesh", range(10))
def test_inside_decisions_at_symmetric_points_equal_the_oracle(orc, mesh):
    # the product of the triangles' unit numbers meets the cut of its angle
    # exactly at such points, in an order of the triangles that depends on the
    # mesh: many orders, centre and lattice points off the surface.  The
    # double evaluation is off by about 1e-15 there, so equality
    import paper_2308_01629_gb300 as gs
    V, T, c = _symmetric_meshes()[mesh]
    rng = np.random.default_rng(42 + mesh)
    half = 0.5 * (V.max(0) - V.min(0))
    k = np.arange(-5, 6) / 4.0
    off = np.array([(x, y, z) for x in k for y in k for z in k])
    if mesh == 3:       # |x| + |y| + |z| style faces: keep clear of them
        keep = np.min([np.abs(off @ n - 1.0) for n in ((1, 1, -1), (1, -1, 1), (-1, 1, 1), (-1, -1, -1))], 0) > 1e-3
    elif mesh in (4, 5):
        P = np.linalg.solve(V[:3].T, (off * half).T).T
        keep = np.abs(np.abs(P).sum(1) - 1.0) > 1e-3
    else:
        keep = np.abs(np.abs(off).max(1) - 1.0) > 1e-3
    cand = c + off[keep] * half
    r = 0.02 * float(half.max())
    for _ in range(60):
        P = T[rng.permutation(len(T))]
        P = np.array([np.roll(t, rng.integers(3)) for t in P], np.int32)
        rc, sel, inside = gs.gs_sample_volume(V, P, cand, r)
        ref_sel, ref_inside = orc.sample_volume(V, P, cand, r)
        assert rc == gs.GS_OK and ref_inside[np.flatnonzero(keep).searchsorted(len(off) // 2)]
        np.testing.assert_array_equal(inside, ref_inside)
        np.testing.assert_array_equal(sel, ref_sel)


@pytest.mark.parametrize("mesh", ["box", "sphere"])
def test_far_candidates_equal_the_oracle(orc, mesh):
    # from about 2e6 box sizes on the single-precision products leave their
    # range, from 1e13 on the lengths do: up to there and beyond it
    import paper_2308_01629_gb300 as gs
    V, T = scenes.box_mesh((0, 0, 0), (1e-3, 2e-3, 1e-3)) if mesh == "box" else scenes.icosphere((0, 0, 0), 1e-3, 2)
    rng = np.random.default_rng(43)
    d = rng.normal(size=(4000, 3))
    d[::4, 1:] = 0.0                                  # along an axis: in the planes of a box's faces or not at all
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    size = float((V.max(0) - V.min(0)).max())
    far = V.mean(0) + d * size * 10.0 ** rng.uniform(3.0, 17.0, (len(d), 1))
    cand = np.concatenate([scenes.volume_candidates(V, 1e-4, seed=44), far])
    rc, sel, inside = gs.gs_sample_volume(V, T, cand, 1e-4)
    ref_sel, ref_inside = orc.sample_volume(V, T, cand, 1e-4)
    assert rc == gs.GS_OK and not inside[-len(far):].any()
    np.testing.assert_array_equal(inside, ref_inside)
    np.testing.assert_array_equal(sel, ref_sel)


@pytest.mark.parametrize("shift", [1e9, 1e11, 1e13, 3e14])
@pytest.mark.parametrize("surface", [False, True])
def test_picks_far_from_the_origin_equal_the_oracle(orc, surface, shift):
    # in units of r: the distance test's positions are relative to cell
    # centres, which round by 2^-53 of the coordinate; beyond some 1e10 the
    # rounding is no longer small against the test's margin.  The candidates
    # themselves are exact, so equality
    import paper_2308_01629_gb300 as gs
    V, T = scenes.box_mesh((0, 0, 0), (24, 18, 21))
    V = V + np.array([shift, -shift, 0.5 * shift])
    rng = np.random.default_rng(45)
    if surface:
        cand = np.rint(scenes.surface_candidates(V, T, 1.0, per_cell=30.0, seed=46))
        cand = np.clip(cand + rng.integers(-64, 65, cand.shape) / 64.0, V.min(0), V.max(0))
        rc, sel = gs.gs_sample_surface(V, cand, 1.0)
        ref = orc.sample_surface(V, cand, 1.0)
    else:
        cand = scenes.volume_candidates(V, 1.0, per_cell=30.0, seed=46)
        rc, sel, inside = gs.gs_sample_volume(V, T, cand, 1.0)
        ref, ref_inside = orc.sample_volume(V, T, cand, 1.0)
        np.testing.assert_array_equal(inside, ref_inside)
    assert rc == gs.GS_OK
    np.testing.assert_array_equal(sel, ref)
