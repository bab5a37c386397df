"""The HR frame's reverse mode over the ways its warps take their HR particles:
staged LR particles (HR side by side), more of them than the stage holds
(compressed), more rows of cells than lanes (scattered order), and a last warp
that is not full.  All against the 64-bit oracle."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu
DT = 1.0 / 60.0


def _state(n_low, ratio, squeeze):
    sc = scenes.stir(scenes.column(seed=scenes.SEED_BASE + 77, n_low=n_low, ratio=ratio, z0=0.05), seed=3, v_scale=0.2)
    for k in ("lr_pos", "hr_pos"):
        mid = np.float32([0.3, 0.3, 0.05])
        sc[k][:, :3] = mid + np.float32(squeeze) * (sc[k][:, :3] - mid)
    return sc


# 2e-4 of the gradient's norm: it sums up to about 500 terms in 32 bits (500 *
# 2^-24 = 3e-5 of their absolute sum), and a weight cubes a difference that
# loses about two bits
@pytest.mark.parametrize("deterministic", [False, True])
@pytest.mark.parametrize("order", ["parents", "shuffled"])
@pytest.mark.parametrize("n_low, ratio, squeeze", [(1, 3, 1.0), (37, 7, 1.0), (300, 16, 1.0), (300, 16, 0.45),
                                                   (1500, 3, 1.0)])
def test_reverse_frame_matches_oracle_in_any_order(orc, n_low, ratio, squeeze, order, deterministic):
    import torch

    import paper_2308_01629_gb300 as gs
    from paper_2308_01629_gb300.diff import UpsampleFn
    sc = _state(n_low, ratio, squeeze)
    m = len(sc["hr_pos"])
    rng = np.random.default_rng(11)
    if order == "shuffled":
        perm = rng.permutation(m)
        sc["hr_pos"][:, :3], sc["hr_vel"] = sc["hr_pos"][perm, :3], sc["hr_vel"][perm]
    prm = dict(r_low=float(np.float32(sc["r_low"])), r_high=float(np.float32(sc["r_high"])), dt=float(np.float32(DT)),
               gx=0.0, gy=0.0, gz=float(np.float32(-9.81)), c1=512 / 729, c2=0.6, eps_w=1e-4, eps_x=1e-6)
    host = [sc[k][:, :3] for k in ("lr_pos", "lr_vel", "hr_pos", "hr_vel")]
    keep = (orc.upsample(*host, scenes.sdf_table(sc["sdfs"]), prm)["flag"] == 0)[:, None]
    a, b = ((rng.normal(size=(m, 3)) * keep).astype(np.float32) for _ in range(2))
    ctx = gs.Context(sc, stream="torch")
    if deterministic:
        ctx.set_deterministic_backward(True)
    ins = [torch.from_numpy(sc[k]).cuda().requires_grad_(True) for k in ("lr_pos", "lr_vel", "hr_pos", "hr_vel")]
    ox, ov = UpsampleFn.apply(ctx, DT, *ins)
    g = [torch.from_numpy(np.pad(t, ((0, 0), (0, 1)))).cuda() for t in (a, b)]
    got = torch.autograd.grad([ox, ov], ins, g)
    want = orc.upsample_vjp(*host, scenes.sdf_table(sc["sdfs"]), prm, a, b)
    for t, w in zip(got, want):
        t = t.cpu().numpy()
        assert np.all(t[:, 3] == 0)
        assert np.linalg.norm(t[:, :3] - w) <= 2e-4 * np.linalg.norm(w)
    ctx.close()
