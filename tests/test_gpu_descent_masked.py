"""The descent step where the frame has no depth and the map behind those
pixels holds values whose slopes or gradients are not finite (colours of NaN or
infinity, an occupancy of -inf in front of a surface, occupancies so small that
the reciprocal of their difference overflows): such a ray has no gradient, so
the voxels that only such rays read take the prior's step alone, bit for bit,
and every other voxel stays finite.  The work counters count its ray and hit
as the render's do."""
import numpy as np
import pytest
import torch
from scipy.spatial.transform import Rotation

import synth
from gpu_helpers import bf16_round, make_pair, t

pytestmark = pytest.mark.gpu

LR_OCC, LR_RGB = 2e-6, 1e-5


def sample_points(w, pose, hitk):
    """World positions of the samples k - 1 and k of every pixel ((2, H, W, 3))."""
    v, u = np.mgrid[0:w.height, 0:w.width]
    x, y, z = pose[4], pose[5], pose[6]
    R = Rotation.from_quat([x, y, z, pose[3]]).as_matrix()
    d = np.stack([(u - w.cx) / w.fx, (v - w.cy) / w.fx, np.ones_like(u, dtype=float)], -1) @ R.T
    d /= np.linalg.norm(d, axis=-1, keepdims=True)
    eps = 0.4 * w.voxel
    return np.stack([pose[:3] + (np.maximum(hitk - 1 + m, 0) * eps)[..., None] * d for m in (0, 1)])


@pytest.mark.parametrize("special,storage", [("rgb_nan", "f32"), ("rgb_inf", "bf16"), ("occ_inf", "f32"),
                                             ("occ_tiny", "f32")])
def test_pixels_without_depth_leave_the_map(oracle_mod, special, storage):
    w = synth.tiny(n=32, width=83, height=61)
    s = synth.Sequence(w)
    occ, rgb, vo, vr = (np.array(a, dtype=np.float32) for a in s.settled_map())
    if storage == "bf16":
        occ, rgb = bf16_round(occ), bf16_round(rgb)
    pose = s.pose7(3)
    F, _ = make_pair(w, oracle_mod, storage=storage, map_arrays=(occ, rgb, vo, vr))
    hk = F.render(pose)["hitk"].cpu().numpy()
    assert hk[30, 40] >= 3
    X = sample_points(w, pose, hk)[1, 30, 40]
    ax = w.origin + (np.arange(w.n) + 0.5) * w.voxel
    Z, Y, Xg = np.meshgrid(ax, ax, ax, indexing="ij")
    dist = np.sqrt((Xg - X[0]) ** 2 + (Y - X[1]) ** 2 + (Z - X[2]) ** 2) / w.voxel
    ball = dist <= 2.5
    if special == "rgb_nan":
        rgb[ball] = np.nan
    elif special == "rgb_inf":
        rgb[ball] = np.inf
    elif special == "occ_inf":
        occ[ball & (occ < 0)] = -np.inf
    else:
        occ[ball] *= np.float32(1e-39)
        assert np.abs(occ[ball]).max() > 0
    F.map_load(t(occ), t(rgb), t(vo), t(vr))
    hk = F.render(pose)["hitk"].cpu().numpy()
    # the pixels whose samples read a voxel of the ball (or near it) have no depth
    P = sample_points(w, pose, hk)
    near = (hk >= 2) & (np.sqrt(((P - X) ** 2).sum(-1)).min(0) / w.voxel <= 2.5 + 2.0)
    assert near.sum() >= 20 and ((hk >= 2) & ~near).sum() >= 200
    f = s.frame(3)
    D, C = f["depth"].copy(), f["rgb"]
    D[near] = np.resize(np.array([0.0, np.nan, -1.0, np.inf], np.float32), near.sum())
    before = F.stats()
    F.map_descent(pose[None], t(D[None]), t(C[None]), 0.02, 0.1, LR_OCC, LR_RGB, want_loss=False)
    after = F.stats()
    assert after["render_rays"] - before["render_rays"] == w.width * w.height
    assert after["render_hits"] - before["render_hits"] == int((hk >= 2).sum())
    got = {k: v.cpu().numpy() for k, v in F.map_store().items()}
    inv_v0 = np.float32(1.0 / F.cfg.prior_var)
    for name, m, mu0, lr in (("occ", occ, F.cfg.init_occ, LR_OCC), ("rgb", rgb, F.cfg.init_rgb, LR_RGB)):
        with np.errstate(invalid="ignore", over="ignore", under="ignore"):
            prior = m - np.float32(lr) * ((m - np.float32(mu0)) * inv_v0)
        if storage == "bf16":
            prior = bf16_round(prior)
        fin = np.isfinite(m)
        assert np.isfinite(got[name][fin]).all(), (name, int((~np.isfinite(got[name][fin])).sum()))
        core = ball if m.ndim == 3 else np.broadcast_to(ball[..., None], m.shape)
        assert np.array_equal(got[name][core & fin], prior[core & fin]), name
    assert np.abs(got["occ"] - occ)[np.isfinite(occ) & ~ball].max() > 1e-4   # the other pixels moved the map
    F.close()
