"""The ghost cells beside a map's faces, edges and corners hold the voxels they
clamp to after a map load (of any subset of the arrays) and after a descent
step.  Cameras stand a quarter of a voxel outside the last voxel centres and look
along the face or edge at a wall three voxels on, so that every sample up to the
hit reads ghosts: the outer layer of voxels is below tau but for the walls, everything
inside it above, and the map loaded before it far above, so that a ghost that is
stale or a copy of another voxel moves the hits.  Images against the oracle's
clamped march.  Rows shorter than, equal to and longer than a segment of the
exchange."""
import numpy as np
import pytest
from scipy.spatial.transform import Rotation

from gpu_helpers import bf16_round, check_render, t

pytestmark = pytest.mark.gpu

VS, W, H, FX = 0.1, 40, 24, 220.0
OFF = 0.25   # of a voxel, beyond the last voxel centre


def cameras(shape):
    """(name, pose) for the 26 directions of a face, an edge or a corner."""
    n = np.array(shape[::-1])
    out = []
    for s in np.ndindex(3, 3, 3):
        s = np.array(s) - 1
        if not s.any():
            continue
        g = np.where(s > 0, n - 1 + OFF, np.where(s < 0, -OFF, n // 2))
        free = np.flatnonzero(s == 0)
        d = np.eye(3)[free[0]] if len(free) else np.array([-s[0], 0, 0])
        R = Rotation.align_vectors([d], [[0, 0, 1]])[0]
        x, y, z, w = R.as_quat()
        out.append((tuple(int(a) for a in s), np.concatenate([(g + 0.5) * VS, [w, x, y, z]])))
    return out


def oracle_params(O, shape):
    from synth import tiny
    nz, ny, nx = shape
    return O.params(tiny(), nx=nx, ny=ny, nz=nz, voxel=VS, origin=(0, 0, 0), width=W, height=H, fx=FX, fy=FX,
                    cx=0.5 * (W - 1), cy=0.5 * (H - 1), eps=0.15 * VS)


def fields(shape, seed):
    rng = np.random.default_rng(seed)
    n = np.array(shape[::-1])
    occ = rng.uniform(0.3, 0.7, shape)
    face = np.ones(shape, bool)
    face[1:-1, 1:-1, 1:-1] = False
    occ[face] = rng.uniform(-0.3, -0.05, face.sum())
    for where, pose in cameras(shape):   # the wall: two voxels to each side on a face
        s = np.array(where)
        free = np.flatnonzero(s == 0)
        v = np.where(s > 0, n - 1, np.where(s < 0, 0, n // 2))
        a = free[0] if len(free) else 0
        v[a] += 3 if len(free) else -3 * s[0]
        for o in range(-2, 3) if len(free) == 2 else (0,):
            q = v.copy()
            if len(free) == 2:
                q[free[1]] += o
            occ[q[2], q[1], q[0]] = rng.uniform(0.1, 0.5)
    return occ.astype(np.float32), rng.uniform(0, 1, shape + (3,)).astype(np.float32)


def ghost_hits(pose, hitk, shape):
    """Pixels whose hit sample reads a ghost (by FP64 positions)."""
    v, u = np.mgrid[0:H, 0:W]
    R = Rotation.from_quat([pose[4], pose[5], pose[6], pose[3]]).as_matrix()
    d = np.stack([(u - 0.5 * (W - 1)) / FX, (v - 0.5 * (H - 1)) / FX, np.ones((H, W))], -1) @ R.T
    d /= np.linalg.norm(d, axis=-1, keepdims=True)
    g = (pose[:3] + (hitk * 0.15 * VS)[..., None] * d) / VS - 0.5
    out = (g < 0) | (g > np.array(shape[::-1]) - 1)
    return (hitk >= 2) & out.any(-1)


@pytest.mark.parametrize("shape,storage", [((16, 24, 120), "f32"), ((24, 16, 128), "bf16"), ((16, 16, 136), "f32")])
def test_ghosts_after_load_and_descent(oracle_mod, shape, storage):
    from paper_2212_02988_gb300 import Filter, config
    O = oracle_mod
    nz, ny, nx = shape
    F = Filter(config(nx, VS * nx, W, H, storage=storage, nx=nx, ny=ny, nz=nz, voxel=VS, origin=(0, 0, 0), fx=FX, fy=FX,
                      eps=0.15 * VS), device=0)
    p = oracle_params(O, shape)
    kept = bf16_round if storage == "bf16" else (lambda a: a)

    def stale(occ=True, rgb=True):
        F.map_load(t(np.ones(shape, np.float32)) if occ else None, t(np.full(shape + (3,), 7, np.float32)) if rgb else None)

    def check(occ, rgb, name):
        for where, pose in cameras(shape):
            ref = O.render(p, occ, rgb, pose)
            assert ghost_hits(pose, ref["hitk"], shape).mean() > 0.9, where
            try:
                check_render(F.render(pose), ref)
            except AssertionError as e:
                raise AssertionError(f"{name} {where}: {e}") from None

    occ, rgb = fields(shape, nx)
    stale()
    F.map_load(t(occ), t(rgb))
    check(kept(occ), kept(rgb), "load")
    occ2, rgb2 = fields(shape, nx + 1)
    stale(rgb=False)
    F.map_load(t(occ2), None)              # the occupancy alone, then the colours alone
    check(kept(occ2), kept(rgb), "occupancy")
    stale(occ=False)
    F.map_load(None, t(rgb2))
    check(kept(occ2), kept(rgb2), "colours")
    poses = np.stack([pose for _, pose in cameras(shape)])
    D = np.stack([O.render(p, kept(occ2), kept(rgb2), q)["depth"] for q in poses]).astype(np.float32) * np.float32(1.01)
    C = np.random.default_rng(1).uniform(0, 1, (len(poses), H, W, 3)).astype(np.float32)
    F.map_descent(poses, t(D), t(C), 0.05, 0.1, 1e-6, 1e-4)
    m = {k: v.cpu().numpy() for k, v in F.map_store().items()}
    assert np.abs(m["rgb"] - kept(rgb2)).max() > 1e-3
    for where, pose in cameras(shape):
        check_render(F.render(pose), O.render(p, m["occ"], m["rgb"], pose))
    F.close()
