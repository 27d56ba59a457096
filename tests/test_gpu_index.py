"""The render's empty-space index and the shared start of a warp's rays: on
grids whose 32^3 boxes are partial, with wide and narrow beams, cameras
inside, at the edge of and outside the grid, depth limits, and occupancy of
infinities and NaN, every output equals the march over every sample
(skip_empty = 0) bit for bit, before and after map updates that refresh part
of the index."""
import numpy as np
import pytest
import torch

from gpu_helpers import t

pytestmark = pytest.mark.gpu


def field(shape, seed, extent):
    """A few solid balls in free space (values from far below to above tau), some slabs just under tau."""
    rng = np.random.default_rng(seed)
    nz, ny, nx = shape
    vs = extent / max(shape)
    ax = [(np.arange(m) + 0.5) * vs for m in (nz, ny, nx)]
    Z, Y, X = np.meshgrid(*ax, indexing="ij")
    occ = np.full(shape, -0.2)
    for _ in range(24):
        c = (0.5 + rng.choice([-1, 1], 3) * rng.uniform(0.1, 0.45, 3)) * np.array([nx, ny, nz]) * vs
        r = rng.uniform(0.05, 0.12) * min(shape) * vs
        occ = np.maximum(occ, r - np.sqrt((X - c[0]) ** 2 + (Y - c[1]) ** 2 + (Z - c[2]) ** 2))
    occ[:, ny // 2] = np.maximum(occ[:, ny // 2], -1e-7)
    return occ.astype(np.float32), rng.uniform(0, 1, shape + (3,)).astype(np.float32)


@pytest.mark.parametrize("shape,W,H,fx,storage,special", [
    ((8, 8, 8), 21, 17, 9.0, "f32", False),          # one box; beams wider than it
    ((40, 72, 24), 83, 61, 70.0, "f32", False),      # 5 x 9 x 3 boxes: partial 32^3 boxes on every axis
    ((40, 40, 40), 83, 61, 110.0, "bf16", False),    # narrow beams
    ((64, 64, 64), 64, 48, 55.0, "f32", True),       # infinities and NaN in free space and at surfaces
    ((104, 96, 136), 97, 31, 80.0, "f32", False)])
def test_index_changes_no_render(shape, W, H, fx, storage, special):
    from paper_2212_02988_gb300 import Filter, config, make_state
    extent = 4.0
    occ, rgb = field(shape, sum(shape), extent)
    if special:
        rng = np.random.default_rng(1)
        idx = tuple(rng.integers(0, m, 40) for m in shape)
        occ[idx] = rng.choice(np.array([np.nan, np.inf, -np.inf, -3e38], np.float32), 40)
    vs = extent / max(shape)
    size = np.array(shape[::-1]) * vs
    poses = [np.concatenate([p * size, q]) for p, q in (
        ((0.5, 0.5, 0.5), (0.5, -0.5, 0.5, -0.5)), ((0.02, 0.5, 0.6), (0.9, 0.1, 0.3, -0.2)),
        ((0.999, 0.001, 0.5), (0.2, 0.6, 0.1, -0.7)), ((-0.01, 0.5, 0.5), (0.5, -0.5, 0.5, -0.5)),
        ((0.5, 0.5, 2.0), (0.0, 1.0, 0.0, 0.0)))]
    var = np.full(shape, 0.1, np.float32)
    depth = np.random.default_rng(2).uniform(0.2, 2.0, (H, W)).astype(np.float32)
    depth[H // 3:, :] = 1.3
    col = np.full((H, W, 3), 0.5, np.float32)
    out = []
    for skip in (0, 1):
        res = []
        for max_depth in (0.0, 0.31 * extent):
            cfg = config(max(shape), extent, W, H, storage=storage, nx=shape[2], ny=shape[1], nz=shape[0],
                         origin=(0.0, 0.0, 0.0), fx=fx, fy=fx, skip_empty=skip, max_depth=max_depth)
            F = Filter(cfg, make_state(poses[0]), device=0)
            F.map_load(t(occ), t(rgb), t(var), t(var))
            res += [F.render(p) for p in poses]
            for p in poses[:3]:   # map updates refresh the index of the tiles in view
                F.set_state(make_state(p))
                F.update_map(t(depth), t(col))
                res += [F.render(q) for q in poses]
            samples = F.stats()["render_samples"]
            F.close()
        out.append((res, samples))
    for a, b in zip(out[0][0], out[1][0]):
        for k in ("depth", "rgb", "mask", "hitk"):
            assert torch.equal(torch.nan_to_num(a[k].float(), 7.0, 8.0, 9.0), torch.nan_to_num(b[k].float(), 7.0, 8.0, 9.0)), k
    assert any((r["hitk"] > 1).any() for r in out[0][0])
    assert out[1][1] <= out[0][1]
