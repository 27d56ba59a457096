"""The march's loops (every sample, or by the empty-space index; with and
without the detail counters; several samples at once): limits of 1 to 9 samples
around the number evaluated together, hits at the first samples, odd and
specialised grids.  Images against the oracle; without skipping the samples counted
are the oracle's, and the distinct corners those of the cells that the FP32
march visits (8 for a ray's first cell, then 8 - 4, 6 or 7 shared ones)."""
import numpy as np
import pytest

import synth
from gpu_helpers import check_render, make_pair

pytestmark = pytest.mark.gpu

f32 = np.float32


def fma(a, b, c):
    return (np.asarray(a, np.float64) * np.asarray(b, np.float64) + np.asarray(c, np.float64)).astype(f32)


def visited_corners(w, pose, nsamp):
    """Distinct corners of each ray's samples 1 .. nsamp, by the FP32 recipe."""
    v, u = np.mgrid[0:w.height, 0:w.width]
    q = pose[3:] / np.sqrt((pose[3:] ** 2).sum())
    a, x, y, z = q
    R = np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - a * z), 2 * (x * z + a * y)],
                  [2 * (x * y + a * z), 1 - 2 * (x * x + z * z), 2 * (y * z - a * x)],
                  [2 * (x * z - a * y), 2 * (y * z + a * x), 1 - 2 * (x * x + y * y)]]).astype(f32)
    dx = (u.astype(f32) - f32(w.cx)) * f32(1.0 / w.fx)
    dy = (v.astype(f32) - f32(w.cy)) * f32(1.0 / w.fx)
    d = [fma(R[i, 0], dx, fma(R[i, 1], dy, R[i, 2])) for i in range(3)]
    inv = f32(1.0) / np.sqrt(fma(d[0], d[0], fma(d[1], d[1], d[2] * d[2])))
    ivs, eps = f32(1.0 / w.voxel), f32(0.4 * w.voxel)
    rg = [(d[i] * inv) * ivs for i in range(3)]
    cg = [fma(f32(pose[i]) - f32(w.origin), ivs, f32(-0.5)) for i in range(3)]
    total, last = 0, None
    for k in range(1, int(nsamp.max()) + 1):
        cell = np.stack([np.floor(fma(f32(k) * eps, rg[i], cg[i])) for i in range(3)])
        ch = np.zeros(nsamp.shape, int) if last is None else (cell != last).sum(0)
        n = np.full(nsamp.shape, 8) if last is None else 8 - (8 >> ch)
        total += int(n[nsamp >= k].sum())
        last = cell
    return total


@pytest.mark.parametrize("n,limits", [(32, (1, 2, 3, 4, 5, 6, 9, 0)), (64, (7, 0))])
def test_every_mode_gives_the_same_image(oracle_mod, n, limits):
    O = oracle_mod
    w = synth.tiny(n=n, width=83, height=61)
    s = synth.Sequence(w)
    m = s.settled_map()
    pose = s.pose7(3)
    # further fields: noise around the camera, so that rays hit at their first samples
    c = w.origin + (np.arange(n) + 0.5) * w.voxel
    Z, Y, X = np.meshgrid(c, c, c, indexing="ij")
    r = np.sqrt((X - pose[0]) ** 2 + (Y - pose[1]) ** 2 + (Z - pose[2]) ** 2)
    noise = [(0.05 * (r / (0.4 * w.voxel) - np.random.default_rng(n).uniform(a, a + 24, r.shape))).astype(f32)
             for a in (-4, -8)]
    for limit in limits:
        md = (limit + 0.5) * 0.4 * w.voxel if limit else 0.0
        for occ in (m[0], *noise):
            samples = {}
            for skip in (0, 1):
                F, p = make_pair(w, O, map_arrays=(occ,) + tuple(m[1:]), skip_empty=skip, max_depth=md)
                ref = O.render(p, occ, m[1], pose)
                for detail in (False, True):
                    F.set_detail_counters(detail)
                    before = F.stats()
                    check_render(F.render(pose), ref)
                    after = F.stats()
                    samples[skip, detail] = after["render_samples"] - before["render_samples"]
                    corners = after["render_unique_corners"] - before["render_unique_corners"]
                    assert detail or corners == 0
                    if detail and not skip:
                        # a ray's samples: up to its hit (a hit at the first sample is -1), or to its end
                        occ_out = O.render(p, np.full_like(occ, -1.0), m[1], pose)["n_samples"]
                        hk = ref["hitk"].reshape(w.height, w.width)
                        if limit and occ_out == limit * hk.size:   # no ray leaves the grid before the limit
                            per_ray = np.where(hk == -1, 1, np.where(hk > 0, hk, limit))
                            assert corners == visited_corners(w, pose, per_ray)
                F.close()
            assert samples[0, False] == samples[0, True] == ref["n_samples"]
            assert samples[1, False] == samples[1, True] <= samples[0, False]
