"""The descent's loss is as good as an FP64 sum of the squared FP32 residuals
over the whole range of FP32: residuals whose squares add up past FP32's
largest value, squares that FP32 cannot hold, and every size together.  Bar:
2^-53 of the sum for each addition that the sum takes in FP64 (a block's or, for
squares outside FP32's comfortable range, a thread's)."""
import math

import numpy as np
import pytest
import torch

import synth
from gpu_helpers import make_pair, t

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.mark.parametrize("kind", ["plain", "large", "tiny", "mixed"])
def test_prior_term(kind):
    from paper_2212_02988_gb300 import Filter, config
    nx, ny, nz = 136, 24, 40
    F = Filter(config(nx, 4.0, 33, 25, nx=nx, ny=ny, nz=nz, init_occ=0.0, init_rgb=0.25, tau=1e30), device=0)
    rng = np.random.default_rng(5)
    size = 4 * nx * ny * nz
    v = {"plain": lambda: rng.normal(size=size), "large": lambda: np.full(size, 9.9e17),
         "tiny": lambda: np.full(size, 1e-25) * rng.choice([-1, 1], size),
         "mixed": lambda: 10.0 ** rng.uniform(-30, 30, size) * rng.choice([-1, 0, 1], size)}[kind]().astype(np.float32)
    occ, rgb = v[:nx * ny * nz].reshape(nz, ny, nx), v[nx * ny * nz:].reshape(nz, ny, nx, 3)
    if kind == "tiny":
        rgb = np.full_like(rgb, 0.25)
    F.map_load(t(occ), t(rgb))
    pose = np.array([0.0, 0, 0, 1, 0, 0, 0])
    z = torch.zeros((1, 25, 33), device="cuda")
    loss = F.map_descent(pose[None], z, torch.zeros((1, 25, 33, 3), device="cuda"), 0.02, 0.1, 0.0, 0.0)
    dm = np.concatenate([(occ - np.float32(0.0)).ravel(), (rgb - np.float32(0.25)).ravel()]).astype(np.float64)
    want = math.fsum(dm * dm) * (0.5 / F.cfg.prior_var)   # (each square is exact in FP64)
    rows = (ny + 2) * (nz + 2)
    adds = rows if kind in ("plain",) else 32 * rows * 8   # at most one a block, or a few a lane of every row
    assert 0 < want < math.inf
    assert abs(loss - want) <= (adds + 8) * U * want, (loss, want)
    F.close()


def test_frame_term_beyond_fp32(oracle_mod):
    w = synth.tiny(n=32, width=83, height=61)
    s = synth.Sequence(w)
    F, _ = make_pair(w, oracle_mod, map_arrays=s.settled_map())
    poses = np.stack([s.pose7(i) for i in (2, 4)])
    D = np.stack([s.frame(i)["depth"] for i in (2, 4)])
    C = np.full((2, w.height, w.width, 3), 9.9e17, np.float32)
    n = sum(int(((F.render(p)["hitk"].cpu().numpy() >= 2) & np.isfinite(d) & (d > 0)).sum()) for p, d in zip(poses, D))
    loss = F.map_descent(poses, t(D), t(C), 0.02, 0.1, 0.0, 0.0)
    # the rendered colours and the other terms are lost beside 9.9e17
    want = 3 * n * float(np.float32(9.9e17)) ** 2 * (0.5 / (0.1 * 0.1))
    assert n > 4000
    assert abs(loss - want) <= (2 * w.width * w.height + 8) * U * want, (loss, want)
    F.close()
