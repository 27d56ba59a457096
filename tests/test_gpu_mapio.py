"""Map exchange by segments: rows shorter than, equal to and longer than a
segment, unequal axes, both storages, any subset of the arrays, tensors at odd
offsets; what comes out is what went in (rounded to the storage), arrays left
out stay, and the render's clamped corners (ghost cells) see the edge voxels."""
import numpy as np
import pytest
import torch

from gpu_helpers import t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(8, 8, 8), (8, 16, 120), (16, 8, 128), (8, 8, 136), (24, 40, 264)])
@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_exchange(shape, storage):
    from paper_2212_02988_gb300 import Filter, config
    nz, ny, nx = shape
    F = Filter(config(max(shape), 4.0, 33, 25, storage=storage, nx=nx, ny=ny, nz=nz, origin=(0.0, 0.0, 0.0)), device=0)
    rng = np.random.default_rng(nx)

    def odd(sh):   # contiguous, its first element 4 bytes past a 16-byte boundary
        n = int(np.prod(sh))
        return t(rng.normal(size=n + 1).astype(np.float32))[1:].view(sh)

    kept = (lambda x: x.to(torch.bfloat16).float()) if storage == "bf16" else (lambda x: x)
    occ, rgb, vo, vr = odd(shape), odd(shape + (3,)), odd(shape).abs(), odd(shape).abs()
    F.map_load(occ, rgb, vo, vr)
    m = F.map_store()
    for k, x in (("occ", occ), ("rgb", rgb), ("var_occ", vo), ("var_rgb", vr)):
        assert torch.equal(m[k], kept(x)), k
    occ2, vr2 = odd(shape), odd(shape).abs()
    F.map_load(occ2, None)
    F.map_load(None, None, None, vr2)
    m = F.map_store()
    for k, x in (("occ", occ2), ("rgb", rgb), ("var_occ", vo), ("var_rgb", vr2)):
        assert torch.equal(m[k], kept(x)), k
    # a constant map but for one voxel layer at each face: rays that end beside a
    # face interpolate with its ghosts, which hold the face's own values
    F.map_load(torch.full(shape, -1.0, device="cuda"), torch.zeros(shape + (3,), device="cuda"))
    face = torch.full(shape, -1.0, device="cuda")
    face[:, :, 0] = face[:, :, -1] = face[:, 0] = face[:, -1] = face[0] = face[-1] = 1.0
    F.map_load(face, torch.ones(shape + (3,), device="cuda"))
    vs = 4.0 / max(shape)
    pose = np.array([0.5 * nx * vs, 0.5 * ny * vs, 0.5 * nz * vs, 0.5, -0.5, 0.5, -0.5])
    out = F.render(pose)
    assert (out["hitk"] > 1).all() and torch.allclose(out["rgb"], torch.ones_like(out["rgb"]))
    F.close()
