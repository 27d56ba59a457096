"""The descent step over more frames than one launch takes, each frame with a
pose, a depth and a colour of its own: the loss is the sum of the single frames' losses
(bar: 2^-53 of it for each FP64 addition, one a block and frame), and the step is the
oracle's over all frames (bars of test_gpu_mapping).  A frame left out, read at
another frame's offset or rendered with another frame's matrices misses both
bars.  And a residual whose square passes FP32's range, in one frame."""
import numpy as np
import pytest

import synth
from gpu_helpers import bf16_round, make_pair, t
from test_gpu_mapping import check_change

pytestmark = pytest.mark.gpu

SD, SC = 0.02, 0.1
LR_OCC, LR_RGB = 2e-7, 2e-6


def problem(n):
    """Frames that differ by far more than the bars: the last one of a launch and
    those past it look elsewhere and are further off the map."""
    w = synth.tiny(n=32, width=83, height=61)
    s = synth.Sequence(w, n_frames=72)
    occ, rgb, vo, vr = s.settled_map()
    occ = (occ - np.float32(0.03)).astype(np.float32)
    fr = [s.frame(j) for j in range(n)]
    poses = np.stack([s.pose7(j) for j in range(n)])
    D = np.stack([f["depth"] for f in fr])
    C = np.stack([f["rgb"] for f in fr])
    D *= (1 + 0.01 * np.arange(n, dtype=np.float32) / n)[:, None, None]
    D[31:] *= np.float32(1.05)
    D[:, ::7, ::5] = np.nan
    D[:, 1::9] = 0.0
    return w, (occ, rgb, vo, vr), poses, D, C


@pytest.mark.parametrize("n,storage", [(1, "f32"), (32, "f32"), (33, "bf16"), (65, "f32")])
def test_loss_and_step_over_batches(oracle_mod, n, storage):
    O = oracle_mod
    w, m, poses, D, C = problem(n)
    F, p = make_pair(w, O, storage=storage, map_arrays=m)
    one = lambda q, d, c, a=0.0, b=0.0: F.map_descent(q, t(d), t(c), SD, SC, a, b)
    prior = one(poses[:1], np.zeros_like(D[:1]), C[:1])
    single = [one(poses[j:j + 1], D[j:j + 1], C[j:j + 1]) - prior for j in range(n)]
    total = one(poses, D, C)
    blocks = ((w.width + 15) // 16) * ((w.height + 7) // 8)
    assert min(single) > 1e-3 * total / n
    assert abs(total - (sum(single) + prior)) <= 2 * n * (blocks + 16) * 2.0 ** -53 * total
    start = [bf16_round(a) if storage == "bf16" else a for a in m[:2]]
    one(poses, D, C, LR_OCC, LR_RGB)
    got = {k: v.cpu().numpy() for k, v in F.map_store().items()}
    occ_r, rgb_r, loss_r = O.map_descent(p, start[0], start[1], list(poses), list(D), list(C), SD, SC, LR_OCC, LR_RGB)
    assert abs(total - loss_r) <= 1e-3 * loss_r
    if storage == "f32":
        check_change(got["occ"], m[0], occ_r, "occ")
        check_change(got["rgb"], m[1], rgb_r, "rgb")
    else:   # half a unit of bfloat16 more: the stored mean is rounded
        for name, a, r in (("occ", start[0], occ_r), ("rgb", start[1], rgb_r)):
            d = np.abs(r - a)
            err = np.abs(got[name] - r)
            assert np.all(err <= 1e-4 * d.max() + 5e-3 * d + 2.0 ** -8 * np.abs(r) * 1.01), name
    assert np.abs(occ_r - start[0]).max() > 1e-4   # (the oracle moved the map)
    F.close()


def test_a_residual_beyond_fp32(oracle_mod):
    w, m, poses, D, C = problem(1)
    F, _ = make_pair(w, oracle_mod, map_arrays=m)
    assert F.render(poses[0])["hitk"][30, 40] >= 2 and np.isfinite(D[0, 30, 40]) and D[0, 30, 40] > 0
    C[0, 30, 40] = 3e25          # all three channels: their squares pass FP32's range
    total = F.map_descent(poses, t(D), t(C), SD, SC, 0.0, 0.0)
    assert total == pytest.approx(3 * 0.5 * float(np.float32(3e25)) ** 2 / 0.01, rel=1e-6)
    F.close()
