"""The descent step's loss over more frames than one launch takes, with
invalid depths and residuals whose squares leave FP32's range: a zero step
over n frames reports the sum of the single frames' losses (each less the
prior's share, which a frame without a valid depth reports alone)."""
import numpy as np
import pytest
import torch

import synth
from gpu_helpers import make_pair, t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,storage", [(1, "f32"), (32, "f32"), (33, "bf16"), (65, "f32")])
def test_loss_is_the_sum_over_frames(oracle_mod, n, storage):
    w = synth.tiny(n=32, width=83, height=61)
    s = synth.Sequence(w)
    F, _ = make_pair(w, oracle_mod, storage=storage, map_arrays=s.settled_map())
    frames = [s.frame(i % 5) for i in range(n)]
    poses = np.stack([s.pose7(i % 5) for i in range(n)])
    D = np.stack([f["depth"] for f in frames])
    C = np.stack([f["rgb"] for f in frames])
    D[:, ::7, ::5] = np.nan
    D[:, 1::9] = 0.0
    C[0, 30, 40] = 3e25          # all three channels: their squares pass FP32's range
    one = lambda p, d, c: F.map_descent(p, t(d), t(c), 0.02, 0.1, 0.0, 0.0)
    prior = one(poses[:1], np.zeros_like(D[:1]), C[:1])
    assert 0 < prior < np.inf
    single = [one(poses[j:j + 1], D[j:j + 1], C[j:j + 1]) - prior for j in range(n)]
    total = one(poses, D, C)
    # FP64 sums of the same FP32 residuals, in another order
    assert abs(total - (sum(single) + prior)) <= 1e-11 * abs(total)
    # the large residual, if its pixel renders a surface
    if F.render(poses[0])["hitk"][30, 40] >= 2 and np.isfinite(D[0, 30, 40]) and D[0, 30, 40] > 0:
        assert total == pytest.approx(3 * 0.5 * float(np.float32(3e25)) ** 2 / 0.01, rel=1e-6)
    F.close()
