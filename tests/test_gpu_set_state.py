"""set_state runs in stream order: it neither waits nor touches the anchor."""
import numpy as np
import pytest
import torch

import synth
from gpu_helpers import make_pair, t
from test_gpu_track import frames

pytestmark = pytest.mark.gpu


def belief(s, i):
    from paper_2212_02988_gb300 import make_state
    cov = np.diag([1e-6] * 3 + [1e-7] * 3 + [1e-4] * 6)
    return make_state(s.pose7(i), s.velocity(i), cov, n_localised=i + 1)


def test_the_anchor_stays(oracle_mod):
    """The anchor loaded before the state is written localises as one loaded after it; the
    written state reads back exactly."""
    from paper_2212_02988_gb300 import state_arrays
    w = synth.ROOM64
    s = synth.Sequence(w)
    out = []
    for anchor_first in (True, False):
        F, _ = make_pair(w, oracle_mod)
        A, a_d, a_rgb, f = frames(s, w, 3, 4)
        if anchor_first:
            F.anchor_load(A, t(a_d), t(a_rgb))
            F.step(None, w.dt, t(f["depth"]), t(f["rgb"]))   # work in flight when the state is written
            F.anchor_load(A, t(a_d), t(a_rgb))
        F.set_state(belief(s, 3))
        back, want = state_arrays(F.get_state()), state_arrays(belief(s, 3))
        assert np.array_equal(back["cov"], want["cov"]) and np.array_equal(back["vel"], want["vel"])
        assert np.array_equal(back["pose"][:3], want["pose"][:3]) and back["n_localised"] == want["n_localised"]
        np.testing.assert_allclose(back["pose"], want["pose"], rtol=0, atol=4e-16)   # (the quaternion normalised)
        if not anchor_first:
            F.anchor_load(A, t(a_d), t(a_rgb))
        F.predict(s.imu_window(4), w.dt)
        out.append(state_arrays(F.localise(t(f["depth"]), t(f["rgb"]))))
        F.close()
    assert all(np.array_equal(out[0][k], out[1][k]) for k in ("pose", "vel", "cov"))


@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_a_mapping_loop_without_waits(storage):
    """States and frames written back to back give the map of a loop that waits after each call."""
    from paper_2212_02988_gb300 import Filter, config
    w = synth.ROOM64
    s = synth.Sequence(w)
    fr = [(belief(s, i), t(s.frame(i)["depth"]), t(s.frame(i)["rgb"])) for i in range(6)]
    maps = []
    for wait in (False, True):
        F = Filter(config(w.n, w.extent, w.width, w.height, storage=storage), fr[0][0], device=0)
        for b, d, c in fr:
            F.set_state(b)
            if wait:
                torch.cuda.synchronize()
            F.update_map(d, c)
            if wait:
                torch.cuda.synchronize()
        maps.append(F.map_store())
        F.close()
    for k in ("occ", "rgb", "var_occ", "var_rgb"):
        assert torch.equal(maps[0][k], maps[1][k]), k
