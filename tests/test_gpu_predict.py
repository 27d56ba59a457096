"""The prediction at the edges of its IMU reduction (windows shorter than,
equal to and longer than a warp, one sample, none) against the oracle, with
the bars of the rollout test, and its refusal of a covariance that is not
finite wherever the entry lies."""
import numpy as np
import pytest

import synth
from gpu_helpers import make_pair, t
from test_gpu_rollout import check_states, start_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0, 1, 2, 31, 32, 33, 64, 65, 200])
def test_windows_match_oracle(oracle_mod, n):
    O = oracle_mod
    from paper_2212_02988_gb300 import make_state
    w = synth.tiny()
    s = synth.Sequence(w)
    F, p = make_pair(w, O)
    pose, vel, cov = start_state(s, 2)
    rng = np.random.default_rng(n)
    imu = np.concatenate([1.0 + np.arange(n)[:, None] * 1e-3, rng.normal(0, 3, (n, 3)) + [0, -9.8, 0], rng.normal(0, 1, (n, 3))], axis=1)
    F.set_state(make_state(pose, vel, cov))
    got = F.rollout([[imu, imu[: n // 2]]], 0.1, images=False)["states"][0]
    ref, _ = O.rollout(p, O.make_state(pose, vel, cov), [imu, imu[: n // 2]], [0.1, 0.1])
    for g, r in zip(got, ref):
        check_states(g, r)
    F.close()


@pytest.mark.parametrize("i,j,v", [(0, 0, np.nan), (7, 8, np.inf), (11, 2, -np.inf), (9, 9, np.nan)])
def test_covariance_that_is_not_finite_is_refused(oracle_mod, i, j, v):
    from paper_2212_02988_gb300 import PrismError, _lib, make_state, state_arrays
    w = synth.tiny()
    s = synth.Sequence(w)
    F, _ = make_pair(w, oracle_mod, map_arrays=s.settled_map(), s1_pose=s.pose7(0), vel=s.velocity(0))
    f = s.frame(0)
    F.step(None, w.dt, t(f["depth"]), t(f["rgb"]))
    cov = np.eye(12) * 1e-4
    cov[i, j] = v
    F.set_state(make_state(s.pose7(0), s.velocity(0), cov))
    F.render()
    before = F.map_store()
    f = s.frame(1)
    with pytest.raises(PrismError) as e:
        F.step(s.imu_window(1), w.dt, t(f["depth"]), t(f["rgb"]), want_state=True)
    assert e.value.status == _lib.ENOTPD
    after = F.map_store()
    assert all((before[k] == after[k]).all() for k in before)
    F.close()
