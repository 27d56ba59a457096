"""The Adam kernel at the edges of its pixel range: a warp of drawn
pixels and one more, every thread of the block.  The observation of a step is loaded
during the step before it, so a second step tests the handed-over draw.

The bars are those of the first steps in test_gpu_adam.py: step 1 moves every
component by exactly its step size; in step 2 a component's FP32 gradient error
counts, and the bar is 1 % of a step.  (A single pixel on an axis-aligned wall
has gradient components that are zero but for rounding, whose sign decides the
step: it has no bar.)"""
import numpy as np
import pytest

import synth
from gpu_helpers import quat_angle_deg
from test_gpu_adam import localise_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pixels", [33, 256])
@pytest.mark.parametrize("steps", [1, 2])
def test_draws_at_the_edges_of_the_range(oracle_mod, pixels, steps):
    w = synth.ROOM64
    got, ref = localise_both(oracle_mod, w, synth.Sequence(w), 3, 4, adam_steps=steps, adam_pixels=pixels)
    dt = np.linalg.norm(got["pose"][:3] - ref["pose"][:3])
    da = np.radians(quat_angle_deg(got["pose"][3:], ref["pose"][3:]))
    if steps == 1:
        assert dt < 1e-9 and da < 1e-8
    else:
        assert dt < 1e-2 * 1e-3 and da < 1e-2 * 3.6e-4
