"""Frames whose sizes leave the server's 32x8 packing tiles partly empty on
either side, two such streams in one batch: the packed anchors decide the next
frame's localisation, whose state must be prism_step's bit for bit."""
import dataclasses

import pytest

import synth
from test_gpu_serve import run_filter, run_server, same_state, stream_spec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(81, 57), (65, 64), (95, 49)])
def test_partial_packing_tiles(size):
    odd = dataclasses.replace(synth.ROOM64, width=size[0], height=size[1])
    specs = [stream_spec(odd, 5, 3, "settled"), stream_spec(synth.ROOM64, 6, 3, "settled")]
    res, _, _ = run_server(specs, "f32")
    for got, spec in zip(res, specs):
        ref, _ = run_filter(spec, "f32")
        assert len(got) == len(ref) == 3
        assert all(same_state(a, b) for a, b in zip(got, ref))
