"""The tile lists of the map update hold one map's tiles.  Counters that a failed
call left behind must never become writes or reads past a list's end; the
buffers of this check are long enough that either would only show in its
output.  With the counters at zero the lists are those of the frustum."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    from paper_2212_02988_gb300 import build as B
    exe = str(tmp_path_factory.mktemp("fuse_lists") / "fuse_lists_check")
    subprocess.check_call([B.nvcc(), *B.ARCH, "-O1", "-std=c++17", "-fmad=false",
                           "-I" + os.path.join(ROOT, "paper_2212_02988_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "cuda", "fuse_lists_check.cu"), "-o", exe])
    return exe


def test_counters_left_behind_stay_inside_the_lists(checker):
    run = lambda start: [int(x) for x in subprocess.run([checker, str(start)], capture_output=True, text=True,
                                                        check=True).stdout.split()]
    listed, past, took, beyond = run(0)
    assert 100 < listed <= 1024 and past == 0 and took == 1 and beyond == 0
    for start in (500, 509, 512, 600):
        n, past, took, beyond = run(start)
        assert past == 0 and took == 1 and beyond == 0
        assert n == 2 * max(512 - start, 0)   # (more tiles than that are in view)
