"""The rule that chooses the sweep kernel by a launch's tiles and the device's SMs."""
import os
import shutil
import subprocess

import pytest

from test_pose_math import CSRC, HERE

TILES, STREAM, ROWS, ROWS_FEW = range(4)


@pytest.fixture(scope="module")
def modes(tmp_path_factory):
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("sweep_mode") / "sweep_mode")
    res = subprocess.run([exe, "-x", "cu", "-gencode=arch=compute_103a,code=sm_103a", "-std=c++17", "-I", CSRC, "-o",
                          out, os.path.join(HERE, "math_host", "sweep_mode.cu")], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-4000:]

    def query(pairs):
        res = subprocess.run([out], input="\n".join("%d %d" % p for p in pairs), capture_output=True, text=True)
        assert res.returncode == 0
        return [tuple(map(int, line.split())) for line in res.stdout.splitlines()]

    return query


def test_limits_at_152_sms(modes):
    got = dict(zip([1, 76, 77, 114, 115, 304, 305, 608, 609, 12288],
                   modes([(n, 152) for n in [1, 76, 77, 114, 115, 304, 305, 608, 609, 12288]])))
    assert [got[n][0] for n in (1, 114, 115, 304, 305, 608, 609, 12288)] == \
        [ROWS_FEW, ROWS_FEW, ROWS, ROWS, TILES, TILES, STREAM, STREAM]
    assert [got[n][1] for n in (1, 76, 77, 114, 304, 12288)] == [ROWS, ROWS, TILES, TILES, TILES, TILES]


@pytest.mark.parametrize("sms", [1, 20, 76, 132, 148])
def test_limits_follow_the_sms(modes, sms):
    """Rows with more registers only where all row blocks (4 a tile) fit at 3 per SM, FP64
    rows where they fit at 2; streamed stores only above one wave of 4 blocks per SM."""
    sizes = range(1, 6 * sms + 2)
    for n, (f32, f64) in zip(sizes, modes([(n, sms) for n in sizes])):
        assert f32 == (ROWS_FEW if 4 * n <= 3 * sms else ROWS if n <= 2 * sms else TILES if n <= 4 * sms else STREAM)
        assert f64 == (ROWS if 4 * n <= 2 * sms else TILES)
