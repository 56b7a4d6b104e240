"""The projector's bounded wait (csrc/async.cuh) gives every lane of a warp the same verdict: when the
phase completes, when some lanes have given up before it completes, and when the limit runs out."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_a_wait_has_one_verdict_per_warp(tmp_path):
    from paper_1008_2042_gb300 import build

    exe = str(tmp_path / "waits")
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, os.path.join(HERE, "waits.cu"), "-o", exe],
                   check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=60).stdout
    completes, split, runs_out = [tuple(map(int, line.split())) for line in out.splitlines()]
    assert completes == (32, 0)
    assert split == (0, 1)
    assert runs_out == (0, 1)
