"""Rows of 2^32 16-byte vectors and more: a count of vectors cut to 32 bits was zero, and the host divided by it.  No GPU is visible
to the call, which ends at the launch."""
import os
import subprocess
import sys

import pytest

import paper_2210_00129_b200 as sbp
from paper_2210_00129_b200 import build as sbp_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FAKE = 0x10000          # never reaches a device


@pytest.mark.parametrize("call", [
    f"sbp.sbp_forward_cache(1, {FAKE}, 4, 2 ** 35, {FAKE}, None, 2, {FAKE}, stream=0, check=False)",
    f"sbp.sbp_patch_cache(1, {FAKE}, 1, 64, 64, 2 ** 23, 64, 64, {FAKE}, None, 1, {FAKE}, stream=0, check=False)",
    f"sbp.sbp_patch_scatter(1, {FAKE}, 1, 64, 64, 2 ** 23, 64, 64, {FAKE}, None, 1, {FAKE}, {FAKE}, 256, None, stream=0, check=False)",
    f"sbp.sbp_patch_scatter(1, {FAKE}, 1, 64, 64, 2 ** 23, 1, 64, {FAKE}, None, 1, {FAKE}, {FAKE}, 256, None, stream=0, check=False)",
])
def test_host_side_of_long_rows(call):
    sbp_build.build()
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="", PYTHONPATH=ROOT)
    run = subprocess.run([sys.executable, "-c", f"import paper_2210_00129_b200 as sbp; print({call})"], env=env, cwd=ROOT,
                         capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stderr
    assert int(run.stdout) == sbp.SBP_ERR_CUDA
