"""`[C_out, C_in]` weights: the call for dX alone asks for the workspace at every weight size, not only where copies are made.  No GPU is
visible to the calls, which end at the check or at the launch."""
import os
import subprocess
import sys

import pytest

import paper_2210_00129_b200 as sbp
from paper_2210_00129_b200 import build as sbp_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("dt,C_in,C_out", [(0, 64, 64), (0, 768, 768), (1, 128, 256), (1, 768, 3072)])
def test_dx_alone(dt, C_in, C_out):
    sbp_build.build()
    code = f"""
import paper_2210_00129_b200 as sbp
p, ws = 0x10000, sbp.sbp_linear_backward_workspace_bytes({dt}, 64, 32, {C_in}, {C_out})
call = lambda flags, space, n: sbp.sbp_linear_backward({dt}, None, p, p, p, None, 64, 32, {C_in}, {C_out}, None, None, p, flags, space, n,
                                                       None, stream=0, check=False)
print(call(64, None, 0), call(64, p, ws - 1), call(64, p, ws), call(0, None, 0))
"""
    run = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, CUDA_VISIBLE_DEVICES="", PYTHONPATH=ROOT), cwd=ROOT,
                         capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stderr
    short, enough = sbp.SBP_ERR_WORKSPACE, sbp.SBP_ERR_CUDA              # (without the flag dX alone needs no workspace)
    assert [int(v) for v in run.stdout.split()] == [short, short, enough, enough]
