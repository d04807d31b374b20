"""A footprint that never arrives: the bounded waits run out, the kernels return NaN,
and the context stays usable.  Runs in the debug build, whose waits are short and where
the copies of one view can be left out (bp_bounds_check, op 3)."""
import json
import os
import subprocess
import sys

import pytest
import torch

pytestmark = [pytest.mark.gpu, pytest.mark.slow]

if not torch.cuda.is_available():  # pragma: no cover - GPU machine only
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

HERE = os.path.dirname(os.path.abspath(__file__))


def test_lost_copy_ends_in_nan_and_leaves_the_context_usable():
    from paper_2401_09283_gb300 import build
    env = dict(os.environ, BP_GB300_LIB=build.build_library(variant="bounds"))
    r = subprocess.run([sys.executable, os.path.join(HERE, "lost_copy_probe.py")], env=env,
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    print(out)
    # the waits last a 64th of the release build's, 2^14 tries of 3 us in that build: eight
    # calls of each type lose a copy in one kernel at least
    assert out["seconds"] >= 8 * 0.03
    for dtype in ("torch.float32", "torch.bfloat16"):
        for name, q in out[dtype].items():
            assert q["finite"], (dtype, name)
            # (the fused kernel's motion part too: its sums have a fixed order)
            assert q["same after"], (dtype, name)
            if name in ("motion", "both", "exact"):
                # (the view before it may still be summed when the wait runs out)
                assert q["early kept"] and q["lost nan"], (dtype, name, q)
            elif name == "batch-half":  # the batch's forward does not stage these tiles
                assert 0.0 < q["nan"] < 1.0, (dtype, name, q)
            else:  # every voxel, and through the loss every view of a job
                assert q["nan"] == 1.0, (dtype, name, q)
