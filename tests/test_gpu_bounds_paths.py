"""The bounds-checking debug build on the paths that need larger problems, jobs or
batches (see tests/bounds_probe_paths.py): no check may fire, and the results still
match the oracle (the specification's bounds: 1e-5, motion gradients 1e-3)."""
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


def test_bounds_checks_of_jobs_batches_and_copied_rows():
    from paper_2401_09283_gb300 import build
    lib = build.build_library(variant="bounds")
    r = subprocess.run([sys.executable, os.path.join(HERE, "bounds_probe_paths.py")],
                       env=dict(os.environ, BP_GB300_LIB=lib), capture_output=True, text=True,
                       timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    print(out)
    assert out["library"] == lib
    assert out["flags"] == 0 and out["first"] == -1, out
    for name, e_vol, e_grad, same in out["cases"]:
        assert e_vol <= 1e-5 and e_grad <= 1e-3 and same, (name, e_vol, e_grad, same)
