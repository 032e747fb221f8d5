"""IDKM_NO_COOP: a launch per iteration whatever the weights' dimension (B200 only)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = """
import sys, torch
from paper_2312_07759_b200 import binding as B
d, k = int(sys.argv[1]), int(sys.argv[2])
W = torch.randn(20000, d, device="cuda") * 0.03
ctx = B.Context()
ctx.forward(W, W[:k].contiguous(), 0.01, 0.0, 25)
torch.cuda.synchronize()
print(ctx.launches)
"""


@pytest.mark.parametrize("d,k", [(1, 4), (1, 40), (2, 4), (4, 16)])
def test_every_iteration_is_a_launch(d, k):
    n = {}
    for off in ("", "1"):
        env = {key: v for key, v in os.environ.items() if key != "IDKM_NO_COOP"}
        if off:
            env["IDKM_NO_COOP"] = off
        out = subprocess.run([sys.executable, "-c", PROGRAM, str(d), str(k)], env=env, cwd=ROOT, capture_output=True, text=True, timeout=300)
        assert out.returncode == 0, out.stderr
        n[off] = int(out.stdout)
    assert n[""] <= 4 and n["1"] >= 25
