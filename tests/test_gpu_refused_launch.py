"""A launch that the runtime refuses inside a device-side loop ends the call
with an error status and leaves the library usable (in a process of its own)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import os, sys
sys.path.insert(0, {root!r})
import torch
from paper_1106_5694_gb300 import binding as B
from paper_1106_5694_gb300 import inputs
a = torch.from_numpy(inputs.peer_shaped({n}, 1)).cuda()
opts = dict(algorithm=B.{algorithm}, max_sweeps=20)
os.environ["DGS_FAKE_LOOP_REFUSAL"] = "1"
for _ in range(3):
    assert B.dgs_solve_ex(a, **opts)[0] == B.DGS_ERR_CUDA
    assert "loop body" in B.dgs_last_cuda_error(), B.dgs_last_cuda_error()
del os.environ["DGS_FAKE_LOOP_REFUSAL"]
st, sig, f, _ = B.dgs_solve_ex(a, **opts)
assert st in (B.DGS_OK, B.DGS_TIMEOUT), B.dgs_last_cuda_error()
assert torch.equal(torch.sort(sig).values, torch.arange({n}, device="cuda", dtype=torch.int32))
assert f == int(a[torch.arange({n}, device="cuda"), sig.long()].long().sum())
"""


@pytest.mark.parametrize("algorithm", ["DGS_ALG_PARALLEL", "DGS_ALG_SEQUENTIAL"])
def test_refused_launch_in_a_loop_body(algorithm):
    from paper_1106_5694_gb300 import build_ext
    build_ext.build()
    r = subprocess.run([sys.executable, "-c", CODE.format(root=ROOT, algorithm=algorithm, n=1000)],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, f"exit {r.returncode}: " + r.stdout[-2000:] + r.stderr[-3000:]
