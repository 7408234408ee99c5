"""Kernels whose dynamic shared memory depends on n, in processes of their own:
which kernel's limit was raised before must not matter, whatever public call
raised it.  Each result against another route of the library."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = """
import sys
sys.path.insert(0, {root!r})
import torch
from paper_1106_5694_gb300 import binding as B

def matrix(n, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randint(0, 10016, (n, n), generator=g, device="cuda", dtype=torch.int32)

def evaluate(n):
    st, *_ = B.dgs_evaluate(matrix(n, n), torch.arange(n, device="cuda", dtype=torch.int32))
    assert st == B.DGS_OK, B.dgs_last_cuda_error()

def batch(*sizes):
    mats = [matrix(n, n) for n in sizes]
    st, outs, objs, _, _ = B.dgs_solve_batched(mats, max_sweeps=40)
    assert st in (B.DGS_OK, B.DGS_TIMEOUT), (st, B.dgs_last_cuda_error())
    for a, out, obj in zip(mats, outs, objs):
        ref_st, ref, ref_obj, _ = B.dgs_solve_ex(a, max_sweeps=40)
        assert ref_st in (B.DGS_OK, B.DGS_TIMEOUT), B.dgs_last_cuda_error()
        assert obj == ref_obj and torch.equal(out, ref)
"""


def _run(code, **env):
    r = subprocess.run([sys.executable, "-c", PRELUDE.format(root=ROOT) + code], capture_output=True, text=True,
                       timeout=300, env={**os.environ, **env})
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-3000:]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1106_5694_gb300 import build_ext
    build_ext.build()


# A batch above n = 4096 takes the row task kernel of 512 threads; above n =
# 8192 its rows need more shared memory than a kernel has by default.
@pytest.mark.parametrize("code", ["evaluate(256); batch(9000, 64)",
                                  "batch(9000, 64); evaluate(256); batch(12300, 65)",
                                  "batch(64, 4097); batch(12300); evaluate(4096); batch(9000)"])
def test_batches_of_large_instances_beside_evaluations(code):
    _run(code)


def test_served_large_instance_after_an_evaluation():
    _run("""
evaluate(256)
a = matrix(9000, 1)
s = B.Server(4 << 30)
st, t = s.dgs_submit(a)
assert st == B.DGS_OK
res = s.dgs_server_wait(t)
ref_st, ref, ref_obj, _ = B.dgs_solve_ex(a)
assert res[0] == B.DGS_OK == ref_st, (res[0], B.dgs_last_cuda_error())
assert res[2] == ref_obj and torch.equal(torch.as_tensor(res[1]).cpu(), ref.cpu())
""", DGS_SERVER_SOLO_N="0")


# 48 KB of a kernel's shared memory need no raised limit, static and dynamic
# taken together: rows of exactly 48 KB beside the static part do.
@pytest.mark.parametrize("n,evaluation,other", [(12225, "TILE_PAIRS", "ROW_OWNER"), (12288, "TILE_PAIRS", "ROW_OWNER"),
                                                (6144, "ROW_OWNER", "TILE_PAIRS"), (6081, "ROW_OWNER", "TILE_PAIRS")])
def test_rows_of_48_kb_in_a_fresh_process(n, evaluation, other):
    _run(f"""
a = matrix({n}, 1)
st, sig, f, _ = B.dgs_solve_ex(a, max_sweeps=40, evaluation=B.DGS_EVAL_{evaluation})
assert st in (B.DGS_OK, B.DGS_TIMEOUT), (st, B.dgs_last_cuda_error())
big = matrix(12800, 2)  # raises every limit
assert B.dgs_solve_ex(big, max_sweeps=1, evaluation=B.DGS_EVAL_{evaluation})[0] in (B.DGS_OK, B.DGS_TIMEOUT)
st, ref, ref_f, _ = B.dgs_solve_ex(a, max_sweeps=40, evaluation=B.DGS_EVAL_{other})
assert st in (B.DGS_OK, B.DGS_TIMEOUT), (st, B.dgs_last_cuda_error())
assert f == ref_f and torch.equal(sig, ref)
""")


@pytest.mark.parametrize("n", [6144, 6110])
def test_sequential_algorithm_of_48_kb_in_a_fresh_process(n):
    _run(f"""
def seq(a):
    st, sig, f, _ = B.dgs_solve_ex(a, max_sweeps=5, algorithm=B.DGS_ALG_SEQUENTIAL)
    assert st in (B.DGS_OK, B.DGS_TIMEOUT), (st, B.dgs_last_cuda_error())
    return sig, f

a = matrix({n}, 1)
sig, f = seq(a)
seq(matrix(6400, 2))  # raises the limit
ref, ref_f = seq(a)
assert f == ref_f and torch.equal(sig, ref)
""")
