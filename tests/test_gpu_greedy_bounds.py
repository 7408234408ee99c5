"""The greedy start by deferred acceptance from tile bounds: sizes around the
edges of its tiles (64 jobs; wider ones for a batched instance above n =
1024), values at the ends of the range, and rows whose best tiles tie, against
the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1106_5694_gb300 import binding as B
from paper_1106_5694_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1106_5694_gb300 import build_ext
    build_ext.build()
    oracle.build()
    B.load()


def _make(kind, n):
    if kind == "peer":
        return inputs.peer_shaped(n, n)
    if kind == "ties":  # every tile of every row reaches the maximum
        return inputs.uniform(n, 0, 3, n)
    a = inputs.uniform(n, -(2**29) + 1, 2**29, n)  # "ends"
    a[::3, ::5] = 2**29 - 1
    a[1::3, 1::7] = -(2**29) + 1
    return a


@pytest.mark.parametrize("kind", ["peer", "ties", "ends"])
@pytest.mark.parametrize("n", [1, 2, 63, 65, 127, 129, 255, 1025, 2051])
def test_greedy_start_equals_oracle(kind, n):
    a = _make(kind, n)
    st, sig = B.dgs_greedy_init(torch.from_numpy(a).cuda())
    assert st == B.DGS_OK
    np.testing.assert_array_equal(sig.cpu().numpy(), oracle.greedy_init(a))


@pytest.mark.parametrize("kind", ["peer", "ties"])
def test_batched_greedy_start_equals_oracle(kind):
    """max_sweeps = 1 would commit exchanges, so the batched start is compared
    through whole solves' initial objectives and results."""
    sizes = [1, 3, 64, 65, 1000, 1023, 1024, 1025, 1100, 2049]
    mats = [_make(kind, n) for n in sizes]
    st, outs, objs, _, stats = B.dgs_solve_batched([torch.from_numpy(a).cuda() for a in mats])
    assert st == B.DGS_OK
    for a, out, obj, s in zip(mats, outs, objs, stats):
        tau = oracle.greedy_init(a)
        assert s["initial_objective"] == int(a[np.arange(a.shape[0]), tau].astype(np.int64).sum())
        ref_st, ref_sig, ref_obj, _ = B.dgs_solve_ex(torch.from_numpy(a).cuda())
        assert ref_st == B.DGS_OK and obj == ref_obj
        np.testing.assert_array_equal(out.cpu().numpy(), ref_sig.cpu().numpy())


@pytest.mark.parametrize("kind", ["negative", "zeros", "ties", "mixed"])
@pytest.mark.parametrize("n,m", [(1, 2), (2, 1), (5, 70), (70, 5), (64, 65), (200, 130), (130, 300), (700, 40)])
def test_padded_start_equals_oracle(kind, n, m):
    """Rectangular instances: benefits below, at and above the dummies' zero,
    with ties between real and dummy pairs."""
    rng = np.random.default_rng(n * 1000 + m)
    lo, hi = {"negative": (-50, 0), "zeros": (0, 1), "ties": (-1, 2), "mixed": (-500, 500)}[kind]
    a = rng.integers(lo, hi, size=(n, m), dtype=np.int32)
    st_o, assign_o, f_o, sweeps_o = oracle.dgs_rect(a)
    assert st_o == oracle.OK
    st, assign, f, stats = B.dgs_solve_rect(torch.from_numpy(a).cuda())
    assert st == B.DGS_OK, B.dgs_last_cuda_error()
    np.testing.assert_array_equal(assign.cpu().numpy(), assign_o)
    assert f == f_o and stats["sweeps"] == sweeps_o
    s = max(n, m)
    square = np.zeros((s, s), np.int32)
    square[:n, :m] = a
    tau = oracle.greedy_init(square)
    assert stats["initial_objective"] == int(square[np.arange(s), tau].astype(np.int64).sum())
