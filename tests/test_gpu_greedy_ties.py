"""The greedy start where many agents want the same jobs: few different values,
constant rows or columns, identical agents in blocks.  Proposals then follow one
another over tied jobs without a look at the bounds, 128 jobs at a time; the
sizes lie around those windows, the tiles of 64 and the numbers of chains in
flight.  Against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1106_5694_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1106_5694_gb300 import build_ext
    build_ext.build()
    oracle.build()
    B.load()


def _make(kind, n, m=None):
    m = n if m is None else m
    rng = np.random.default_rng(n * 7 + m)
    if kind == "constant":
        a = np.full((n, m), -(2**29) + 1)
    elif kind == "two":
        a = rng.integers(0, 2, size=(n, m))
    elif kind == "five":
        a = rng.integers(-2, 3, size=(n, m))
    elif kind == "rows":  # every job is worth the same to an agent
        a = np.broadcast_to(rng.integers(0, 50, size=(n, 1)), (n, m))
    elif kind == "columns":  # every agent ranks the jobs alike
        a = np.broadcast_to(rng.integers(0, 10**6, size=(1, m)), (n, m))
    else:  # "blocks": identical agents in blocks of 37, jobs in blocks of 150
        a = rng.integers(0, 9, size=((n + 36) // 37, (m + 149) // 150)).repeat(37, 0).repeat(150, 1)[:n, :m]
    return np.ascontiguousarray(a, dtype=np.int32)


KINDS = ["constant", "two", "five", "rows", "columns", "blocks"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", [3, 64, 127, 128, 129, 191, 193, 511, 513, 1537, 2500])
def test_greedy_start_equals_oracle(kind, n):
    a = _make(kind, n)
    d = torch.from_numpy(a).cuda()
    want = oracle.greedy_init(a)
    for _ in range(3):  # (the chains meet differently each time)
        st, sig = B.dgs_greedy_init(d)
        assert st == B.DGS_OK, B.dgs_last_cuda_error()
        np.testing.assert_array_equal(sig.cpu().numpy(), want)


@pytest.mark.parametrize("kind", KINDS)
def test_batched_greedy_start_equals_oracle(kind):
    """A look of a batched instance covers wider tiles, a walk the same 128 jobs."""
    mats = [_make(kind, n) for n in (2, 65, 129, 1000, 1025, 2049)]
    st, _, _, _, stats = B.dgs_solve_batched([torch.from_numpy(a).cuda() for a in mats], max_sweeps=1)
    assert st in (B.DGS_OK, B.DGS_TIMEOUT), B.dgs_last_cuda_error()
    for a, s in zip(mats, stats):
        tau = oracle.greedy_init(a)
        assert s["initial_objective"] == int(a[np.arange(a.shape[0]), tau].astype(np.int64).sum())


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n,m", [(129, 200), (200, 129), (600, 900), (900, 600)])
def test_padded_start_equals_oracle(kind, n, m):
    """Ties at, above and below the dummies' zero, over the real jobs only."""
    for shift in (0, -3):
        a = _make(kind, n, m) + np.int32(shift if kind != "constant" else 2**29 - 1 + shift)
        st_o, assign_o, f_o, sweeps_o = oracle.dgs_rect(a)
        assert st_o == oracle.OK
        st, assign, f, stats = B.dgs_solve_rect(torch.from_numpy(a).cuda())
        assert st == B.DGS_OK, B.dgs_last_cuda_error()
        np.testing.assert_array_equal(assign.cpu().numpy(), assign_o)
        assert f == f_o and stats["sweeps"] == sweeps_o
