"""Evaluations that find the range of the matrix as they read it: matrices
whose sampled elements allow packed keys while other elements do not, values
out of range, and bad permutations, against the oracle and the status that the
range check comes first with."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1106_5694_gb300 import binding as B
from paper_1106_5694_gb300 import inputs

pytestmark = pytest.mark.gpu

LIMIT = 1 << 29  # |a| below it


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1106_5694_gb300 import build_ext
    build_ext.build()
    oracle.build()
    B.load()


def _small(n, seed):
    rng = np.random.default_rng(seed)
    return rng.integers(-100, 100, (n, n)).astype(np.int32)


@pytest.mark.parametrize("n", [4, 64, 68, 128, 260, 516])
@pytest.mark.parametrize("value", [LIMIT - 1, -(LIMIT - 1), 1 << 22])
def test_outliers_that_a_sample_may_miss(n, value):
    tau = inputs.random_permutation(n, n)
    for seed in range(3):
        a = _small(n, seed)
        rng = np.random.default_rng(100 + seed)
        a[rng.integers(n), rng.integers(n)] = value
        a[n - 1, n - 1] = value // 2
        st, *got = B.dgs_evaluate(torch.from_numpy(a).cuda(), torch.from_numpy(tau).cuda())
        assert st == B.DGS_OK
        for g, e in zip(got, oracle.evaluate_all(a, tau)):
            np.testing.assert_array_equal(g.cpu().numpy(), e)


@pytest.mark.parametrize("n", [4, 64, 260])
@pytest.mark.parametrize("value", [LIMIT, -LIMIT, np.iinfo(np.int32).min, np.iinfo(np.int32).max])
@pytest.mark.parametrize("bad_start", [False, True])
def test_values_out_of_range(n, value, bad_start):
    tau = inputs.random_permutation(n, n)
    if bad_start:
        tau = tau.copy()
        tau[1] = tau[0]
    for at in ((0, 0), (n - 1, n - 2), (n // 2, n - 1)):
        a = _small(n, 7)
        a[at] = value
        st, *got = B.dgs_evaluate(torch.from_numpy(a).cuda(), torch.from_numpy(tau).cuda())
        assert st == B.DGS_ERR_RANGE
        assert all(bool((g == 0).all()) for g in got[0::2]) and all(bool((g == -1).all()) for g in got[1::2])
