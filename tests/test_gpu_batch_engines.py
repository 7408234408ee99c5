"""Batched calls that reuse an engine of an earlier call: other instances,
counts and sizes of the same classes, calls from several threads at once, and
after dgs_release_cached_memory, each against the single solve."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1106_5694_gb300 import binding as B
from paper_1106_5694_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1106_5694_gb300 import build_ext
    build_ext.build()
    B.load()


def _check(sizes, seed):
    mats = [torch.from_numpy(inputs.peer_shaped(n, seed + k)).cuda() for k, n in enumerate(sizes)]
    st, outs, objs, statuses, _ = B.dgs_solve_batched(mats)
    assert st == B.DGS_OK and set(statuses) == {B.DGS_OK}
    for a, out, obj in zip(mats, outs, objs):
        ref_st, ref, ref_obj, _ = B.dgs_solve_ex(a)
        assert ref_st == B.DGS_OK and obj == ref_obj
        np.testing.assert_array_equal(out.cpu().numpy(), ref.cpu().numpy())


def test_reused_engine_gives_the_single_solves_results():
    for seed, sizes in enumerate([[70, 255, 256], [256] * 16, [1], [33, 100], [257, 300, 384], [90] * 17]):
        _check(sizes, 10 * seed)
    assert B.dgs_release_cached_memory() == B.DGS_OK
    _check([70, 200], 99)


def test_concurrent_batched_calls_use_engines_of_their_own():
    errors = []

    def work(seed):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for r in range(4):
                    _check([60 + 7 * seed, 128, 200 + r], 1000 * seed + 10 * r)
        except BaseException as e:  # noqa: BLE001 - reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
