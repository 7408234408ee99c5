"""Rules that the kernels' sources keep because no test of results can show
their breach: whether a warp or a CTA does something together must not depend
on how the compiler, or the timing of other CTAs, happens to arrange it."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCES = sorted(glob.glob(os.path.join(ROOT, "paper_1106_5694_gb300", "csrc", "*.cu*")))


def _code(path):
    """The source without its comments."""
    text = re.sub(r"/\*.*?\*/", "", open(path).read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def test_no_mask_is_taken_from_the_threads_that_happen_to_be_there():
    assert SOURCES
    for path in SOURCES:
        assert "__activemask" not in _code(path), path


def test_a_cta_that_sums_together_reads_the_loop_status_as_one():
    """add_objective is a barrier and a warp sum of the whole CTA; a thread that
    returned alone, on a status that another CTA wrote meanwhile, would be
    missing from it."""
    found = 0
    for path in SOURCES:
        for function in re.split(r"\n}\n", _code(path)):
            if "add_objective(st, f);" not in function:
                continue
            found += 1
            body = function[function.rindex("DeviceState* st = w.st;"):]
            returns = re.findall(r"if \(([^;\n]*)\) return;", body)
            assert returns == ["__syncthreads_or(st->status != kRunning)"], (path, returns)
    assert found == 2
