"""Host-side arithmetic of batches at the ends of their range, on the CPU: the
library's own functions in a small program."""
import shutil
import subprocess

import pytest

from paper_1106_5694_gb300 import build_ext

DEVICE_BYTES = 300 * 10**9  # more than a GB300 has


def _run(tmp_path, body):
    nvcc = build_ext._nvcc()
    if shutil.which(nvcc) is None:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "limits.cu", tmp_path / "limits"
    src.write_text('#include <cstdio>\n#include <cstdint>\n#include "dgs_internal.cuh"\nint main() {\n' + body + "\n}\n")
    subprocess.check_call([nvcc, *build_ext.ARCH, "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-I", build_ext.CSRC,
                           "-o", str(exe), str(src)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
    return r.stdout


def test_queued_row_weights_fit_their_prefix_sums(tmp_path):
    """As many instances of one size as their transposed copies leave room for,
    half the rows of each queued; the sum is kept in int32."""
    _run(tmp_path, f"""
    for (int64_t n = 1; n <= DGS_BATCH_MAX_N; ++n) {{
        const int64_t most = {DEVICE_BYTES}ll / (4 * n * ((n + 63) / 64 * 64));
        for (int64_t slots = most; slots > 0; slots /= 2) {{
            const int64_t sum = slots * (n / 2) * dgs::row_weight((int32_t)n, (int32_t)slots);
            if (sum > INT32_MAX) {{ printf("%lld instances of %lld: %lld\\n", (long long)slots, (long long)n, (long long)sum); return 1; }}
        }}
    }}
    return 0;""")


def test_engine_slots_cover_the_count_and_waste_nothing_that_is_not_kept(tmp_path):
    _run(tmp_path, """
    for (int64_t c = 1; c <= INT32_MAX; c += 1 + c / 64) {
        const int64_t s = dgs::engine_slots((int32_t)c);
        if (s < c || (s > 4096 && s != c) || (s <= 4096 && s > 16 && 2 * s > 3 * c)) { printf("%lld: %lld\\n", (long long)c, (long long)s); return 1; }
    }
    return dgs::engine_slots(INT32_MAX) == INT32_MAX ? 0 : 1;""")
