"""Sizes that the host derives from the device, for devices other than the one at
hand: the header's own functions, compiled into a small program (no GPU)."""
import os
import subprocess

import pytest

from paper_2502_10579_gb300 import _build


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    """Print an expression over `n` for every given n, from the library's headers."""
    d = tmp_path_factory.mktemp("limits")

    def run(expr, values):
        src, exe = os.path.join(d, "limits.cpp"), os.path.join(d, "limits")
        with open(src, "w") as f:
            f.write('#include <cstdio>\n#include "svv_ctx.h"\nusing namespace svv;\nint main() {\n'
                    "  for (long long n : {%s}) std::printf(\"%%lld\\n\", (long long)(%s));\n}\n"
                    % (", ".join(f"{v}ll" for v in values), expr))
        r = subprocess.run([_build._nvcc(), "-std=c++17", "-I", _build.CSRC, src, "-o", exe], capture_output=True, text=True)
        assert r.returncode == 0, r.stdout + r.stderr
        return [int(x) for x in subprocess.check_output([exe], text=True).split()]

    return run


def test_layout_counters_fit_the_sums_of_a_small_device(evaluate):
    """The layout builder keeps its counters in the per-CTA sums, which held 32
    words per SM: too few for 1,068 words below 34 SMs."""
    sms = [1, 2, 14, 17, 33, 34, 76, 152]
    words = evaluate("part_words((int)n)", sms)
    need = evaluate("kLayoutWords", [0])[0]
    assert need >= 1068
    for n, got in zip(sms, words):
        assert got >= need and got >= 32 * n, (n, got)


def test_grids_stay_within_what_the_barrier_counts(evaluate):
    """The error marks of 4,096 CTAs wrap the barrier's 64-bit word to no mark."""
    sms = [1, 34, 152, 1023, 1024, 1365, 5000]
    for per_sm in (1, 2, 3, 4):
        for n, got in zip(sms, evaluate(f"grid_blocks((int)n, {per_sm})", sms)):
            assert got == min(n * per_sm, 4095), (n, per_sm, got)
