"""Rules that turn the caller's tuning parameters into launch shapes, run on the host as the library compiles them."""
import os
import subprocess

import pytest

from paper_2602_19652_gb300 import build


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    """Values of expressions over the library's headers."""
    out = tmp_path_factory.mktemp("rules")

    def run(header, exprs):
        src, exe = os.path.join(out, "r.cu"), os.path.join(out, "r")
        with open(src, "w") as f:
            f.write(f'#include <stdio.h>\n#include "{header}"\nusing namespace st;\nint main() {{\n'
                    + "".join(f'    printf("%lld\\n", (long long)({e}));\n' for e in exprs) + "    return 0;\n}\n")
        subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, "-I",
                        build.INCLUDE, src, "-o", exe], check=True)
        return [int(x) for x in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()]

    return run


def test_refill_lanes_are_the_callers(rules):
    """st_tune.refill_lanes means what it says, up to the lanes in use; 0 takes the kernel's default."""
    want = list(range(1, 33))
    got = rules("st_trace_dev.cuh", [f"trv::refill_at({n}, trv::kRefillClosest, 32, 16)" for n in want])
    assert got == want
    assert rules("st_trace_dev.cuh", [f"trv::refill_at({n}, trv::kRefillAny, 5, 1)" for n in (1, 4, 5, 6, 32)]) == [1, 4, 5, 5, 5]
    assert rules("st_trace_dev.cuh", ["trv::refill_at(0, trv::kRefillClosest, 32, 16)",
                                      "trv::refill_at(0, trv::kRefillAny, 32, 28)",
                                      "trv::refill_at(0, trv::kRefillClosest, 4, 2)",
                                      "trv::refill_at(0, trv::kRefillClosest, 1, 0)"]) == [16, 28, 2, 1]


def test_few_bin_budget_keeps_three_ctas(rules):
    """A budget set for the general accumulator's two CTAs an SM does not reach the few-bin kernel; a smaller one does."""
    assert rules("st_internal.cuh", [f"few_budget({kb})" for kb in (0, 32, 71, 72, 73, 108, 160)]) == [
        1024 * kb for kb in (72, 32, 71, 72, 72, 72, 72)]
