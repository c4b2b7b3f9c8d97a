"""The rule on the device memory that window records may take."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GB = 1 << 30


@pytest.fixture(scope="module")
def allowed(tmp_path_factory):
    d = tmp_path_factory.mktemp("budget")
    (d / "t.cpp").write_text('#include "tsp_records_budget.h"\n#include <cstdio>\n#include <cstdlib>\n'
                             "int main(int, char** a) { std::printf(\"%d\", records_allowed("
                             "std::strtoull(a[1], 0, 10), std::strtoull(a[2], 0, 10), "
                             "std::strtoull(a[3], 0, 10))); }\n")
    exe = str(d / "t")
    subprocess.run(["g++", "-std=c++17", "-I",
                    os.path.join(ROOT, "paper_1502_07478_gb300", "csrc"), str(d / "t.cpp"), "-o",
                    exe], check=True)
    return lambda *a: subprocess.run([exe, *map(str, a)], capture_output=True,
                                     text=True).stdout == "1"


def test_one_context_takes_a_quarter(allowed):
    assert allowed(70 * GB, 0, 280 * GB)
    assert not allowed(70 * GB + 1, 0, 280 * GB)
    assert allowed(0, 0, 0) and not allowed(1, 0, 0)


def test_a_batch_takes_a_quarter_together(allowed):
    """Members one after another, each as large as it may be: the rest of the memory
    stays free for event buffers."""
    free, held, step = 280 * GB, 0, GB
    while allowed(step, held, free - held):
        held += step
    assert held == 70 * GB
