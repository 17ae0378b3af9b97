"""Host-side plans of the checks (csrc/hr_internal.h), compiled for the CPU: the items a shadow
clear is cut into."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


def run_cpp(tmp_path, body, args=""):
    """The output of a program over csrc/hr_internal.h, one line per line."""
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text('#include <cuda_runtime.h>\n#include <cstdio>\n#include "hr_internal.h"\nint main(){%s}\n' % body)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(CUDA, "include"),
                    "-I", os.path.join(ROOT, "paper_2401_04701_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    return [line.split() for line in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()]


@pytest.mark.parametrize("step", ["HR_RUN_CLEAR_WORDS", "HR_CLEAR_WORDS"])
def test_clear_items_stay_far_from_32_bits(tmp_path, step):
    """Every clear covers the region, and the clears of all 2^13 kernel-tag groups leave seven
    eighths of the 32-bit item numbers to the records."""
    sizes = [1, 8191, 8192, 8193, (1 << 29) - 1, 1 << 29, (1 << 29) + 1, (1 << 31) + 12345, (1 << 32) - 1, 1 << 32]
    body = "for (unsigned long long n : {%s}) printf(\"%%llu %%llu\\n\", n, hr_clear_words(n, %s));" % (
        ", ".join("%dull" % n for n in sizes), step)
    got = [tuple(map(int, g)) for g in run_cpp(tmp_path, body)]
    assert [n for n, _ in got] == sizes
    for n, words in got:
        items = -(-n // words)
        assert items * words >= n > (items - 1) * words and words % 8192 == 0
        assert items * (1 << 13) <= 1 << 29
