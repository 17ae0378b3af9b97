"""Host-side plans of the checks (csrc/hr_internal.h, csrc/hr_per_device.h), compiled for the CPU:
the items a shadow clear is cut into, and launch state per device."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


def run_cpp(tmp_path, body):
    """The lines, split, that a program over the plans prints."""
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text('#include <cuda_runtime.h>\n#include <cstdio>\n#include <atomic>\n#include <thread>\n#include <vector>\n'
                   '#include "hr_internal.h"\n#include "hr_per_device.h"\nint main(){%s}\n' % body)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", os.path.join(CUDA, "include"),
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


def test_launch_state_is_made_once_per_device(tmp_path):
    """Eight threads ask for devices 0 to 3 and for one past the table: each device's value is its
    own and was made once; past the table it is made each time."""
    got = run_cpp(tmp_path, """
        static hr_per_device<int> values;
        static std::atomic<int> made[100];
        std::vector<std::thread> threads;
        for (int t = 0; t < 8; ++t)
            threads.emplace_back([] {
                for (int i = 0; i < 1000; ++i)
                    for (int dev : {0, 1, 2, 3, 99})
                        if (values.get(dev, [dev] { ++made[dev]; return 10 + dev; }) != 10 + dev) printf("wrong\\n");
            });
        for (auto& t : threads) t.join();
        for (int dev : {0, 1, 2, 3, 99}) printf("%d %d\\n", dev, made[dev].load());""")
    assert got == [["0", "1"], ["1", "1"], ["2", "1"], ["3", "1"], ["99", "8000"]]
