"""Host-side plans of the checks (csrc/hr_internal.h, csrc/hr_per_device.h), compiled for the CPU:
the items a shadow clear is cut into, launch state per device, and the pieces of a host trace."""
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


def test_host_pieces_are_checked_faster_than_copied(tmp_path):
    """A piece for the chosen binned checker, which goes over the whole shadow each time, is copied
    (76 ps a record) in at least the time its check takes (75 us, 18 ps a record, 2.5 or 4.5 ps a
    word), unless its group is one piece already; the others take 2^21 records."""
    sizes = [(n, w, b) for n in (1, 1 << 20, 5_000_000, (1 << 23) + 7, 9_404_416, (1 << 24) - 1, 1 << 24)
             for w in (1, 1 << 20, 1 << 22, 1 << 24, 33_554_431, 1 << 26) for b in (4, 8)]
    body = "".join("printf(\"%%llu %%llu\\n\", hr_host_piece(%dull, true, %dull, %d), hr_host_piece(%dull, false, %dull, %d));"
                   % (x + x) for x in sizes)
    for (n, words, shadow_bytes), (binned, other) in zip(sizes, run_cpp(tmp_path, body)):
        piece, parts = int(binned), -(-n // int(binned))
        check = 75e6 + 18 * piece + (4.5 if shadow_bytes == 4 else 2.5) * words
        assert parts == 1 or (piece >= 1 << 21 and check < 76 * piece and n - (parts - 1) * piece > piece // 2)
        assert int(other) == 1 << 21
