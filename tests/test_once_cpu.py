"""csrc/once.h on the CPU: many threads set a device up side by side, under the compiler's race detector where it is there."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_10666_b200", "csrc")
SOURCE = """
#include "once.h"
#include <cstdio>
#include <thread>
#include <vector>
static SamOncePerDevice<4> once;
static int set_up[4], failures = 2;                         // plain words: only once may touch them
int main() {
    std::atomic<int> wrong{0};
    std::vector<std::thread> all;
    for (int t = 0; t < 8; t++)
        all.emplace_back([&, t] {
            for (int i = 0; i < 2000; i++) {
                const int d = (t + i) % 4;
                const int rc = once(d, [&] { if (d == 3 && failures > 0) { failures--; return 7; } set_up[d]++; return 0; });
                if (rc != 0 && !(d == 3 && rc == 7)) wrong++;
                if (rc == 0 && set_up[d] != 1) wrong++;      // done, and seen to be done
            }
        });
    for (auto& t : all) t.join();
    if (once(-1, [] { return 0; }) != -1 || once(4, [] { return 0; }) != -1) wrong++;
    printf("%d %d %d %d %d\\n", wrong.load(), set_up[0], set_up[1], set_up[2], set_up[3]);
    return 0;
}
"""


@pytest.mark.parametrize("sanitize", [False, True])
def test_once_per_device_from_many_threads(tmp_path, sanitize):
    src, exe = str(tmp_path / "t.cpp"), str(tmp_path / "t")
    with open(src, "w") as f:
        f.write(SOURCE)
    cmd = [os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-pthread", "-I", CSRC, "-o", exe, src]
    if sanitize:
        if subprocess.run(cmd + ["-fsanitize=thread"], capture_output=True).returncode != 0:
            pytest.skip("no thread sanitizer here")
    else:
        subprocess.check_call(cmd)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    if "unexpected memory mapping" in out.stderr:
        pytest.skip("the thread sanitizer does not run under this kernel")
    assert out.returncode == 0, out.stderr[-2000:]
    assert out.stdout.split() == ["0", "1", "1", "1", "1"]


def test_the_library_keeps_no_other_word_of_its_own_between_calls():
    """Function-local statics are set by several threads at once (the calls run without Python's lock): none but what once.h guards."""
    import re
    for name in os.listdir(CSRC):
        if name.endswith((".cu", ".cuh", ".cpp", ".h")):
            for line in open(os.path.join(CSRC, name)):
                assert not re.match(r"\s+static (bool|int|int32_t|size_t|void\*)\s+\w+(\[|;| =)", line), (name, line)
