"""What is set once per device (kernel attributes) is set on each device of a process: the helper is plain
host code, compiled and driven here with counted calls. Every kernel that asks for more shared memory than
the default goes through it."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1612_02120_gb300", "csrc")

PROGRAM = """
#include <cstdio>
#include "per_device.h"
int main() {
    static std::atomic<uint64_t> done{0};
    int calls = 0;
    auto once = [&](int device, mb_status result) {
        return mb::once_per_device(done, device, [&] { ++calls; return result; });
    };
    bool ok = once(0, MB_OK) == MB_OK && once(0, MB_OK) == MB_OK && calls == 1;
    ok = ok && once(1, MB_ERR_CUDA) == MB_ERR_CUDA && calls == 2;          // a failure is not remembered
    ok = ok && once(1, MB_OK) == MB_OK && once(1, MB_OK) == MB_OK && calls == 3;
    ok = ok && once(63, MB_OK) == MB_OK && once(63, MB_OK) == MB_OK && calls == 4;
    ok = ok && once(64, MB_OK) == MB_OK && once(64, MB_OK) == MB_OK && calls == 6;  // no bit for it
    ok = ok && once(0, MB_OK) == MB_OK && calls == 6;
    std::puts(ok ? "ok" : "wrong");
    return ok ? 0 : 1;
}
"""


def test_set_once_on_each_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout == "ok\n"


def test_shared_memory_attributes_go_through_the_helper():
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        assert ("cudaFuncSetAttribute(" in text) == (name == "internal.h"), name
    assert "once_per_device" in open(os.path.join(CSRC, "internal.h")).read()
