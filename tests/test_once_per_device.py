"""Kernel attributes are set once for each kernel on each device (csrc/zf_once.h),
checked on the host with counted calls in the place of CUDA's."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_08190_gb300", "csrc")

HARNESS = r"""
#include "zf_once.h"
#include <cstdio>

int main() {
    zf::OncePerDevice once;
    int kernel_a = 0, kernel_b = 0, calls = 0, result = 0;
    auto set = [&] { calls++; return result; };
    auto expect = [&](int device, const void* kernel, int want_calls, int want) {
        const int got = once(device, kernel, set);
        if (calls != want_calls || got != want) {
            printf("device %d: %d calls, result %d\n", device, calls, got);
            return false;
        }
        return true;
    };
    bool ok = expect(0, &kernel_a, 1, 0) && expect(0, &kernel_a, 1, 0);   // once
    ok = ok && expect(1, &kernel_a, 2, 0) && expect(1, &kernel_a, 2, 0);  // on a second device too
    ok = ok && expect(0, &kernel_b, 3, 0) && expect(0, &kernel_a, 3, 0);  // and for a second kernel
    result = 7;                                                           // a failure is reported and tried again
    ok = ok && expect(2, &kernel_a, 4, 7);
    result = 0;
    ok = ok && expect(2, &kernel_a, 5, 0) && expect(2, &kernel_a, 5, 0);
    return ok ? 0 : 1;
}
"""


def test_each_device_and_kernel_once(tmp_path):
    (tmp_path / "h.cpp").write_text(HARNESS)
    exe = str(tmp_path / "h")
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, "-o", exe, str(tmp_path / "h.cpp")], check=True)
    subprocess.run([exe], check=True)


def test_every_launcher_uses_it():
    for f in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, f)).read() if f.endswith(".cu") else ""
        if "cudaFuncAttributeMaxDynamicSharedMemorySize" in text and f != "zf_mlp.cu":   # set by each network for its device
            assert "zf::OncePerDevice" in text, f
