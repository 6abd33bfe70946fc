"""What a launcher sets once is set once on every device: the helper that keeps it, compiled for the host against a CUDA runtime whose
current device the test chooses, and no launcher that keeps such a thing for the whole process."""
import glob
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1701_06538_b200", "csrc")

HOST = r"""
#include "per_device.h"
#include <stdio.h>
static int device = 0, raised[70];
static bool broken = false;
extern "C" cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int bytes) {
    if (broken || bytes != 100000) return cudaErrorInvalidValue;
    ++raised[device];
    return cudaSuccess;
}
static void kernel(int) {}
int main() {
    static moe::PerDevice done, value;
    const int order[] = {0, 0, 1, 0, 1, 63, 63, 64, 64};
    for (int d : order) {
        device = d;
        if (!moe::allow_shared(done, kernel, 100000)) return 1;
    }
    printf("%d %d %d %d %d\n", raised[0], raised[1], raised[2], raised[63], raised[64]);
    device = 2;
    broken = true;
    if (moe::allow_shared(done, kernel, 100000)) return 2;   // reported, and tried again
    broken = false;
    if (!moe::allow_shared(done, kernel, 100000)) return 3;
    for (int d = 0; d < 3; ++d) { device = d; value.get([&]() { return 10 + d; }); }
    for (int d = 0; d < 3; ++d) { device = d; printf("%d ", value.get([&]() { return -1; })); }
    return 0;
}
"""


def test_every_device_is_set_up_once(tmp_path):
    src, exe = tmp_path / "host.cpp", tmp_path / "host"
    src.write_text(HOST)
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, "-I", "/usr/local/cuda/include", str(src), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0
    assert out.stdout.split() == ["1", "1", "0", "1", "2", "10", "11", "12"]  # beyond the table: on every launch


def test_no_launcher_keeps_device_state_for_the_process():
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        text = open(path).read()
        assert not re.search(r"static (bool|int) \w+ = (false|0);\s*\n\s*(if|cudaLaunchConfig_t)", text), path
        for call in ("cudaFuncSetAttribute", "cudaOccupancyMaxActiveClusters"):
            for at in (m.start() for m in re.finditer(call, text)):
                assert ".get([&]()" in text[max(0, at - 500):at], f"{path}: {call}"
