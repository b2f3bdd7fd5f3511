"""What the library does once per device (csrc/per_device.cuh), compiled with a
fake of the CUDA calls: each device is asked on its own, from several threads,
and a failure is not taken for done."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2012_11744_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

PROG = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.cuh"
static thread_local int device = 0;
static thread_local bool broken = false;
static std::atomic<int> asked[80];
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaGetLastError(void) { return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) {
    if (broken) return cudaErrorInvalidValue;
    asked[device]++;
    return cudaSuccess;
}
int main() {
    paris::SmemOptIn o{};
    paris::DeviceValue v{};
    int bad = 0;
    device = 1;
    broken = true;
    bad += paris::allow_smem(o, nullptr, 100) == cudaSuccess;
    bad += paris::device_value(v, [](int) { return 0; }) != 1;
    broken = false;
    std::vector<std::thread> t;
    std::atomic<int> wrong{0};
    for (int q = 0; q < 16; ++q)
        t.emplace_back([&] {
            for (int rep = 0; rep < 1000; ++rep)
                for (int d : {0, 1, 63, 70}) {
                    device = d;
                    wrong += paris::allow_smem(o, nullptr, 100) != cudaSuccess;
                    wrong += paris::device_value(v, [](int dev) { return 100 + dev; }) != 100 + d;
                }
        });
    for (auto& x : t) x.join();
    for (int d : {0, 1, 63}) bad += asked[d] < 1 || asked[d] > 16;  // once, or once a thread that met it first
    bad += asked[70] != 16000;                                     // not kept: asked each time
    printf("%d %d\n", bad, wrong.load());
    return bad + wrong.load();
}
"""


def test_asked_once_on_every_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROG)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-I", os.path.join(CUDA, "include"),
                           str(src), "-o", str(exe)])
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout.split() == ["0", "0"]


def test_function_attributes_only_through_it():
    for name in sorted(os.listdir(CSRC)):
        if name == "per_device.cuh" or not name.endswith((".cu", ".cuh")):
            continue
        src = re.sub(r"//.*", "", open(os.path.join(CSRC, name)).read())
        assert "cudaFuncSetAttribute" not in src, name
