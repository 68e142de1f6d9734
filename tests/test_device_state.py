"""What the host side keeps about devices (csrc/goq_device.h), against a fake of the CUDA runtime calls that it makes: no GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_26092_b200", "csrc")

FAKE = r"""
#include "goq_device.h"
#include <chrono>
#include <cstdio>
#include <map>
#include <thread>
#include <vector>
thread_local int device = 0;
static std::atomic<int> arrived{0};
static void pause_ms(int ms) { std::this_thread::sleep_for(std::chrono::milliseconds(ms)); }
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return device < 0 ? cudaErrorNoDevice : cudaSuccess; }
"""


def _run(tmp_path, body):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(FAKE + body)
    cuda = "/usr/local/cuda/include"
    if not os.path.isdir(cuda):
        pytest.skip("no CUDA headers")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", cuda, "-I", CSRC, str(src), "-o", str(exe), "-pthread"], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stdout + out.stderr


def test_sm_count_is_each_devices_own_for_threads_that_ask_first_together(tmp_path):
    """Sixteen threads on two devices of 148 and 100 SMs, all inside the first question at once: everybody gets its device's number, then and later; a device
    beyond the table is asked each time, and one that cannot be asked counts as 148."""
    _run(tmp_path, r"""
static std::atomic<int> asked{0};
extern "C" cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int dev) {
    ++asked; ++arrived;
    for (int i = 0; i < 500 && arrived < 16; ++i) pause_ms(1);   // all of them are here before the first returns
    *v = dev == 0 ? 148 : dev == 1 ? 100 : 64;
    return cudaSuccess;
}
int main() {
    std::atomic<int> wrong{0};
    std::vector<std::thread> t;
    for (int i = 0; i < 16; ++i)
        t.emplace_back([&, i] { device = i & 1; for (int k = 0; k < 100; ++k) wrong += goq::sm_count() != (device ? 100 : 148); });
    for (auto& x : t) x.join();
    const int first = asked;
    device = 200; wrong += goq::sm_count() != 64; wrong += goq::sm_count() != 64;
    device = -1; wrong += goq::sm_count() != 148;
    std::printf("wrong %d asked %d\n", wrong.load(), first);
    return wrong != 0 || first > 16 || asked != first + 2;
}
""")


def test_shared_memory_limit_never_falls_below_what_is_noted(tmp_path):
    """A call of 200000 bytes is held up between setting the limit and noting it; one of 100000 on another thread sets it meanwhile, if it is let. Whatever is
    noted as set then is: a later call of 200000 finds the limit there or sets it again. Per device."""
    _run(tmp_path, r"""
static std::atomic<int> limit[2];
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int v) {
    if (v == 200000) { limit[device] = v; pause_ms(100); }
    else { pause_ms(30); limit[device] = v; }
    return cudaSuccess;
}
static void kernel() {}
int main() {
    goq::SmemAttrCache cache;
    std::vector<std::thread> t;
    for (int i = 0; i < 4; ++i) t.emplace_back([&, i] { device = i >> 1; goq::ensure_dynamic_smem(kernel, (i & 1) ? 100000 : 200000, cache); });
    for (auto& x : t) x.join();
    int wrong = 0;
    for (device = 0; device < 2; ++device) {
        goq::ensure_dynamic_smem(kernel, 200000, cache);
        wrong += limit[device] != 200000;
        goq::ensure_dynamic_smem(kernel, 100000, cache);
        wrong += limit[device] != 200000;
    }
    std::printf("limits %d %d\n", limit[0].load(), limit[1].load());
    return wrong;
}
""")


def test_one_place_asks_for_the_number_of_sms():
    """Every launcher plans with goq_device.h's count: no copy with a cache of its own (one was halved in place by whoever came first, some kept the first
    device's number for all)."""
    users = [f for f in sorted(os.listdir(CSRC)) if "cudaDevAttrMultiProcessorCount" in open(os.path.join(CSRC, f)).read()]
    assert users == ["goq_device.h"]
