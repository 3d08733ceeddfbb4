"""Launch state that belongs to a device: set up at each device's first use, a
failure returned and not kept (host arithmetic, on a stand-in for the runtime's
two calls)."""
import os
import shutil
import subprocess

import pytest
import torch

from paper_2605_30574_gb300 import build as B
from paper_2605_30574_gb300 import decoder as K

SOURCE = r"""
#include "per_device.h"
#include <cstdio>
#include <thread>
#include <vector>
static thread_local int device = 0;
static int cleared = 0;
static cudaError_t query = cudaSuccess;
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return query; }
extern "C" cudaError_t cudaGetLastError() { ++cleared; return cudaSuccess; }
struct State { int dev, n; };
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
    static splice::PerDevice<State> kept;
    std::atomic<int> made{0};
    bool fails = true;
    auto make = [&](int d, State* s) {
        *s = {d, 100 + d};
        ++made;
        return fails ? cudaErrorInvalidValue : cudaSuccess;
    };
    State s{};
    CHECK(kept.get(&s, make) == cudaErrorInvalidValue && made == 1 && cleared == 1);
    fails = false;
    CHECK(kept.get(&s, make) == cudaSuccess && made == 2 && s.n == 100);
    CHECK(kept.get(&s, make) == cudaSuccess && made == 2 && s.n == 100);
    device = 3;
    CHECK(kept.get(&s, make) == cudaSuccess && made == 3 && s.dev == 3 && s.n == 103);
    device = 0;
    CHECK(kept.get(&s, make) == cudaSuccess && made == 3 && s.n == 100);
    for (int i = 0; i < 2; ++i) {
        device = 1000;
        CHECK(kept.get(&s, make) == cudaSuccess && made == 4 + i && s.n == 1100);
    }
    query = cudaErrorNoDevice;
    CHECK(kept.get(&s, make) == cudaErrorNoDevice && made == 5 && cleared == 2);
    query = cudaSuccess;
    std::vector<std::thread> ts;
    std::atomic<int> wrong{0};
    for (int t = 0; t < 8; ++t)
        ts.emplace_back([&, t] {
            for (int i = 0; i < 2000; ++i) {
                device = (i + t) % 64;
                State x{};
                if (kept.get(&x, make) != cudaSuccess || x.n != 100 + device) ++wrong;
            }
        });
    for (auto& t : ts) t.join();
    CHECK(wrong == 0);
    const int before = made;
    for (device = 0; device < 64; ++device) CHECK(kept.get(&s, make) == cudaSuccess && s.dev == device);
    CHECK(made == before);
    return 0;
}
"""


def test_state_per_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = tmp_path / "t.cpp"
    src.write_text(SOURCE)
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    subprocess.run([cxx, "-std=c++17", "-pthread", "-I", os.path.join(B.PKG, "csrc"), "-I", include, str(src), "-o",
                    str(tmp_path / "t")], check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.skipif(torch.cuda.is_available(), reason="asks for launches where there is no device")
def test_without_a_device_the_runtimes_error_comes_back():
    B.build()
    p = 1 << 20
    for _ in range(2):
        for mode in (0, 1, 2):
            assert K.lib().decoder_gemm(mode, p, p, p, None, p, 8, 64, 64, None) > 1
        assert K.lib().decoder_causal(p, p, p, p, 8, 1, 1, 64, 0.125, None) > 1
