"""Launch state and launch arithmetic of the library (csrc/dm_launch.h,
compiled for the host, devices and settings made up)."""

import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_06502_gb300", "csrc")

SRC = r"""
#include "dm_launch.h"

#include <chrono>
#include <thread>
#include <vector>

static std::atomic<size_t> allowed[dm::kDevices];   // the made-up setting per device
static std::atomic<int> calls;

static int set_to(int dev, size_t bytes) {
    ++calls;
    std::this_thread::sleep_for(std::chrono::microseconds(200));
    allowed[dev] = bytes;
    return 0;
}

// Launches on two devices, one after the other: 0 if both were allowed the size.
extern "C" int two_devices() {
    dm::SmemOptIn opt;
    for (int dev : {0, 1, 0}) {
        if (opt.raise(dev, 60000, [&] { return set_to(dev, 60000); })) return 1;
        if (allowed[dev] < 60000) return 2;
    }
    return calls == 2 ? 0 : 3;
}

// Threads whose launches need different sizes: the number of launches that
// found less allowed than they need.
extern "C" int racing_sizes() {
    std::atomic<int> refused{0};
    for (int round = 0; round < 20; ++round) {
        dm::SmemOptIn opt;
        allowed[2] = 0;
        std::vector<std::thread> ts;
        for (int t = 0; t < 8; ++t)
            ts.emplace_back([&, t] {
                const size_t need = 50000 + 10000 * ((t * 5) % 8);
                for (int k = 0; k < 3; ++k) {
                    opt.raise(2, need, [&] { return set_to(2, need); });
                    std::this_thread::sleep_for(std::chrono::microseconds(300));
                    if (allowed[2] < need) ++refused;   // the launch
                }
            });
        for (auto &t : ts) t.join();
    }
    return refused;
}

// A setting that fails is reported and asked for again.
extern "C" int failure_is_not_kept() {
    dm::SmemOptIn opt;
    if (opt.raise(3, 60000, [] { return 700; }) != 700) return 1;
    return opt.raise(3, 60000, [] { return set_to(3, 60000); }) || allowed[3] != 60000 ? 2 : 0;
}

extern "C" void potc_shape(uint32_t trials, uint32_t sms, uint32_t *per_cta, uint32_t *grid) {
    const dm::PotcShape s = dm::potc_shape(trials, sms);
    *per_cta = s.per_cta;
    *grid = s.grid;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("launch")
    (d / "launch.cpp").write_text(SRC)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-pthread", "-Wall", "-Wextra", "-I", CSRC,
                           str(d / "launch.cpp"), "-o", str(d / "launch.so")])
    return C.CDLL(str(d / "launch.so"))


@pytest.mark.parametrize("check", ["two_devices", "racing_sizes", "failure_is_not_kept"])
def test_shared_memory_opt_in(lib, check):
    assert getattr(lib, check)() == 0


@pytest.mark.parametrize("trials", [1, 31, 32, 33, 152, 4864, 4865, 10_000, 1 << 31, (1 << 32) - 4864,
                                    (1 << 32) - 4863, (1 << 32) - 1])
@pytest.mark.parametrize("sms", [1, 148, 152])
def test_sweep_shape_covers_every_trial(lib, trials, sms):
    T, grid = C.c_uint32(), C.c_uint32()
    lib.potc_shape(trials, sms, C.byref(T), C.byref(grid))
    assert 1 <= T.value <= 32 and (grid.value - 1) * T.value < trials <= grid.value * T.value
    assert grid.value < 1 << 31 or sms == 1
