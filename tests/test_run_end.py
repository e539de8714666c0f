"""The search for the end of a resident run (csrc/dm_run_end.h, compiled for
the host): exact on leading runs from any guess, and on residencies that are no
leading run (lookups that gave up) every probed block lies inside the prompt,
the rounds stay few, and the answer is a block found missing or the prompt's
end."""

import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_06502_gb300", "csrc")

SRC = r"""
#include "dm_run_end.h"
// The run's end; *rounds (stops at 1000), *top: the largest block probed.
extern "C" uint32_t run_end(uint32_t nblk, uint32_t guess, const uint8_t *resident, uint32_t *rounds, uint32_t *top) {
    dm::RunEnd e(nblk, guess);
    *rounds = *top = 0;
    while (e.open() && *rounds < 1000) {
        bool in[3];
        for (int q = 0; q < 3; ++q) {
            if (e.b[q] > *top) *top = e.b[q];
            in[q] = e.b[q] < nblk && resident[e.b[q]];
        }
        ++*rounds;
        e.narrow(in);
    }
    return e.hi;
}
"""


@pytest.fixture(scope="module")
def run_end(tmp_path_factory):
    d = tmp_path_factory.mktemp("run_end")
    (d / "run_end.cpp").write_text(SRC)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-Wall", "-Wextra", "-I", CSRC,
                           str(d / "run_end.cpp"), "-o", str(d / "run_end.so")])
    f = C.CDLL(str(d / "run_end.so")).run_end
    f.restype = C.c_uint32
    f.argtypes = [C.c_uint32, C.c_uint32, C.c_void_p, C.POINTER(C.c_uint32), C.POINTER(C.c_uint32)]

    def call(resident, guess):
        rounds, top = C.c_uint32(), C.c_uint32()
        r = f(len(resident), guess, resident.ctypes.data, C.byref(rounds), C.byref(top))
        return r, rounds.value, top.value
    return call


def test_leading_runs(run_end):
    for nblk in list(range(1, 70)) + [127, 128, 129, 500]:
        for run in range(1, nblk + 1):
            resident = (np.arange(nblk) < run).astype(np.uint8)
            for guess in {0, 1, run - 1, run, min(run + 1, nblk), nblk // 3, nblk}:
                end, rounds, top = run_end(resident, guess)
                assert end == run and top < nblk and rounds <= 2 + nblk.bit_length(), (nblk, run, guess)


def test_residencies_that_are_no_leading_run(run_end):
    # the lower probe missing and the higher one resident: nblk / 4 and nblk / 2 from no guess
    resident = np.ones(40, np.uint8)
    resident[8:16] = 0
    assert run_end(resident, 0) == (10, 1, 20)
    rng = np.random.default_rng(1)
    for _ in range(20_000):
        nblk = int(rng.integers(1, 200))
        resident = (rng.random(nblk) < rng.random()).astype(np.uint8)
        resident[0] = 1
        end, rounds, top = run_end(resident, int(rng.integers(0, nblk + 1)))
        assert top < nblk and rounds <= 2 + nblk.bit_length()
        assert end <= nblk and (end == nblk or not resident[end])
