"""The autotuner's candidate schedules (host code): every one is taken by
sp_set_schedule, and the largest accepted capacity of every residency level is
tried, also where the largest capacity at that level is refused."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "sp_schedule.h"
extern "C" int candidates(int cap_max, int (*fits)(int, int), int (*blocks)(int, int), int* out) {
  int n = 0;
  for (const auto& s : sp::schedule_candidates(cap_max, fits, blocks)) {
    out[n++] = s.first;
    out[n++] = s.second;
  }
  return n / 2;
}
"""
FN = C.CFUNCTYPE(C.c_int, C.c_int, C.c_int)


@pytest.fixture(scope="module")
def candidates(tmp_path_factory):
    d = tmp_path_factory.mktemp("schedule")
    src, lib = d / "s.cpp", d / "s.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2506_23917_gb300", "csrc"), str(src), "-o", str(lib)], check=True)
    L = C.CDLL(str(lib))

    def run(fits, blocks):
        out = (C.c_int * 256)()
        n = L.candidates(1024, FN(fits), FN(blocks), out)
        return [(out[2 * i], out[2 * i + 1]) for i in range(n)]

    return run


# bytes per warp that a schedule is admitted by and those it takes, FP64 and FP32
ADMIT = {"fp64": (6928, 33), "fp32": (4240, 17)}
TAKES = {"fp64": (5504, 30), "fp32": (3200, 14)}


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_every_level_is_tried(candidates, prec):
    a, t = ADMIT[prec], TAKES[prec]
    fits = lambda cap, w: int(w * ((a[0] + a[1] * cap + 15) // 16 * 16) <= 232448)  # noqa: E731
    blocks = lambda cap, w: min(233472 // (w * (t[0] + t[1] * cap) + 1024), 64 // w)  # noqa: E731
    got = candidates(fits, blocks)
    assert len(set(got)) == len(got)
    assert all(fits(*s) for s in got)
    for w in (2, 4, 8):
        for cap in (128, 256, 384, 512, 768, 1024):
            assert ((cap, w) in got) == bool(fits(cap, w))
        ok = [cap for cap in range(128, 1025, 32) if fits(cap, w)]
        for level in {blocks(cap, w) for cap in ok}:
            assert (max(cap for cap in ok if blocks(cap, w) == level), w) in got
    if prec == "fp64":  # (672, 8) to (768, 8) have its one block per SM too, but are refused
        assert (640, 8) in got and blocks(768, 8) == blocks(640, 8) == 1
