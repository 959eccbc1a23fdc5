"""Planning of the sweep's bins (kimad_common.h) compiled for the host: it ends, with finite needs and as many bins as fit,
whatever the estimates it starts from."""
import ctypes
import math
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = r'''
#include "kimad_common.h"
extern "C" float need_of(float dens, float load, float error) { return kimad::bins_needed(dens, load, error); }
extern "C" int coarsen(const uint32_t* bot, const uint32_t* top, uint32_t* shift, const float* need, uint32_t n, uint32_t most, uint32_t* left) {
    uint32_t fine = 0;
    for (uint32_t g = 0; g < n; ++g) fine += (top[g] - bot[g] + 1) << (kimad::kCellShift - shift[g]);
    return kimad::coarsen_groups(kimad::OneLane{}, bot, top, shift, need, n, fine, most, left);
}
extern "C" uint32_t cluster_of(uint64_t most, uint64_t layers, const uint32_t* resident) { return kimad::sample_cluster(most, layers, resident); }
'''


@pytest.fixture(scope="module")
def planner(tmp_path_factory):
    d = tmp_path_factory.mktemp("planner")
    (d / "planner.cpp").write_text(CODE)
    so = str(d / "planner.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2312_08053_b200", "csrc"), "-o", so, str(d / "planner.cpp")], check=True)
    lib = ctypes.CDLL(so)
    lib.need_of.restype = ctypes.c_float
    lib.need_of.argtypes = [ctypes.c_float] * 3
    return lib


def test_needs_are_finite(planner):
    values = [0.0, 1e-45, 1e-38, 1e-20, 1.0, 2048.0, 1e20, 3e38, math.inf, math.nan]
    for dens in values:
        for load in values:
            for error in values:
                x = planner.need_of(dens, load, error)
                assert 0.0 <= x <= 1024.0, (dens, load, error, x)
    assert planner.need_of(4096.0, 0.0, 1.0) == 2.0


def test_coarsening_ends(planner):
    rng = random.Random(1)
    odd = [math.inf, math.nan, 0.0, 1e-30, 1024.0, 3e38]
    for _ in range(500):
        n = rng.randint(1, 128)
        cells = [int(math.exp(rng.uniform(0, math.log(12288 / n)))) for _ in range(n)]
        bot, top, at = [], [], 70000
        for c in cells:
            at -= c + rng.randint(0, 3)
            bot.append(at)
            top.append(at + c - 1)
        shift = [rng.randint(5, 15) for _ in range(n)]
        strange = 0.5 * rng.randint(0, 1)
        need = [rng.choice(odd) if rng.random() < strange else math.exp(rng.uniform(-10, 10)) for _ in range(n)]
        most = rng.choice([12288, sum(cells), max(1, sum(cells) // 2)])
        u32, f32 = ctypes.c_uint32 * n, ctypes.c_float * n
        s, left = u32(*shift), ctypes.c_uint32(0)
        ok = planner.coarsen(u32(*bot), u32(*top), s, f32(*need), ctypes.c_uint32(n), ctypes.c_uint32(most), ctypes.byref(left))
        fine = sum(c << (15 - x) for c, x in zip(cells, s))
        assert all(a <= b <= 15 for a, b in zip(shift, s))
        if ok:
            assert fine + left.value == most
        else:
            assert all(x == 15 for x in s) and fine > most
        if all(1e-6 < v < 1e6 for v in need):  # one step at a time comes to the same
            one = list(shift)
            while sum(c << (15 - x) for c, x in zip(cells, one)) > most and min(one) < 15:
                g = min((v * 2 ** x, g) for g, (v, x) in enumerate(zip(f32(*need), one)) if x < 15)[1]
                one[g] += 1
            assert one == list(s)


@pytest.mark.parametrize("resident", [(148, 74, 33, 15), (148, 74, 32, 12), (100, 44, 20, 0), (1, 0, 0, 0)])
def test_clusters_are_resident_and_have_work(planner, resident):
    """A layer's sample is read by a cluster only where all clusters run at once and none of their CTAs is without units."""
    r = (ctypes.c_uint32 * 4)(*resident)
    seen = set()
    for most in (4097, 5000, 8192, 16384, 16385, 24577, 32768, 40000, 65536, 70000, 98304, 110000, 131072, 10 ** 6, 2 ** 32 - 1):
        units = -(-most // 32)
        units = units if units <= 1024 else min(max(units // 2, 1024), 2047)
        for layers in (1, 2, 12, 13, 15, 16, 20, 21, 32, 33, 34, 44, 64, 65, 74, 75, 128, 149, 2000):
            n = planner.cluster_of(ctypes.c_uint64(most), ctypes.c_uint64(layers), r)
            seen.add(n)
            assert n in (1, 2, 4, 8)
            if n > 1:
                assert layers <= resident[n.bit_length() - 1]
                assert n * 256 < units + 2 * 256  # at most one CTA of a cluster idles
    assert seen == {1 << i for i in range(4) if resident[i]}
