"""The blocked NDFT's phase constants (host arithmetic done at every launch):
fractions of a turn and the bins of phase 0 against exact integers, and only the
passes in use computed, so that the launch of one does not pay for 64."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WRAP = """
#include "ndft_const.cuh"
extern "C" void consts(uint64_t a0, uint64_t da, uint64_t D, int N, int mt, uint64_t *f, int *dc) {
  const auto n = ddhf::blocked::make_ndft_const(a0, da, D, N, (N + 31) / 32, mt);
  f[0] = n.f_u; f[1] = n.f_k8; f[2] = n.f_v;
  for (int i = 0; i < 64; ++i) f[3 + i] = n.f_row[i];
  dc[0] = n.dc_first; dc[1] = n.dc_step;
}
"""


@pytest.fixture(scope="module")
def consts(tmp_path_factory):
    d = tmp_path_factory.mktemp("ndft_const")
    src, lib = str(d / "wrap.cc"), str(d / "wrap.so")
    with open(src, "w") as f:
        f.write(WRAP)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2603_08386_gb300", "csrc"), src, "-o", lib],
                   check=True)
    fn = ctypes.CDLL(lib).consts
    fn.argtypes = [ctypes.c_uint64] * 3 + [ctypes.c_int] * 2 + [ctypes.c_void_p] * 2

    def call(a0, da, D, N, mt):
        f, dc = np.zeros(67, np.uint64), np.zeros(2, np.int32)
        fn(a0, da, D, N, mt, f.ctypes.data, dc.ctypes.data)
        return [int(v) for v in f], [int(v) for v in dc]
    return call


def turn(num, den):
    return (((num % den) << 64) + den // 2) // den % (1 << 64)


def grids():
    rng = np.random.default_rng(1)
    yield from [(0, 2000, 10**9, 750), (500, 500, 10**9, 10_000), (0, 1, 1, 40), (7, 3, 1, 5),
                (1, 2, 4, 300), (6, 4, 10, 100), (5, 5, 5, 33), (0, 1, 30_000, 16_384),
                (2**31 - 1, 1, 2**31 - 1, 16_384), (4 * 10**9, 17_000, 2**31 - 1, 9_000),
                (3, 2**20, 2**20, 64), (1, 10**8, 97, 1)]
    for _ in range(300):
        N = int(rng.integers(1, 16_385))
        D = int(rng.integers(1, rng.choice([3, 100, 20_000, 2**31])))
        da = int(rng.integers(1, max(2, min(2 * D, (2**32 - 1) // (N + 31) // 2))))
        yield int(rng.integers(0, min(3 * D, 2**31) + 1)), da, D, N


@pytest.mark.parametrize("mt", [1, 2, 3, 4])
def test_constants_are_exact(consts, mt):
    for a0, da, D, N in grids():
        assert a0 + da * (N + 30) < 2**32
        f, (first, step) = consts(a0, da, D, N, mt)
        assert f[:3] == [turn(da, D), turn(17 * da, 2 * D), turn(32 * da, D)]
        for i, v in enumerate(f[3:]):
            used = 8 * mt * i < (N + 31) // 32
            num = 2 * a0 + (64 * (8 * mt * i + 4 * mt) + 31) * da
            assert v == (turn(num, 2 * D) if used else 0), (a0, da, D, N, i)
        zero = np.flatnonzero((a0 + da * np.arange(N, dtype=np.int64)) % D == 0)
        got = np.arange(first, N, step) if first >= 0 else np.empty(0, int)
        assert np.array_equal(got, zero), (a0, da, D, N)
