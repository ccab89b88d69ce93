"""The parts of the CUDA path's headers that compile for the host too, built with
g++ and checked without a GPU."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2109_01329_gb300", "csrc")
INCLUDE = os.path.join(ROOT, "include")


def _build(path, code, *flags):
    """Compiles C++ source text against the headers; the path of what it makes."""
    src, out = str(path / "t.cpp"), str(path / "t.bin")
    with open(src, "w") as f:
        f.write(code)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, "-I", INCLUDE, src, "-o", out, *flags],
                   check=True, timeout=300)
    return out


def test_jump_table_is_aligned_for_16_byte_loads(tmp_path):
    """The kernels read the table of jump matrices in 16-byte pieces: the type, not
    the order in which a linker lays globals, has to place every row and second
    matrix on such a boundary."""
    exe = _build(tmp_path, """
#include <cstdio>
#include "mrg_tables.h"
int main() { std::printf("%zu %zu", alignof(grng::mrg::DigitTable), sizeof(grng::mrg::DigitTable::row[0])); }
""")
    align, row = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert align % 16 == 0 and row % 16 == 0


def test_batch_launch_count_heals_after_overlaps(tmp_path):
    """CTAs of up to three launches of one batch arriving in any order: a launch
    that runs alone shows one count to all of its CTAs, and once launches that
    overlapped are over the count is their number, exactly."""
    exe = _build(tmp_path, """
#include <algorithm>
#include <cstdio>
#include <random>
#include <vector>
#include "grng_internal.h"
using namespace grng;
int main() {
  std::mt19937 r(7);
  uint64_t arrivals = 0, launches = 0;
  const uint32_t grids[] = {1, 2, 3, 152, 4864, 1u << kArrivalBits};
  for (int trial = 0; trial < 300; ++trial) {
    std::vector<uint64_t> shares;  // what the CTAs of this trial's launches add
    const int k = trial % 3 + 1;
    for (int i = 0; i < k; ++i) {
      const uint32_t ctas = grids[r() % (trial < 6 ? 6 : 5)];
      for (uint32_t c = 0; c < ctas; ++c) shares.push_back(batch_arrival(c, ctas));
    }
    std::shuffle(shares.begin(), shares.end(), r);
    for (uint64_t s : shares) {
      if (k == 1 && arrivals >> kArrivalBits != launches) return std::puts("a CTA saw another count"), 1;
      arrivals += s;
    }
    launches += k;
    if (arrivals != launches << kArrivalBits) return std::puts("the count is off"), 1;
  }
}
""")
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


@pytest.fixture(scope="module")
def bm64(tmp_path_factory):
    """neg2_log and the square root after it, of the FP64 fixed-point transforms."""
    lib = ctypes.CDLL(_build(tmp_path_factory.mktemp("bm64"), """
#include "bm64_fixed.cuh"
using namespace grng::bm64;
// words of pairs -> |z0|, |z1| = p 2^k
extern "C" void pairs(int n, const uint32_t* w, uint64_t* p, int* k) {
  for (int i = 0; i < n; ++i) {
    const FixedPair f = box_muller_fixed(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
    p[2 * i] = f.p0;
    p[2 * i + 1] = f.p1;
    k[i] = f.k;
  }
}
// for u1 = m 2^-53: -2 ln u1 = X 2^E and its root s 2^k
extern "C" void rho(int n, const uint64_t* m, uint64_t* X, int* E, uint64_t* s, int* k) {
  for (int i = 0; i < n; ++i) {
    neg2_log((uint32_t)(m[i] >> 21), (uint32_t)(m[i] << 11), X[i], E[i]);
    sqrt_fixed(X[i], E[i], s[i], k[i]);
  }
}
""", "-shared", "-fPIC"))

    def pairs(w):
        p, k = np.empty(w.size // 2, np.uint64), np.empty(w.size // 4, np.int32)
        lib.pairs(w.size // 4, *(a.ctypes.data_as(ctypes.c_void_p) for a in (w, p, k)))
        return p.reshape(-1, 2), k

    def rho(m):
        m = np.ascontiguousarray(m, dtype=np.uint64)
        X, s = np.empty_like(m), np.empty_like(m)
        E, k = np.empty(m.size, np.int32), np.empty(m.size, np.int32)
        lib.rho(m.size, *(a.ctypes.data_as(ctypes.c_void_p) for a in (m, X, E, s, k)))
        return X, E, s, k

    rho.pairs = pairs
    return rho


def test_fp64_logarithm_keeps_64_bit_units(bm64):
    """-ln u1 for u1 in [1/2, 1) in units of 2^-64, and below 1/2 within 58 of them and
    what the result holds: the sum's terms truncate by at most that (r^3/3: 5 units
    of 2^-59 times 32/3; the others 5 more), and e ln 2 adds nothing of its size."""
    mp = pytest.importorskip("mpmath")
    mp.mp.prec = 160
    r = np.random.Generator(np.random.PCG64(64))
    top = 1 << 53
    band = r.integers(top - (top >> 9), top - (top >> 10), 2000)  # u1 in (1 - 2^-9, 1 - 2^-10)
    X, E, _, _ = bm64(band)
    # 2 L in units of 2^-63: odd half of the time
    odd = [(int(x) << (int(e) + 63) if e >= -63 else int(x) >> (-63 - int(e))) & 1 for x, e in zip(X, E)]
    assert 800 < sum(odd) < 1200
    worst = 0
    for e in range(1, 21):
        m = r.integers(top >> (e + 1), top >> e, 500)
        X, E, _, _ = bm64(m)
        for mi, x, ex in zip(m.tolist(), X.tolist(), E.tolist()):
            worst = max(worst, abs(mp.ldexp(x, ex - 1) + mp.log(mp.ldexp(mi, -53))))
    # X holds -2 ln u1 < 32 to 2^-58, -ln u1 to half of that
    assert worst < mp.ldexp(58, -64) + mp.ldexp(1, -59)


@pytest.mark.parametrize("k", [-3, -2, -1, 0, 1, 2])
def test_fp64_root_where_its_reciprocal_rounds_to_two(bm64, k):
    """rho = sqrt(-2 ln u1) on both sides of -2 ln u1 = 4^k, where x in [1/4, 1) is
    just above 1/4 and just below 1: within 2^-51, as stated (relative, or absolute
    below 1)."""
    mp = pytest.importorskip("mpmath")
    mp.mp.prec = 160
    m0 = int(mp.floor(mp.ldexp(mp.exp(-mp.ldexp(1, 2 * k) / 2), 53)))
    m = np.arange(max(1, m0 - 1500), m0 + 1500)
    _, _, s, e = bm64(m)
    rho = [mp.sqrt(-2 * mp.log(mp.ldexp(v, -53))) for v in m.tolist()]
    worst = max(abs(mp.ldexp(int(a), int(b)) - r) / max(1, r) for a, b, r in zip(s, e, rho))
    assert worst < mp.ldexp(1, -51)


def test_fp64_pairs_before_rounding_are_near_the_middle(bm64):
    """The fixed-point pair ahead of its rounding to even: low by less than 2 of its
    units on average (a result of rho's own size has 2^8 or more in its last place)."""
    mp = pytest.importorskip("mpmath")
    mp.mp.prec = 130
    w = np.random.Generator(np.random.PCG64(65)).integers(0, 1 << 32, 4 * 4000, dtype=np.uint32)
    p, k = bm64.pairs(w)
    total = mp.mpf(0)
    for (a, b, c, d), q, e in zip(w.reshape(-1, 4).tolist(), p.tolist(), k.tolist()):
        rho = mp.sqrt(-2 * mp.log(mp.ldexp((((a << 32) | b) >> 11) + 1, -53)))
        turn = mp.ldexp(((c << 32) | d) >> 11, -52)
        total += q[0] - mp.ldexp(rho * abs(mp.cospi(turn)), -e) + q[1] - mp.ldexp(rho * abs(mp.sinpi(turn)), -e)
    assert -2 < total / (2 * k.size) < 2


def test_fp64_inverse_cdf_before_rounding_is_near_the_middle(tmp_path):
    """t = -Phi^-1(p) in its units of 2^-59: off by less than 3 on average (the fits
    stay below 6 of them)."""
    mp = pytest.importorskip("mpmath")
    mp.mp.prec = 130
    lib = ctypes.CDLL(_build(tmp_path, """
#include "icdf64_fixed.cuh"
extern "C" uint64_t t59(uint64_t m) { return grng::icdf64::neg_icdf(m); }
""", "-shared", "-fPIC"))
    lib.t59.argtypes, lib.t59.restype = [ctypes.c_uint64], ctypes.c_uint64
    total, n = mp.mpf(0), 600
    for m in np.random.Generator(np.random.PCG64(66)).integers(1, 1 << 51, n).tolist():
        m = 2 * m + 1
        t = mp.ldexp(lib.t59(m), -59)
        # one Newton step from t, which is right to 2^-50: then to 2^-99
        density = mp.exp(-t * t / 2) / mp.sqrt(2 * mp.pi)
        total += mp.ldexp((mp.ldexp(m, -53) - mp.erfc(t / mp.sqrt(2)) / 2) / density, 59)
    assert -3 < total / n < 3
