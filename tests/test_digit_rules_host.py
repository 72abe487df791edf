"""Host checks of the digits behind the FP64 products from BF16 digits: the rules
that the library runs (csrc/digit_rules.h, compiled here) and a restatement of the
splitting in exact integers (base 512; csrc/sliced.cu, put_all_digits).

* the remainders and dropped pairs of d digits and w weights stay below the bound
  stated for `slices`, for every number of slices;
* every INT32 sum and every sum over the slabs of a weight fits, whatever the
  output's size;
* an accumulator never holds more than 2^24 between drains: by the rule itself
  over the norms' range, and on digits that reach the norms."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1606_03416_gb300", "csrc")
SOURCE = r"""
#include "digit_rules.h"
using namespace dg;
extern "C" {
int n_digits(int s) { return digits_for(s); }
int n_weights(int s) { return weights_for(s); }
int n_pairs(int d, int t) { return pairs_of_weight(d, t); }
int max_pairs() { return kMaxPairs; }
int max_digits() { return kMaxDigits; }
int groups(int d, int w, int64_t tiles, int nsm, uint8_t* count) {
  const PairGroups g = pair_groups(d, w, tiles, nsm);
  std::copy(g.count, g.count + 16, count);
  return g.total;
}
int end_of(int np, int q, int count) { return group_end(np, q, count); }
int drain(uint64_t sq, int per_slice) { return drain_slices(sq, per_slice != 0); }
}
"""
SLICES = range(2, 17)
CHUNK = 4096


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "r.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "r.so"), str(d / "r.cpp")],
                   check=True)
    r = ctypes.CDLL(str(d / "r.so"))
    r.groups.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int64, ctypes.c_int, ctypes.c_void_p]
    r.drain.argtypes = [ctypes.c_uint64, ctypes.c_int]
    return r


def pairs(d, w):
    return [(i, j) for i in range(d) for j in range(d) if i + j < w]


def digits(x, e, d):
    """q_0 .. q_{d-1} of |x| < 2^e: x ~ 2^e sum q_i 2^(-8 - 9 i)."""
    v = Fraction(x) / Fraction(2) ** e
    if d <= 7:  # rounded once, half away from zero, then balanced digits from the last
        F = int(abs(v) * 2 ** (9 * d) + 1) // 2 * (1 if v >= 0 else -1)
        q = []
        for _ in range(d - 1):
            q.append((F + 256) % 512 - 256)
            F = (F - q[-1]) // 512
        return [F] + q[::-1]
    q, r = [], v * 256
    for _ in range(d):  # each digit rounded to nearest (ties to even) and subtracted
        q.append(round(r))
        r = (r - q[-1]) * 512
    return q


def test_counts(lib):
    for s in SLICES:
        d, w = lib.n_digits(s), lib.n_weights(s)
        assert 9 * d >= 6 * s + 1 and d <= lib.max_digits() and d <= w <= d + 1
        assert sum(lib.n_pairs(d, t) for t in range(w)) == len(pairs(d, w)) <= lib.max_pairs()
        # remainders and dropped pairs of a chunk, over L m_r n_c (2^e <= 2 m): stated for `slices`
        assert 4 * (d + 2) * Fraction(2) ** (-9 * d) <= (s + 4) * Fraction(2) ** (-6 * s)
    assert lib.n_digits(10) == 7 and len(pairs(7, lib.n_weights(10))) == 28


@pytest.mark.parametrize("nsm", [1, 2, 148, 152])
def test_integer_sums_fit(lib, nsm):
    for s in SLICES:
        d, w = lib.n_digits(s), lib.n_weights(s)
        for tiles in [1, 2, 3, 7, 40, 76, 500, 2 ** 20, 2 ** 40]:
            count = np.zeros(16, dtype=np.uint8)
            total = lib.groups(d, w, tiles, nsm, count.ctypes.data)
            assert total == count[:w].sum() and not count[w:].any()
            for t in range(w):
                np_, c = lib.n_pairs(d, t), int(count[t])
                assert c >= 1
                ends = [0] + [lib.end_of(np_, q, c) for q in range(c)]
                sizes = np.diff(ends)
                assert ends[-1] == np_ and sizes.min() >= 1
                assert sizes.max() * CHUNK * 2 ** 16 < 2 ** 31  # one INT32 sum
                assert np_ * CHUNK * 2 ** 16 < 2 ** 32          # the slabs of a weight together


@pytest.mark.parametrize("s", SLICES)
def test_digits_and_remainders(lib, s):
    d = lib.n_digits(s)
    rng = np.random.default_rng(s)
    x = rng.standard_normal(200) * 2.0 ** rng.integers(-70, 1, 200)
    x = np.concatenate([x, [0.0, 1.0 - 2.0 ** -53, -(1.0 - 2.0 ** -53), 0.5, 511 / 1024, 5e-324, 130816 / 2 ** 17]])
    e = int(np.frexp(np.abs(x).max())[1])
    for v in x:
        q = digits(float(v), e, d)
        assert all(abs(k) <= 256 for k in q)
        rest = Fraction(float(v)) - Fraction(2) ** e * sum(k * Fraction(2) ** (-8 - 9 * i) for i, k in enumerate(q))
        assert abs(rest) <= Fraction(2) ** (e - 9 * d)


@pytest.mark.parametrize("s", SLICES)
def test_products_meet_the_stated_bound(lib, s):
    """Rows whose rounding errors and digits have one sign are the worst for a sum."""
    d, w, L = lib.n_digits(s), lib.n_weights(s), 24
    rng = np.random.default_rng(100 + s)
    rows = [rng.standard_normal(L), np.abs(rng.standard_normal(L)), np.full(L, 1.0 - 2.0 ** -53),
            rng.uniform(0.999, 1.0, L), 2.0 ** rng.integers(-60, 1, L).astype(float)]
    for a in rows:
        for b in rows:
            ea, eb = (int(np.frexp(np.abs(v).max())[1]) for v in (a, b))
            qa, qb = ([digits(float(x), e, d) for x in v] for v, e in ((a, ea), (b, eb)))
            got = sum(Fraction(sum(qa[k][i] * qb[k][j] for k in range(L))) * Fraction(2) ** (-16 - 9 * (i + j))
                      for i, j in pairs(d, w)) * Fraction(2) ** (ea + eb)
            exact = sum(Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b))
            top = Fraction(float(np.abs(a).max())) * Fraction(float(np.abs(b).max()))
            assert abs(got - exact) <= L * top * (s + 4) * Fraction(2) ** (-6 * s)


@pytest.mark.parametrize("per_slice", [0, 1])
def test_drain_rule(lib, per_slice):
    block = 64 if per_slice else 512  # terms of a norm
    top = block * 2 ** 16             # its largest value
    rng = np.random.default_rng(7)
    norms = [0, 1, top] + [int(2.0 ** x) for x in rng.uniform(0, np.log2(top), 3000)]
    edges = [(2 ** 24 * 64 // (n * block)) ** 2 for n in range(1, 65)]  # sq at which n slices stop being allowed
    cases = [(a, b) for a, b in zip(norms, reversed(norms))] + [(q + k, 1) for q in edges for k in (-1, 0, 1) if q + k >= 0]
    for a, b in cases:
        n = lib.drain(a * b, per_slice)
        assert 4 <= n <= 64
        if n > 4:  # (n 64 / block) |a| |b| <= 2^24
            assert (n * 64) ** 2 * a * b <= (2 ** 24 * block) ** 2
            assert per_slice or n % 8 == 0
    assert lib.drain(top * top, per_slice) == 4 and lib.drain(0, per_slice) == 64


@pytest.mark.parametrize("per_slice", [0, 1])
@pytest.mark.parametrize("kind", ["equal", "sparse", "gauss"])
def test_no_accumulator_passes_2_24(lib, per_slice, kind):
    """Both operands the same digits, so that the norms' bound is reached."""
    block = 64 if per_slice else 512
    rng = np.random.default_rng(3)
    for v in [1, 2, 16, 100, 181, 255, 256]:
        a = np.full(CHUNK, v, dtype=np.int64)
        if kind == "sparse":
            a[rng.random(CHUNK) < 0.7] = 0
        if kind == "gauss":
            a = np.clip(np.rint(rng.standard_normal(CHUNK) * v / 2), -256, 256).astype(np.int64)
        norm = int((a.reshape(-1, block) ** 2).sum(1).max())
        n = lib.drain(norm * norm, per_slice)
        for k0 in range(0, CHUNK, 64 * n):
            assert (a[k0:k0 + 64 * n] ** 2).sum() <= 2 ** 24
