"""The rule by which the solver kernels add a CTA's fp32 partial of an Eq. 2 /
Eq. 4 sum into an fp64 accumulator (quantize_partial in the kernels' internal
header): the partial is rounded up to a multiple of 2^-32 first. Pinned here by
arithmetic, on the host: sums of such terms below 2^21 are exact, hence the
same in every order of addition (the order in which CTAs arrive), while plain
fp64 sums of the same fp32 partials are not; a nonzero partial stays nonzero.
"""
from fractions import Fraction

import numpy as np

SCALE = 2.0 ** 32


def quantize_up(v32):
    return np.ceil(v32.astype(np.float64) * SCALE) / SCALE


def _partials(rng, n):
    # magnitudes from converged errors (1e-14) to early-iteration ones (1e3)
    return (10.0 ** rng.uniform(-14, 3, n)).astype(np.float32)


def test_rounding_is_up_by_less_than_one_step_and_keeps_nonzero():
    rng = np.random.default_rng(1)
    v = np.concatenate([_partials(rng, 5000), np.array([0.0, 1e-30, 2.0 ** -33, 2.0 ** -32], np.float32)])
    q = quantize_up(v)
    d = np.array([Fraction(float(a)) - Fraction(float(b)) for a, b in zip(q, v)])
    assert (d >= 0).all() and (d < Fraction(1, 2 ** 32)).all()
    assert ((q > 0) == (v > 0)).all()
    assert q[-1] == 2.0 ** -32 and q[-2] == 2.0 ** -32 and q[-4] == 0.0
    assert np.array_equal(q * SCALE, np.round(q * SCALE))   # multiples of 2^-32


def test_fp32_form_of_the_rounding_is_the_same():
    """The kernels round in fp32: values from 2^-9 on are multiples of 2^-32 as
    they are, smaller ones are scaled, rounded up and scaled back exactly."""
    rng = np.random.default_rng(4)
    edge = np.float32(2.0 ** -9)
    v = np.concatenate([_partials(rng, 20000), np.exp(rng.uniform(-100, 85, 20000)).astype(np.float32),
                        np.array([0.0, 1e-45, 2.0 ** -33, 2.0 ** -32, edge, np.nextafter(edge, np.float32(0)),
                                  np.nextafter(edge, np.float32(1)), 3e38, np.inf], np.float32)])
    v = np.concatenate([v, -v])
    with np.errstate(over="ignore"):
        got = np.where(np.abs(v) < edge, np.ceil(v * np.float32(SCALE)) * np.float32(1 / SCALE), v)
    assert got.dtype == np.float32
    assert np.array_equal(got.astype(np.float64), quantize_up(v))


def test_quantized_sums_are_exact_in_every_order():
    rng = np.random.default_rng(2)
    checked = 0
    for _ in range(30):
        n = int(rng.integers(2, 700))
        q = quantize_up(_partials(rng, n))
        exact = sum(Fraction(float(x)) for x in q)
        if exact >= 2 ** 21:
            continue
        for _ in range(20):
            s = 0.0
            for x in q[rng.permutation(n)]:
                s += float(x)
            assert Fraction(s) == exact
        checked += 1
    assert checked >= 20


def test_unquantized_fp64_sums_depend_on_the_order():
    """Why the rule exists: without it, the order of arrival moves the last bits."""
    rng = np.random.default_rng(3)
    differs = 0
    for _ in range(20):
        v = _partials(rng, 300).astype(np.float64)
        sums = set()
        for _ in range(20):
            s = 0.0
            for x in v[rng.permutation(len(v))]:
                s += float(x)
            sums.add(s)
        differs += len(sums) > 1
    assert differs > 0


PAIR_CHECK = r"""
#include "pa_pair.h"
#include <cstdint>
#include <cstdio>
int main() {
  uint64_t s = 88172645463325252ull;
  auto rnd = [&] { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; };
  int64_t bad = 0, short_bad = 0;
  for (int i = 0; i < 2000000; ++i) {
    // whole numbers, so that sums are exact in 64 bits: a high part of 24 bits in
    // units of 2^32 and a low part of 24 bits in units of 1 to 128
    const int64_t ah = (int64_t)(rnd() >> 41) + (1 << 22), dh = (int64_t)(rnd() >> 41) >> (rnd() % 24);
    auto low = [&] { return ((int64_t)(rnd() >> 40) - (1 << 23)) * ((int64_t)1 << (rnd() % 8)); };
    const int64_t al = low(), bl = low(), bh = -(ah - dh);  // from nearly -a to unrelated
    const pa::Pair a = {(float)ah * 0x1p32f, (float)al}, b = {(float)bh * 0x1p32f, (float)bl};
    const double want = (double)(((ah + bh) << 32) + al + bl), bound = 4 * 0x1p-48 * (want < 0 ? -want : want);
    auto off = [&](pa::Pair r) { const double d = pa::pair_value(r) - want; return (d < 0 ? -d : d) > bound; };
    bad += off(pa::pair_sub_full(a, pa::Pair{-b.h, -b.l}));
    short_bad += off(pa::pair_sub(a, pa::Pair{-b.h, -b.l}));
  }
  std::printf("%lld %d\n", (long long)bad, short_bad > 0);
  return 0;
}
"""


def test_pair_differences_are_accurate_where_they_cancel(tmp_path):
    """The difference F - G of a Parareal correction, compiled for the host: its
    error is bounded by the result however far the operands cancel, which that
    of the shorter subtraction is not."""
    import os
    import subprocess
    from paper_2609_36522_gb300 import build as pa_build
    src, exe = tmp_path / "pair.cpp", tmp_path / "pair"
    src.write_text(PAIR_CHECK)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", pa_build.CSRC, str(src), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    assert out == "0 1\n"
    with open(os.path.join(pa_build.CSRC, "k_srds.cu")) as f:
        assert "pair_sub_full(fv[k], gv[k])" in f.read()
