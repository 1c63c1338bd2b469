"""The FP64 helpers in integer and FP32 arithmetic (csrc/wf_bits.cuh), compiled for the host with the
intrinsics they use, against NumPy: conversions bit for bit (subnormals, ties, carries, both ends of
FP32's range, infinities and NaN), the reciprocal to the 0.51 units in the last place it states (and
bit for bit where it divides), the tests on the bits; signed overflow traps."""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_1210_4931_gb300", "csrc", "wf_bits.cuh")

HOST = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>
#define __device__
#define __forceinline__ inline
template <typename A, typename B> static A as(B b) { A a; static_assert(sizeof a == sizeof b, ""); std::memcpy(&a, &b, sizeof a); return a; }
static unsigned __float_as_uint(float f) { return as<unsigned>(f); }
static float __uint_as_float(unsigned u) { return as<float>(u); }
static long long __double_as_longlong(double v) { return as<long long>(v); }
static int __double2hiint(double v) { return (int)(as<unsigned long long>(v) >> 32); }
static int __double2loint(double v) { return (int)as<unsigned long long>(v); }
static double __hiloint2double(int h, int l) { return as<double>((unsigned long long)(unsigned)h << 32 | (unsigned)l); }
static float __frcp_rn(float f) { return 1.0f / f; }
using std::fma;
#include "wf_bits.cuh"
struct Out { double inv, wide; float narrow; int flags; };
int main()
{
    double v;
    while (std::fread(&v, 8, 1, stdin) == 1) {
        Out o;
        o.inv = wf::inverse(v);
        o.narrow = wf::narrow(v);
        o.wide = wf::widen(as<float>((unsigned)as<unsigned long long>(v)));  // the low word as an FP32 number
        o.flags = wf::positive_finite(v) | wf::finite_bits(v) << 1 | wf::positive(v) << 2 | wf::nonzero(v) << 3;
        std::fwrite(&o, sizeof o, 1, stdout);
    }
}
"""


def _values():
    rng = np.random.default_rng(3)
    anything = rng.integers(0, 1 << 64, 400000, dtype=np.uint64)
    sign = rng.integers(0, 2, 200000).astype(np.uint64) << np.uint64(63)
    # exponents of FP32 numbers, of its subnormals and of its largest; mantissas that tie, carry or are next to it
    e = rng.integers(1023 - 151, 1023 + 130, 200000).astype(np.uint64) << np.uint64(52)
    keep = rng.integers(0, 1 << 24, 200000).astype(np.uint64)
    keep[::5] = 0xffffff
    rest = rng.integers(0, 1 << 28, 200000).astype(np.uint64)
    rest[::3] = 0x8000000
    rest[1::3] = rng.integers(0x7fffffe, 0x8000003, rest[1::3].size).astype(np.uint64)
    ties = sign | e | (keep << np.uint64(28) | rest)
    ends = rng.integers(0, 1 << 52, 40000).astype(np.uint64) | rng.choice(
        [0, 1, 2, 21, 22, 23, 24, 895, 896, 897, 898, 1148, 1149, 1150, 1151, 2022, 2023, 2024, 2045, 2046, 2047],
        40000).astype(np.uint64) << np.uint64(52)
    words = np.array([0, 1, 0x7fffff, 0x800000, 0x7f7fffff, 0x7f800000, 0x7fc00000], dtype=np.uint64)
    words = np.concatenate([words, words | np.uint64(0x80000000)])  # low words: FP32 zeros, subnormals, ends
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.0 ** -126, 2.0 ** -149, 2.0 ** -150,
                        np.finfo(np.float32).max, np.finfo(float).max, np.finfo(float).tiny, 1.0, -1.0, 2.0]).view(np.uint64)
    return np.concatenate([anything, ties, ends, words, special]).view(np.float64)


@pytest.fixture(scope="module")
def results(tmp_path_factory):
    d = tmp_path_factory.mktemp("bits")
    src = d / "bits.cpp"
    src.write_text(HOST)
    exe = str(d / "bits")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fsanitize=signed-integer-overflow",
                    "-fsanitize-undefined-trap-on-error", "-I", os.path.dirname(HEADER), str(src), "-o", exe], check=True)
    v = _values()
    r = subprocess.run([exe], input=v.tobytes(), stdout=subprocess.PIPE, check=True)
    out = np.frombuffer(r.stdout, dtype=[("inv", "f8"), ("wide", "f8"), ("narrow", "f4"), ("flags", "i4")])
    assert out.size == v.size
    return v, out


def _same(a, b):
    assert np.all((a == b) & (np.signbit(a) == np.signbit(b)) | (np.isnan(a) & np.isnan(b)))


def test_narrow_and_widen(results):
    v, out = results
    with np.errstate(over="ignore", under="ignore", invalid="ignore"):
        _same(out["narrow"], v.astype(np.float32))
        _same(out["wide"], (v.view(np.uint64) & np.uint64(0xffffffff)).astype(np.uint32).view(np.float32).astype(np.float64))


def test_inverse(results):
    v, out = results
    with np.errstate(all="ignore"):
        q = 1.0 / v
        e = (v.view(np.uint64) >> np.uint64(52)) & np.uint64(0x7ff)
        series = (e >= 23) & (e <= 2023)
        _same(out["inv"][~series], q[~series])
        if np.finfo(np.longdouble).nmant < 60:
            pytest.skip("no extended precision")
        x, y = v[series].astype(np.longdouble), out["inv"][series]
        ulp = np.spacing(np.abs(q[series]))
        assert np.max(np.abs((y - 1 / x) / ulp)) < 0.51


def test_tests_on_the_bits(results):
    v, out = results
    with np.errstate(invalid="ignore"):
        want = (((v > 0) & np.isfinite(v)) | np.isfinite(v) << 1 | ((v > 0) & ~np.isnan(v)) << 2 | (v != 0) << 3)
    np.testing.assert_array_equal(out["flags"], want)
