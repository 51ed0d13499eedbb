"""FP32 terms summed as integers (fix_term and fix_value in csrc/gfmc_packed.cuh), compiled
for the host from their own source: for |x| < 4 - 2^-20 the value is x to 2^-42 whatever the
bits of x (ties, subnormals, both ends), the flags stay clear, and non-finite values
and values out of range up to the largest float set them.  A sum of 2047 terms is exact
in the terms and does not depend on their order."""
import shutil
import subprocess

import pytest

from test_fixed_point import ROOT

SRC = f"{ROOT}/paper_1303_6016_gb300/csrc/gfmc_packed.cuh"

PRELUDE = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <cstdint>
#define __device__
#define __forceinline__ inline
static float __fadd_rn(float a, float b) { volatile float r = a + b; return r; }
static float __fsub_rn(float a, float b) { volatile float r = a - b; return r; }
struct float2 { float x, y; };
static float2 make_float2(float x, float y) { return {x, y}; }
static float2 __fadd2_rn(float2 a, float2 b) { return {__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y)}; }
static float2 __ffma2_rn(float2 a, float2 b, float2 c) { return {std::fma(a.x, b.x, c.x), std::fma(a.y, b.y, c.y)}; }
static int __float_as_int(float x) { int i; std::memcpy(&i, &x, 4); return i; }
static unsigned __float_as_uint(float x) { unsigned i; std::memcpy(&i, &x, 4); return i; }
"""

DRIVER = r"""
static int check(float x)
{
    unsigned bad = 0;
    const FixTerm t = fix_term(x, bad);
    const long long q = fix_value(t.hi, t.lo);
    FixTerm a, b;  // the packed form, in either place
    unsigned bad2 = 0;
    fix_terms(make_float2(x, 0.25f), a, b, bad2);
    if (bad2 != (bad | 0x41440000u) || (!(bad & kFixBad) && (a.hi != t.hi || a.lo != t.lo || fix_value(b.hi, b.lo) != 1ll << 58))) return 1;
    bad2 = 0;
    fix_terms(make_float2(-1.f, x), a, b, bad2);
    if (!(bad & kFixBad) && (b.hi != t.hi || b.lo != t.lo || fix_value(a.hi, a.lo) != -(1ll << 60) || (bad2 & kFixBad))) return 1;
    const bool ok = (bad & kFixBad) == 0;
    if (!(std::fabs(x) < 4.f - 0x1p-20f)) return std::fabs(x) < 4.1f ? 0 : ok;  // at the end of the range either is right
    if (!ok) return 1;
    if (t.lo > (1 << 20) || t.lo < -(1 << 20)) return 1;
    // |q 2^-60 - x| <= 2^-42, in integers of 2^-70 (x is a multiple of 2^-149: compare in long double)
    const long double d = (long double)q * 0x1p-60L - (long double)x;
    return !(std::fabs((double)d) <= 0x1p-42);
}

int main()
{
    int bad = 0;
    unsigned long long rng = 7;
    auto next = [&]() { rng = rng * 6364136223846793005ull + 1442695040888963407ull; return (unsigned)(rng >> 32); };
    auto from = [](unsigned b) { float x; std::memcpy(&x, &b, 4); return x; };
    for (int i = 0; i < 2000000; ++i) {
        const unsigned b = next();
        const float x = from((b & 0x80000000u) | (b % 0x40800001u));  // 0 .. 4, every exponent
        bad += check(x);
        bad += check(((int)next()) * 0x1p-31f);
        bad += check(((int)(next() % 4097u) - 2048) * 0x1p-21f);  // ties of the upper part
        bad += check(((int)(next() % 4097u) - 2048) * 0x1p-42f);  // ties of the lower part
    }
    const float odd[] = {0.f, -0.f, 3.999998f, -3.999998f, 1.f, -1.f, 0x1p-149f, -0x1p-149f, 0x1p-126f};
    for (float x : odd) bad += check(x);
    const float out[] = {INFINITY, -INFINITY, NAN, -NAN, 4.0000005f, -4.0000005f, 5.f, -7.5f, 100.f, -100.f, 0x1p127f, -0x1p127f, 3e38f};
    for (float x : out)
        bad += check(x);
    // sums: forward and backward the same, and the sum of the single terms
    int hi[2] = {0, 0}, lo[2] = {0, 0};
    long long want = 0;
    float v[2047];
    unsigned f = 0;
    for (int i = 0; i < 2047; ++i) v[i] = ((int)next()) * 0x1p-42f;
    for (int i = 0; i < 2047; ++i) {
        const FixTerm a = fix_term(v[i], f), b = fix_term(v[2046 - i], f);
        hi[0] += a.hi; lo[0] += a.lo; hi[1] += b.hi; lo[1] += b.lo;
        want += fix_value(a.hi, a.lo);
    }
    if (fix_value(hi[0], lo[0]) != want || fix_value(hi[1], lo[1]) != want) ++bad;
    std::printf("bad %d\n", bad);
    return bad != 0;
}
"""


def test_fix_term(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src = open(SRC).read()
    a = src.index("struct FixTerm {")
    b = src.index("\n}\n", src.index("void fix_terms")) + 3
    f = tmp_path / "fix.cpp"
    f.write_text(PRELUDE + src[a:b] + DRIVER)
    exe = tmp_path / "fix"
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-o", str(exe), str(f)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
