"""The FP64 path's fixed-point functions (csrc/fixed_math.cuh), compiled for the
host with the device intrinsics in plain C++, against long double: errors
relative to each result, however small it is, in units of 2^-53.

Bounds: the rounding to double is 1 unit at most (half a unit in the last
place next to a power of two); the sine's polynomial is off by 1.1 units at
most (its d^2/6 is kept to 2^-55 and d^2 to 2^-52.4), so 2.25 for sine and
cosine; the radius has half a unit before it is rounded, a normal is the
product of the two with one rounding, or, near a multiple of a quarter turn, of
three rounded factors: 3.
"""
import os
import re
import subprocess

import pytest

from paper_1908_03869_gb300 import build

SHIM = r"""
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <string>
#define __device__
#define __forceinline__ inline
#define __noinline__
#define __align__(n) __attribute__((aligned(n)))
using std::max;
using std::min;
struct ulonglong2 { unsigned long long x, y; };
struct double2 { double x, y; };
double2 make_double2(double x, double y) { return double2{x, y}; }
template <class T> T __ldg(const T *p) { return *p; }
uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
uint64_t words(uint32_t lo, uint32_t hi) { return ((uint64_t)hi << 32) | lo; }
uint32_t __funnelshift_r(uint32_t lo, uint32_t hi, uint32_t s) { return (uint32_t)(words(lo, hi) >> (s & 31)); }
uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, uint32_t s) { return (uint32_t)((words(lo, hi) << (s & 31)) >> 32); }
int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
uint64_t bits(double d) { uint64_t v; memcpy(&v, &d, 8); return v; }
int __double2hiint(double d) { return (int)(bits(d) >> 32); }
int __double2loint(double d) { return (int)bits(d); }
double __hiloint2double(int hi, int lo) { uint64_t v = words((uint32_t)lo, (uint32_t)hi); double d; memcpy(&d, &v, 8); return d; }
uint32_t __float_as_uint(float f) { uint32_t v; memcpy(&v, &f, 4); return v; }
float __uint2float_rz(uint32_t v) {
    const int cut = v < 1u << 24 ? 0 : 8 - __builtin_clz(v);
    return (float)(v >> cut << cut);
}
float __uint2float_rn(uint32_t v) { return (float)v; }
double __uint2double_rn(uint32_t v) { return v; }
uint32_t __float2uint_rz(float f) { return (uint32_t)f; }
void sincospi(double x, double *s, double *c) {
    const double q = std::floor(2 * x + 0.5);  // exact
    const long double r = M_PIl * ((long double)x - (long double)q / 2), a = sinl(r), b = cosl(r);
    const int k = (int)q & 3;
    *s = (double)(k == 0 ? a : k == 1 ? b : k == 2 ? -a : -b);
    *c = (double)(k == 0 ? b : k == 1 ? -a : k == 2 ? -b : a);
}
static double g_seed_error = 0;  // of the special-function unit's reciprocal square root, at most 2^-22.9
"""

PROGRAM = r"""
using namespace sdeb;
static long double units(double got, long double want) { return want == 0 ? (got == 0 ? 0 : INFINITY) : fabsl((got - want) / want) * 0x1p53L; }
static std::mt19937_64 g(11);
static double uniform(double a, double b) { return std::uniform_real_distribution<double>(a, b)(g); }
static double sign() { return g() & 1 ? 1.0 : -1.0; }
static long double log_of(uint32_t w) {  // ln((w + 1/2) 2^-32)
    return w >> 31 ? log1pl(-((0xffffffffu - w) + 0.5L) * 0x1p-32L) : logl((w + 0.5L) * 0x1p-32L);
}
static uint32_t word(int kind, long i) {
    const uint32_t d = (uint32_t)std::exp2(uniform(0, 32));
    return kind == 0 ? (uint32_t)g() : kind == 1 ? d - 1 : kind == 2 ? 0xffffffffu - (d - 1) : kind == 3 ? (uint32_t)i : 0xffffffffu - (uint32_t)i;
}
int main(int, char **argv) {
    const std::string what = argv[1];
    long double worst = 0;
    auto see = [&](long double u) { if (!(u <= worst)) worst = u; };
    if (what == "phases") {
        for (int kind = 0; kind < 7; ++kind)
            for (long i = 0; i < 400000; ++i) {
                double x = kind == 0 ? uniform(-M_PI, M_PI)
                           : kind == 1 ? sign() * std::exp2(uniform(-14, 24))
                           : kind == 2 ? sign() * std::exp2(uniform(-1074, 900))
                           : kind == 3 ? std::floor(uniform(0, 300)) * M_PI_2 + sign() * std::exp2(uniform(-45, -2))
                           : kind == 4 ? i * M_PI_2
                           : kind == 5 ? i % 65536 * (M_PI / 4096) + sign() * std::exp2(uniform(-50, -10))
                                       : uniform(0x1p-11, 0x1p-7);
                if (i < 6 && kind == 2) {
                    const double ends[6] = {0.0, 0x1p-11, std::nextafter(0x1p-11, 0), 0x1p21, std::nextafter(0x1p21, 0), 0x1p53};
                    x = ends[i];
                }
                double s, c;
                sincos_fixed(x, s, c);
                see(units(s, sinl(x)));
                see(units(c, cosl(x)));
            }
    } else if (what == "radius") {
        for (int seed = -1; seed <= 1; ++seed) {
            g_seed_error = seed * 0x1.125p-23;
            for (int kind = 0; kind < 5; ++kind)
                for (long i = 0; i < 200000; ++i) {
                    const uint32_t w = word(kind, i);
                    int h;
                    const uint64_t r = normal_radius(w, h);
                    const long double want = sqrtl(-2 * log_of(w));
                    see(fabsl((ldexpl((long double)r, h - 63) - want) / want) * 0x1p53L);
                }
        }
    } else if (what == "normals") {
        for (int kind = 0; kind < 5; ++kind)
            for (long i = 0; i < 300000; ++i) {
                const uint32_t a = word(kind % 3, i);
                const uint32_t b = kind < 3 ? (uint32_t)g() : (uint32_t)((g() << 30) + (int64_t)(sign() * std::exp2(uniform(0, 30))));
                double z[2];
                box_muller_fixed(a, b, z[0], z[1]);
                const uint64_t t = 2ull * b + 1;  // 33 bits of a turn
                const long double r = sqrtl(-2 * log_of(a)), f = (t & 0x7fffffffu) * 0x1p-31L;
                long double s = f <= 0.5L ? sinl(M_PI_2l * f) : cosl(M_PI_2l * (1 - f));
                long double c = f <= 0.5L ? cosl(M_PI_2l * f) : sinl(M_PI_2l * (1 - f));
                const int q = (int)(t >> 31);
                see(units(z[0], r * (q == 0 ? c : q == 1 ? -s : q == 2 ? -c : s)));
                see(units(z[1], r * (q == 0 ? s : q == 1 ? c : q == 2 ? -s : -c)));
            }
    }
    printf("%.4Lf\n", worst);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    """Builds a host program of the shim, the header and the given code."""
    where = tmp_path_factory.mktemp("fixed_math")
    os.makedirs(build.GEN_DIR, exist_ok=True)
    build.generate_fixed_tables()
    with open(build.FIXED_INC) as f:
        tables = f.read().replace("#pragma once", "")
    with open(os.path.join(build.CSRC, "fixed_math.cuh")) as f:
        header = f.read()
    header = re.sub(r'#include [<"](cuda_runtime\.h|sdeb_fixed_tables\.inc)[>"].*', "", header.replace("#pragma once", ""))
    header, seeds = re.subn(r'asm\("rsqrt\.approx.*', "r = (float)((1.0 + g_seed_error) / std::sqrt((double)y));", header)
    assert seeds == 1

    def make(code):
        src, exe = str(where / "program.cpp"), str(where / "program")
        with open(src, "w") as f:
            f.write(SHIM + tables + header + code)
        subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", src, "-o", exe], check=True)
        return lambda *args: subprocess.run([exe, *args], check=True, capture_output=True, text=True, timeout=600).stdout
    return make


@pytest.fixture(scope="module")
def worst(program):
    run = program(PROGRAM)
    return lambda what: float(run(what))


@pytest.mark.parametrize("what,bound", [("phases", 2.25), ("radius", 0.5), ("normals", 3.0)])
def test_errors_relative_to_the_result(worst, what, bound):
    assert worst(what) <= bound


SUMS = r"""
using namespace sdeb;
// t 2^-60 as a double, rounded to nearest (ties away from 0)
static double exact(__int128 t) {
    unsigned __int128 m = t < 0 ? -(unsigned __int128)t : (unsigned __int128)t;
    int n = 0;
    while (m >> n >> 53) ++n;
    if (n) m = (m + ((unsigned __int128)1 << (n - 1))) >> n;
    return (t < 0 ? -1 : 1) * std::ldexp((double)(uint64_t)m, n - 60);
}
int main() {
    std::mt19937_64 g(5);
    for (long i = 0; i < 2000000; ++i) {
        __int128 t = (__int128)(((unsigned __int128)g() << 64) | g()) >> (59 + g() % 69);  // at most 2^68
        if (i < 200) t = i - 100;
        const int64_t v = (int64_t)(t >> 6);
        const uint32_t rest = ((uint32_t)t & 63u) << 26;
        if (sum_to_double<true>(v, rest, 54) != exact(t) || sum_to_double<false>(v, rest, 54) != exact(t)) return 1;
    }
    for (long i = 0; i < 500000; ++i) {
        double x = std::exp2(-std::uniform_real_distribution<double>(0, 70)(g));
        const double ends[4] = {0.0, 1.0, 5e-324, 0x1p-60};
        if (i < 4) x = ends[i];
        if (to_q60((uint32_t)__double2hiint(x), (uint32_t)__double2loint(x)) != (uint64_t)std::ldexp(x, 60)) return 2;
    }
    return 0;
}
"""


def test_sums_to_double_and_back(program):
    program(SUMS)()
