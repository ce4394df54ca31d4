"""The 60-bit fixed-point arithmetic of FP64 plans (csrc/fixed.cuh), compiled for the host: values are rounded to
nearest, and no accumulator or limb leaves its word for the largest values under the worst signs."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1201_4060_gb300", "csrc")

PROGRAM = r"""
#define __host__
#define __device__
#define __forceinline__ inline
struct int4 { int x, y, z, w; };
#include "fixed.cuh"
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
using namespace bs::fixed;

static long long to_fixed(double v, int emax, int bits) {
    unsigned long long b;
    std::memcpy(&b, &v, 8);
    return from_double((unsigned)(b >> 32), (unsigned)b, emax, bits);
}

static int rounding() {                                  // |V - v 2^(1022 + bits - emax)| <= 1/2
    std::mt19937_64 r(1);
    std::uniform_real_distribution<double> u(-1, 1);
    for (int k = 0; k < 200000; ++k) {
        const int bits = 59 + (k & 1), emax = 1022;
        const double v = std::ldexp(u(r), -(int)(r() % 70));
        const long double want = std::ldexp((long double)v, bits);
        if (std::fabs((long double)to_fixed(v, emax, bits) - want) > 0.5L) return std::printf("rounding %a\n", v), 1;
    }
    return to_fixed(0.0, 128, 60) || to_fixed(-0.0, 128, 60) || to_fixed(5e-324, 128, 60);
}

// The contraction of values of magnitude 2^bits whose signs follow the derivative weights of the axes in `mask`.
template <int n> int extremes() {
    const long long top = 1LL << value_bits<n>();
    for (int k = 0; k <= 64; ++k) {
        const long long T = k < 64 ? (1LL << 54) * k : (1LL << 60) - 1;
        Limbs w[n], dw[n];
        weights<n>(T, w, dw);
        long double W[n], D[n];
        for (int j = 0; j < n; ++j) W[j] = std::ldexp((long double)value(w[j]), -60), D[j] = std::ldexp((long double)value(dw[j]), -60);
        for (int mask = 0; mask < 16; ++mask) {
            auto sign = [&](int j, int axis) { return (mask >> axis & 1) && value(dw[j]) < 0 ? -1 : 1; };
            auto at = [&](int x, int y, int z) {
                const int s = sign(x, 0) * sign(y, 1) * sign(z, 2) * (mask & 8 ? -1 : 1);
                return limbs(s * top);
            };
            auto wx = [&](int j) { return int4{w[j].hi, w[j].lo, dw[j].hi, dw[j].lo}; };
            long long out[4];
            unsigned size;
            contract<n, true>(at, wx, w, dw, w, dw, out, &size);
            long double want[4] = {0, 0, 0, 0};
            for (int x = 0; x < n; ++x)
                for (int y = 0; y < n; ++y)
                    for (int z = 0; z < n; ++z) {
                        const long double a = (long double)value(at(x, y, z));
                        want[0] += W[x] * W[y] * W[z] * a;
                        want[1] += D[x] * W[y] * W[z] * a;
                        want[2] += W[x] * D[y] * W[z] * a;
                        want[3] += W[x] * W[y] * D[z] * a;
                    }
            for (int e = 0; e < 4; ++e)
                if (std::fabs((long double)out[e] - want[e]) > 32.0L)
                    return std::printf("order %d t %d mask %d result %d: %lld, %.1Lf\n", n, k, mask, e, out[e], want[e]), 1;
            if ((mask & 7) == 0 && size < (unsigned)((top >> 34) - (top >> 44))) return std::printf("size %u\n", size), 1;
        }
    }
    return 0;
}

int main() {
    return rounding() || extremes<3>() || extremes<4>() || extremes<5>() || extremes<6>() || extremes<7>() || extremes<8>();
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host compiler")
def test_rounding_and_extremes(tmp_path):
    """The results are held to 32 units: three levels of rounding (a few units each, times the derivative weights'
    sums of up to 2) and the long double reference's own 2^-64 of values up to 2^61."""
    src, exe = tmp_path / "fixed.cpp", tmp_path / "fixed"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-fwrapv", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
