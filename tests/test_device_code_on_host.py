"""Device functions compiled with the host compiler (no GPU): the rotation of a Hessenberg column by one
warp, its lanes run one after another between warp-wide operations in several orders, and the conversions
between the precisions on integer instructions against the conversions themselves."""
import glob
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1012_4307_gb300", "csrc")

ROTATION = r"""
#include <stdio.h>
#include "warp_on_host.h"
#include "givens.cuh"
#include <complex>
typedef std::complex<double> cd;

static double2 d2(cd v) { return make_double2(v.real(), v.imag()); }
static cd c(double2 v) { return cd(v.x, v.y); }

int main() {
    unsigned long long seed = 1;
    auto rnd = [&]() { seed = seed * 6364136223846793005ull + 1442695040888963407ull; return (double)(seed >> 33) / 1073741824.0 - 1.0; };
    int orders[4][32];
    for (int q = 0; q < 32; q++) {
        orders[0][q] = q;
        orders[1][q] = 31 - q;
        orders[2][q] = (q * 13 + 5) % 32;
        orders[3][q] = q ^ 3;  // lanes 3, 2, 1, 0 first
    }
    const int M = 40, ldh = M + 1;
    for (int o = 0; o < 4; o++) {
        std::vector<double2> H(ldh * M), sn(M), g(M + 1, make_double2(0, 0));
        std::vector<double> cs(M), est(M), host(M);
        std::vector<cd> rg(M + 1, cd(0, 0)), rs(M);
        std::vector<double> rc(M);
        double2 fnorm = make_double2(3.0, 0.0);
        g[0] = make_double2(2.5, 0.0);
        rg[0] = 2.5;
        double worst = 0.0;
        for (int j = 0; j < M; j++) {
            std::vector<cd> col(j + 2);
            for (int i = 0; i <= j; i++) col[i] = cd(rnd(), rnd());
            col[j + 1] = fabs(rnd()) + 0.1;
            for (int i = 0; i <= j + 1; i++) H[ldh * j + i] = d2(col[i]);
            run_warp(orders[o], [&]() { givens_body(H.data(), ldh, j, cs.data(), sn.data(), g.data(), &fnorm, est.data(), host.data()); });
            // the same rotations, one after another
            for (int i = 0; i < j; i++) {
                const cd a = col[i], b = col[i + 1];
                col[i] = rc[i] * a + rs[i] * b;
                col[i + 1] = rc[i] * b - conj(rs[i]) * a;
            }
            const cd a = col[j], b = col[j + 1];
            const double t = sqrt(norm(a) + norm(b));
            rc[j] = abs(a) / t;
            rs[j] = a / abs(a) * conj(b) / t;
            col[j] = rc[j] * a + rs[j] * b;
            col[j + 1] = 0.0;
            rg[j + 1] = -conj(rs[j]) * rg[j];
            rg[j] *= rc[j];
            for (int i = 0; i <= j + 1; i++) worst = fmax(worst, abs(c(H[ldh * j + i]) - col[i]));
            worst = fmax(worst, fabs(cs[j] - rc[j]) + abs(c(sn[j]) - rs[j]) + abs(c(g[j]) - rg[j]) + abs(c(g[j + 1]) - rg[j + 1]));
            worst = fmax(worst, fabs(est[j] - abs(rg[j + 1]) / 3.0) + fabs(host[j] - est[j]));
        }
        // entries of size one, at most some 40 rotations of a few roundings each
        if (!(worst <= 1e-13)) printf("lane order %d: off by %g\n", o, worst);
    }
    return 0;
}
"""

CONVERSIONS = r"""
#include <stdio.h>
#include <stdint.h>
#include "warp_on_host.h"
#include "helm_internal.h"

static uint64_t state = 88172645463325252ull;
static uint64_t next() { state ^= state << 13; state ^= state >> 7; state ^= state << 17; return state; }
static uint32_t fb(float v) { return bits_as<uint32_t>(v); }
static uint64_t db(double v) { return bits_as<uint64_t>(v); }

static void narrow(uint64_t bits) {
    const double x = bits_as<double>(bits);
    const float a = to_float(x), b = (float)x;
    if (fb(a) != fb(b) && !(x != x && a != a)) printf("to_float(%a) = %a, not %a\n", x, a, b);
}

static void widen(uint32_t bits) {
    const float x = bits_as<float>(bits);
    const double a = to_double(x), b = (double)x;
    if (db(a) != db(b) && !(x != x && a != a)) printf("to_double(%a) = %a, not %a\n", x, a, b);
}

int main() {
    // every exponent with the 29 bits below a float's last one at and around one half, either sign
    for (uint64_t e = 0; e < 2048; e++)
        for (uint64_t top : {0ull, 1ull, 2ull, 0x7ffffeull, 0x7fffffull})
            for (uint64_t low : {0ull, 1ull, 0xfffffffull, 0x10000000ull, 0x10000001ull, 0x1fffffffull})
                for (uint64_t s = 0; s < 2; s++) narrow(s << 63 | e << 52 | top << 29 | low);
    for (int q = 0; q < 20000000; q++) {
        const uint64_t v = next();
        narrow(v);
        narrow((v & 0x800fffffffffffffull) | (uint64_t)(860 + v % 330) << 52);  // around float's range
    }
    for (uint32_t e = 0; e < 512; e++)  // either sign, every exponent
        for (uint32_t f : {0u, 1u, 2u, 0x3fffffu, 0x400000u, 0x400001u, 0x7ffffeu, 0x7fffffu}) widen(e << 23 | f);
    for (uint64_t v = 0; v < 1ull << 32; v += 97) widen((uint32_t)v);
    return 0;
}
"""


def run(tmp_path, program):
    cxx = shutil.which("g++")
    inc = [p for p in ["/usr/local/cuda/include"] + glob.glob("/usr/local/cuda*/include") if os.path.exists(p + "/cuda_runtime.h")]
    if cxx is None or not inc:
        pytest.skip("no host C++ compiler or no CUDA headers")
    src, exe = tmp_path / "p.cc", tmp_path / "p"
    src.write_text(program)
    # no contraction beyond the code's own fma, as for the oracle
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-w", "-I", HERE, "-I", CSRC, "-I", inc[0], str(src),
                    "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout


def test_rotation_in_any_lane_order(tmp_path):
    out = run(tmp_path, ROTATION)
    assert out == "", out


def test_conversions_are_bit_equal(tmp_path):
    out = run(tmp_path, CONVERSIONS)
    assert out == "", out[:2000]
