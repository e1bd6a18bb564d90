"""The logarithm of the first guesses, compiled for the host, against the C library's in long double."""

import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_1802_04819_b200" / "csrc"

PROGRAM = r"""
#include <cstdio>
#include <random>
#include "slaq_log.cuh"

static double worst, worst_at;
static const double* tab;

static void look(double x) {
    const long double want = std::log((long double)x);
    if (want == 0.0L) {
        if (slaq::log_of_normal(x, tab) != 0.0) worst = 1e9, worst_at = x;
        return;
    }
    int e;
    std::frexp((double)want, &e);
    const double off = (double)(std::fabs((long double)slaq::log_of_normal(x, tab) - want) / std::ldexp(1.0L, e - 53));
    if (off > worst) worst = off, worst_at = x;
}

int main() {
    tab = slaq::log_table().data();
    std::mt19937_64 rng(7);
    std::uniform_real_distribution<double> u(0.0, 1.0);
    for (int i = 0; i < slaq::kLogBins; ++i) {   // both sides of every bin's edges, at three exponents, and inside
        const int64_t from = (int64_t)(slaq::kLogFrom + (i << slaq::kLogBinShift)) << 32, wide = (int64_t)1 << (32 + slaq::kLogBinShift);
        for (int64_t e : {0, -700, 900})
            for (int64_t k = -3; k <= 3; ++k) look(slaq::log_value(from + k + (e << 52)));
        for (int k = 0; k < 20000; ++k) look(slaq::log_value(from + (int64_t)(u(rng) * wide)));
    }
    for (int k = 0; k < 3000000; ++k) look(1.0 + (u(rng) - 0.5) * 0x1p-6);
    for (int k = 0; k < 1000000; ++k) look(std::exp2(-1021.9 + u(rng) * 2045.0));
    look(0x1p-1022), look(1.0), look(0x1.fffffffffffffp1023), look(0x1.fffffffffffffp-1), look(0x1.0000000000001p0);
    std::printf("%.6f %.17g\n", worst, worst_at);
}
"""


def test_error_in_ulp(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    source, program = tmp_path / "log.cpp", tmp_path / "log"
    source.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", str(CSRC), "-o", str(program), str(source)], check=True)
    worst, at = map(float, subprocess.run([str(program)], check=True, capture_output=True, text=True).stdout.split())
    # half an ulp for the last rounding; what is added before it is below 2^-7 of the result, so its roundings and the series' rest are below 0.01
    assert worst < 0.51, (worst, at)
