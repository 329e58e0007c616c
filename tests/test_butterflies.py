"""The butterflies of csrc/fft_radix.cuh on the host against 64-bit sums, with and without folded twiddles."""
import math
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_08393_b200", "csrc")

SOURCE = r"""
#include "fft_radix.cuh"
#include <cmath>
#include <complex>
#include <cstdio>
#include <random>
using namespace gleam;
template <int R, int DIR, bool FOLD> double error() {
    std::mt19937 gen(R);
    std::normal_distribution<double> normal;
    double e = 0, n = 0;
    for (int it = 0; it < 200; ++it) {
        cf v[R];
        std::complex<double> x[R];
        for (int i = 0; i < R; ++i) { v[i] = make_float2((float)normal(gen), (float)normal(gen)); x[i] = {v[i].x, v[i].y}; }
        Dft<R, DIR, FOLD>::run(v);
        for (int k = 0; k < R; ++k) {
            std::complex<double> s = 0;
            for (int m = 0; m < R; ++m) s += x[m] * std::polar(1.0, DIR * 2 * M_PI * ((m * k) % R) / R);
            e += std::norm(s - std::complex<double>(v[k].x, v[k].y));
            n += std::norm(s);
        }
    }
    return std::sqrt(e / n);
}
template <int R> void line() { printf("%d %.3e %.3e %.3e %.3e\n", R, error<R, -1, false>(), error<R, 1, false>(), error<R, -1, true>(), error<R, 1, true>()); }
int main() { line<2>(); line<4>(); line<5>(); line<6>(); line<8>(); line<10>(); line<12>(); line<15>(); line<16>(); line<20>(); line<23>(); line<32>(); return 0; }
"""


def test_butterflies_against_64_bit_sums(tmp_path):
    src, exe = tmp_path / "butterflies.cu", tmp_path / "butterflies"
    src.write_text(SOURCE)
    subprocess.run(["nvcc", "-std=c++17", "--expt-relaxed-constexpr", "-arch=sm_100", "-I", CSRC, "-O1", str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    for row in out.strip().split("\n"):
        r, *errors = [float(t) for t in row.split()]
        # each of log2 R stages rounds a value a few times (product, sum, constant): at most 2 * 2^-24 of its size per
        # stage in the root mean square; the direct sums of an odd prime P round P / 2 times, which add up as their root
        bound = 2 * 2.0 ** -24 * math.log2(r)
        assert max(errors) <= bound, (row, bound)
        # folding takes operations out: no larger error than without, but for the spread of the sample
        assert max(errors[2:]) <= 1.02 * max(errors[:2]), row
