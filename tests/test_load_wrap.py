"""The load's periodic wrap of a coordinate, the kernel's own function compiled
for the host: bit for bit the remainder that exact arithmetic rounds to (fmod is
exact; a negative one has the box's length added, once rounded), in [0, n), for
coordinates in, near and up to the largest finite number away from the box.
Beyond 2^53 boxes a single pass left a coordinate outside the grid."""
import subprocess

from paper_2509_11100_gb300 import build

SOURCE = r"""
#include "common.cuh"
#include <cstdio>
#include <random>
int main()
{
    std::mt19937_64 r(7);
    std::uniform_real_distribution<double> u(1.0, 2.0);
    long wrong = 0, outside = 0, seen = 0;
    auto check = [&](double x, int n) {
        double want = std::fmod(x, n);
        if (want < 0.0) want += n;
        if (want >= n) want = 0.0;   // rounds to the box's length: its beginning
        const double got = relsim::wrap_coord(x, n);
        outside += !(got >= 0.0 && got < n);
        wrong += got != want;
        ++seen;
    };
    const int ns[] = {3, 4, 5, 37, 99, 128, 251, 1024, 12345, 1 << 20, (1 << 28) - 3};
    for (int n : ns) {
        for (int e = -1074; e <= 1023; ++e)
            for (int k = 0; k < 40; ++k) {
                const double x = std::ldexp(u(r), e);
                check(x, n);
                check(-x, n);
            }
        for (long k = -5; k <= 5; ++k)
            for (int d = -3; d <= 3; ++d) {
                double x = (double)n * k;
                for (int q = 0; q < (d < 0 ? -d : d); ++q) x = std::nextafter(x, d < 0 ? -1e308 : 1e308);
                check(x, n);
            }
        check(3.3e25, n);
        check(1.7976931348623157e308, n);
        check(-1.7976931348623157e308, n);
    }
    std::printf("%ld %ld %ld\n", seen, outside, wrong);
}
"""


def test_wrapped_coordinate_is_the_exact_remainder(tmp_path):
    src, exe = tmp_path / "wrap.cu", tmp_path / "wrap"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc()] + build.ARCH + build.NVFLAGS + [str(src), "-o", str(exe)], check=True)
    seen, outside, wrong = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert seen > 1e6 and outside == 0 and wrong == 0
