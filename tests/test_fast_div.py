"""Division by a number known on the host (FastDiv), run on the host, by the host's expression and by the kernels': divisors at powers of two,
beside them and beyond 2^31 with dividends at multiples of the divisor, beside them and at the ends of their range, and three million drawn pairs."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_05699_b200", "csrc")
SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "kvq_device.cuh"
static int check(long d, long n)
{
    const kvq::FastDiv f(d);
    if (n < 0) return 0;
    if (n < (1L << 31) && f.small((unsigned)n) != n / d) return printf("%ld / %ld: %u\n", n, d, f.small((unsigned)n));
    // what a kernel computes, __umulhi(2u * n, mul) >> shift
    const unsigned high = (unsigned)(((unsigned long)(2u * (unsigned)n) * f.mul) >> 32) >> f.shift;
    if (n < (1L << 31) && high != n / d) return printf("%ld / %ld: %u in a kernel\n", n, d, high);
    if (f(n) != n / d) return printf("%ld / %ld: %ld\n", n, d, (long)f(n));
    return 0;
}
int main()
{
    srand(1);
    for (int p = 0; p < 40; ++p)
        for (int o = -1; o <= 1; ++o) {
            const long d = (1L << p) + o;
            if (d < 1) continue;
            for (long k = 0; k < 50; ++k)
                for (int e = -1; e <= 1; ++e) {
                    const long top = ((1L << 31) - 1) / d * d;
                    if (check(d, k * d + e) || check(d, top - k * d + e) || check(d, (1L << 31) - 1 - k) || check(d, (1L << 31) + k)) return 1;
                }
        }
    for (long it = 0; it < 3000000; ++it) {
        const long d = 1 + (it % 2 ? rand() % 100000 : rand()), n = rand(), k = rand() % 1000;
        if (check(d, n) || check(d, k * d) || check(d, k * d - 1)) return 1;
    }
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="no nvcc")
def test_quotients_are_exact(tmp_path):
    src, exe = tmp_path / "div.cu", tmp_path / "div"
    src.write_text(SOURCE)
    subprocess.run(["nvcc", "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_100a,code=sm_100a", "-I", CSRC, "-o", str(exe), str(src)],
                   check=True, capture_output=True, text=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout
