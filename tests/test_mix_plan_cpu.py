"""The radix plans of the any-length stage kernel, made on the host in the calls that
execute transforms: no host allocation (an exception would leave a C entry), and every
length up to 2048 with factors 2, 3, 5 and 7 has one whose tables index the line
exactly.  The plan source is compiled by itself; nothing here needs a GPU."""
import os
import subprocess

from paper_1501_07350_gb300 import _build

ALLOCATOR = r"""
#include <cstdlib>
#include <new>
bool closed = false;
void* operator new(std::size_t n) { if (closed) std::abort(); return std::malloc(n); }
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
"""

HARNESS = r"""
#include <cstdio>
#include "fft_mix.cuh"

extern bool closed;

int main()
{
    closed = true;
    for (int df = 0; df < 2; ++df)
        for (int n = 1; n <= 2048; ++n) {
            int rest = n;
            for (int f : {2, 3, 5, 7}) while (rest % f == 0) rest /= f;
            const ofg::MixPlan pl = ofg::mix_radix_plan(n, df != 0);
            if ((pl.npass > 0) != (rest == 1)) return std::printf("%d: plan or none\n", n), 1;
            int m = 1;
            for (int p = 0; p < pl.npass; ++p) {
                const ofg::MixPass& ps = pl.pass[p];
                if (ps.radix * ps.nbf != n || ps.m != m || ps.s * m * ps.radix != n) return std::printf("%d: pass %d\n", n, p), 1;
                for (int b = 0; b < ps.nbf; ++b)
                    if ((int)(((unsigned)b * ps.inv) >> 20) != b / m) return std::printf("%d: %d / %d\n", n, b, m), 1;
                m *= ps.radix;
            }
            if (pl.npass && m != n) return std::printf("%d: product\n", n), 1;
        }
    std::puts("ok");
    return 0;
}
"""


def test_plans_of_every_length_without_an_allocation(tmp_path):
    src, alloc, exe = tmp_path / "plans.cu", tmp_path / "alloc.cpp", tmp_path / "plans"
    src.write_text(HARNESS)
    alloc.write_text(ALLOCATOR)
    cmd = [_build._nvcc(), *_build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I" + _build.CSRC, "-I" + _build.INCLUDE,
           str(src), str(alloc), os.path.join(_build.CSRC, "fft_mix_plan.cu"), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", (r.returncode, r.stdout)
