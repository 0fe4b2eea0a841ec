"""Launch shapes of the Euler-Maruyama kernel (csrc/euler_shape.cuh), compiled for the host:
over all particle counts, every CTA of a cluster owns particles (a CTA without any would be
ordered behind nobody while the others fill its barriers), the shares cover the particles
once and fit the block, the block fits the kernel's limits, and the order of the force sums
depends on the particle count alone."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1907_09529_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "euler_shape.cuh"
using namespace pamd;
template <typename R>
int check(int N, int chains, int sms)
{
    const double volume[] = {0.01 * N, 0.3 * N, 1.0 * N};
    for (double v : volume) {
        const EulerShape h = euler_shape<R>(N, chains, v, sms, 227 * 1024 - 1024);
        bool ok = h.cs >= 1 && h.cs <= 8 && (h.cs == 1 || h.cs * (long long)chains <= sms);
        ok = ok && euler_first(N, h.cs, 0) == 0 && euler_first(N, h.cs, h.cs) == N;
        for (int r = 0; r < h.cs; ++r) {
            const int n = euler_first(N, h.cs, r + 1) - euler_first(N, h.cs, r);
            ok = ok && n >= 1 && n <= h.nloc;
        }
        ok = ok && h.lg == euler_shape<R>(N, 1, v, 152, 227 * 1024 - 1024).lg;  // by N alone
        ok = ok && h.vr >= 0 && h.vr <= 2 && h.vr <= h.lg;
        ok = ok && (h.nloc << (h.lg - h.vr)) <= h.nt && h.nt % 32 == 0 && h.nt >= 64 && h.nt <= 1024 && h.lg <= 5;
        ok = ok && h.npad >= N && h.npad % (2 << h.lg) == 0 && h.smem <= 227 * 1024 - 1024 && h.smem % 16 == 0;
        ok = ok && (N <= kEulerDense ? h.cap == 0 && h.lg == (N <= kEulerOrdered ? 3 : N <= 128 ? 5 : 4) && (N > kEulerOrdered || h.vr == 0) : h.cap >= 1);
        if (!ok) {
            std::printf("N %d chains %d sms %d double %d: cs %d nloc %d lg %d nt %d cap %d npad %d smem %zu\n", N, chains,
                        sms, (int)(sizeof(R) == 8), h.cs, h.nloc, h.lg, h.nt, h.cap, h.npad, h.smem);
            return 1;
        }
    }
    return 0;
}
int main()
{
    int bad = 0;
    for (int sms : {152, 148, 60, 1})
        for (int N = 1; N <= 1024; ++N)
            for (int chains : {1, 2, 3, 7, 9, 18, 19, 20, 37, 38, 39, 75, 76, 77, 152, 153, 400})
                bad += check<float>(N, chains, sms) + check<double>(N, chains, sms);
    std::printf("bad %d\n", bad);
    return bad != 0;
}
"""


def test_every_cta_of_a_cluster_owns_particles(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "shape.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "shape")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I" + CSRC, "-o", exe, str(src)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[:2000]
