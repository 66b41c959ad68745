"""Host rules that choose a launch's shape (csrc/ops.h), compiled for the CPU."""
import os
import subprocess

import pytest

from test_ntt_layout import CSRC, ROOT, nvcc

CHECK = r"""
#include "ops.h"
#include <cstdio>
using namespace ichee;
int main()
{
    int bad = 0;
    for (int logn = 10; logn <= 14; ++logn)
        for (u64 n : {1ull, 63ull, 64ull, 152ull, 5000ull}) {
            // a set shape stays, 256 threads among them; few ciphertexts of one image take a wide block each
            for (int set = 32; set <= 1024; set *= 2) {
                if (decrypt_threads(logn, n, set, true, 152) != set) ++bad;
                if (decrypt_threads(logn, n, set, false, 152) != (n < 64 ? 1024 : set)) ++bad;
            }
            // none set: whole warps, no more threads than loads of a polynomial
            for (bool batch : {false, true}) {
                const int t = decrypt_threads(logn, n, 0, batch, 152);
                if (t < 128 || t > 1024 || (t & (t - 1)) || t > (1 << logn) / 2) ++bad;
            }
        }
    // one ciphertext per SM: the fastest block of each ring, as measured
    const int fastest[] = {128, 256, 512, 512, 1024};
    for (int logn = 10; logn <= 14; ++logn)
        for (u64 n : {1ull, 152ull})
            if (decrypt_threads(logn, n, 0, false, 152) != fastest[logn - 10]) ++bad;
    // blend with a one-channel pattern: 16 blocks per SM, whatever their number, or 256 coefficients a share
    for (int sms : {76, 152, 304})
        for (int logn = 10; logn <= 14; ++logn)
            for (u64 px : {1ull, 30ull, 300ull, 3000ull}) {
                const u64 s = blend_splits(logn, px, sms), n = 1ull << logn;
                if (2 * px * s < 16ull * sms && n / s > 256) ++bad;
                if (s > 1 && px * s >= 16ull * sms) ++bad;   // half as many would do
                if (n % s || n / s < 256) ++bad;
            }
    std::printf("bad %d\n", bad);
    return bad != 0;
}
"""


def test_launch_rules(tmp_path):
    cc = nvcc()
    if cc is None:
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "rules.cu", tmp_path / "rules"
    src.write_text(CHECK)
    r = subprocess.run([cc, "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
