"""Host-side transform tables against their definition: powers of a primitive 2N-th root in bit-reversed
order, their inverses, and exact companions floor(w 2^64 / q) (of 32 bits: the upper half), for the
smallest and largest primes and rings."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_03568_gb300", "csrc")

CHECK = r"""
#include "host_math.h"
#include <cstdio>
using namespace ichee::host;
int main()
{
    for (unsigned logn = 10; logn <= 14; logn += 2)
        for (unsigned bits : {20u, 28u, 40u, 60u, 61u}) {
            const u64 q = chain_prime(bits, logn, {}), n = 1ull << logn;
            std::vector<u64> t(4 * n);
            twiddle_pairs(q, logn, t.data());
            const u64 psi = t[2 * (n / 2)];   // bitrev(N/2) = 1
            bool ok = mulm(1, psi, q) == psi && powm(psi, n, q) == q - 1;
            u64 w = 1;
            for (unsigned e = 0; e < n; ++e, w = mulm(w, psi, q)) {
                unsigned k = 0;
                for (unsigned i = 0; i < logn; ++i) k |= ((e >> i) & 1u) << (logn - 1 - i);
                const u64 *f = &t[2 * k], *b = &t[2 * (n + k)];
                ok = ok && f[0] == w && f[1] == shoup_of(w, q) && mulm(f[0], b[0], q) == 1 && b[1] == shoup_of(b[0], q);
                if (bits <= 31) ok = ok && f[1] >> 32 == (w << 32) / q && b[1] >> 32 == (b[0] << 32) / q;
            }
            if (!ok) return std::printf("N = 2^%u, %u bits\n", logn, bits), 1;
        }
    // powers against squaring with 128-bit remainders
    for (u64 m : {3ull, 1048573ull, (1ull << 61) - 1, (1ull << 62) - 57}) {
        u64 w = 1 % m;
        for (unsigned e = 0; e < 70; ++e, w = mulm(w, 12345678901234567ull % m, m))
            if (powm(12345678901234567ull, e, m) != w) return std::printf("power %u mod %llu\n", e, (unsigned long long)m), 1;
    }
    return 0;
}
"""


def test_tables(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not found")
    src, exe = tmp_path / "tables.cpp", tmp_path / "tables"
    src.write_text(CHECK)
    r = subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
