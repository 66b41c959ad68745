"""Lazily reduced 64-bit arithmetic of the transforms and matching (csrc/ntt.cuh, common.cuh): the
three-product quotient, the two-step Montgomery product and the bounds the kernels carry through
the passes, host-compiled and checked against 128-bit integers on the largest operands each
takes; on the GPU, matching and the per-pixel form against the oracle on a ring with primes on both
sides of the size below which a transform folds nothing."""
import os
import subprocess

import numpy as np
import pytest

from test_ntt_layout import CSRC, ROOT, nvcc

CHECK = r'''
#include "ntt.cuh"
#include <cstdio>
#include <cstdlib>
using namespace ichee;
typedef unsigned __int128 u128;
static u64 rnd() { return ((u64)rand() << 42) ^ ((u64)rand() << 21) ^ (u64)rand(); }
static int check_products(u64 q, int caps)
{
    int bad = 0;
    u64 inv = q;
    for (int i = 0; i < 6; ++i) inv *= 2 - q * inv;
    const u64 qinv = 0 - inv;
    const u64 top = caps * (u128)q > ~0ull ? ~0ull : caps * q - 1;   // largest operand of a product by a twiddle
    for (int i = 0; i < 20000; ++i) {
        const u64 w = i & 1 ? q - 1 - (u64)i : rnd() % q, wp = (u64)(((u128)w << 64) / q);
        const u64 x = i % 3 == 0 ? top - (u64)(i / 3) : rnd() % top;
        const u64 r = shoup3(x, w, wp, q);
        if (r >= 4 * q || r % q != (u64)((u128)x * w % q)) ++bad;
        const u64 most = q < (1ull << 50) ? 62 * q - 1 : 4 * q - 1;
        const u64 a = i % 5 == 0 ? most - (u64)(i / 5) : rnd() % most, b = i % 7 == 0 ? most : rnd() % most;
        const u64 m = mont_lazy(a, b, q, qinv);
        // m 2^64 = a b mod q
        const u64 back = (u64)((u128)(m % q) * (u64)(((u128)1 << 64) % q) % q);
        if (q < (1ull << 60) && (m >= 2 * q || back != (u64)((u128)(a % q) * (b % q) % q))) ++bad;
    }
    return bad;
}
template <int E> static int check_bounds(int logn, int cap, int in)
{
    const int le = E == 16 ? 4 : 3;
    int bad = 0, b = in, iv = 4;
    for (int s0 = 0; s0 < logn; s0 += le) {
        const int s = logn - s0 < le ? logn - s0 : le;
        for (int k = 0; k < s; ++k) {
            const int x = fwd_bound(cap, b, k);
            if ((x + 4 > cap ? cap / 2 : x) + 4 > cap || x > cap) ++bad;   // a halved operand starts at most at cap
        }
        b = fwd_bound(cap, b, s);
    }
    for (int s0 = (logn - 1) / le * le; s0 >= 0; s0 -= le) {
        const int s = logn - s0 < le ? logn - s0 : le;
        for (int t = 0; t < s; ++t)
            for (int i = 0; i < (1 << s); ++i)
                if (2 * inv_before(cap, iv, t, i) > cap) ++bad;            // X + Y and X - Y + b q
        iv = inv_bound(cap, iv, s);
    }
    if (cap == 8 && iv != 4) ++bad;
    return bad;
}
int main()
{
    const u64 q60 = 1152921504606748673ull, q61 = 2305843009211662337ull, q40 = 1099511480321ull, q30 = 1073692673ull;
    int bad = check_products(q60, 16) + check_products(q61, 8) + check_products(q40, 62) + check_products(q30, 62) +
              check_products(1125899906777089ull, 62);
    for (int logn = 10; logn <= 14; ++logn)
        for (int cap : {8, 16}) {
            bad += check_bounds<8>(logn, cap, 2) + check_bounds<16>(logn, cap, 2) + check_bounds<8>(logn, cap, 1);
            if (cap == 16) bad += check_bounds<8>(logn, cap, 6);
        }
    // relinearisation's transforms in parts: 2 or 3 coupling stages from canonical values, then a part
    for (int logm = 8; logm <= 11; ++logm) bad += check_bounds<8>(logm, 8, 8);
    for (int ls = 2; ls <= 3; ++ls) {
        if (fwd_bound(8, 1, ls) > 8 || inv_bound(8, 4, ls) > 4) ++bad;
        for (int t = 0; t < ls; ++t)
            for (int i = 0; i < (1 << ls); ++i)
                if (2 * inv_before(8, 4, t, i) > 8) ++bad;
    }
    if (fwd_bound(kNoFold, 6, 13) > 62 || fwd_bound(kNoFold, 2, 13) > 62) ++bad;
    printf("bad %d\n", bad);
    return bad != 0;
}
'''


def test_products_and_bounds(tmp_path):
    cc = nvcc()
    if cc is None:
        pytest.skip("nvcc not found")
    src = tmp_path / "lazy.cu"
    src.write_text(CHECK)
    exe = tmp_path / "lazy"
    r = subprocess.run([cc, "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("ring", [
    dict(log_n=10, prime_bits=[60, 49, 50, 51], log2_scale=40, special_bits=61),
    dict(log_n=11, prime_bits=[60, 50], log2_scale=40, special_bits=61),   # the polynomials in turn up to here
    dict(log_n=12, prime_bits=[51, 50], log2_scale=40, special_bits=61),
    dict(log_n=13, prime_bits=[60, 49], log2_scale=40, special_bits=61),
    dict(log_n=14, prime_bits=[60, 50, 51], log2_scale=40, special_bits=61),
], ids=lambda r: "n%d" % (1 << r["log_n"]))
def test_matching_against_the_oracle(ring):
    torch = pytest.importorskip("torch")
    from oracle import Oracle, Params
    from paper_2409_03568_gb300 import ichee
    ctx = ichee.Context(**ring)
    ctx.keygen(51, with_evk=True)
    o = Oracle(Params(ring["log_n"], ring["prime_bits"], ring["log2_scale"], ring["special_bits"])).keygen(51, with_evk=True)
    n, L = ctx.n, ctx.L
    pa, pb = np.array([0, 255, 9], dtype=np.uint8), np.array([255, 0, 12], dtype=np.uint8)
    a, ma = ctx.encrypt(torch.from_numpy(pa).cuda(), 1, 3, 1, 5)
    b, mb = ctx.encrypt(torch.from_numpy(pb).cuda(), 1, 3, 1, 6)
    oa, ob = o.encrypt_pixels(pa, 5), o.encrypt_pixels(pb, 6)
    out, _ = ctx.eval(ichee.OP_SQDIFF_SUM, a, ma, b, mb, out_n_ct=1, out_level=L - 2)
    assert np.array_equal(out.cpu().numpy().view(np.uint64).reshape(1, 2, L - 1, n), o.match(oa, ob, o.delta)[0])
    out, _ = ctx.eval(ichee.OP_SQDIFF, a, ma, b, mb, out_level=L - 2)
    assert np.array_equal(out.cpu().numpy().view(np.uint64).reshape(3, 2, L - 1, n), o.sqdiff_image(oa, ob, o.delta)[0])
    ctx.close()
