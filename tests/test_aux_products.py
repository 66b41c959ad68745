"""Fresh encryption's exact products modulo 28-bit auxiliary primes (csrc/ntt32.cuh, kernels_enc.cu).

On the CPU: the 32-bit exchange layouts (host-compiled), the butterfly ranges, and the
reconstruction modulo a limb's prime from the CRT digits, with exact Python integers, for every
prime size and ring degree the library accepts. On the GPU: fresh ciphertexts against the oracle on
rings at the edges of the two- and three-prime limbs."""
import os
import random
import subprocess

import numpy as np
import pytest

from test_ntt_layout import CSRC, ROOT, nvcc

CHECK = r'''
#include "ntt32.cuh"
#include <cstdio>
using namespace ichee;
// bounds through the passes of a transform, as the code takes them
template <int E> static int check(int logn)
{
    const int le = E == 16 ? 4 : 3, T = (1 << logn) / E;
    int bad = 0, bf = 1, bt = 2, bi = 2;
    for (int s0 = 0; s0 < logn; s0 += le) {
        const int s = logn - s0 < le ? logn - s0 : le;
        bf = fwd32_bound(bf, s);
        bt = fwd32_bound(bt, s);
        if (bf > 16 || bt > 16) ++bad;
        for (int e = 0; e < E; ++e)
            for (int w = 0; w < T; w += 32) {
                unsigned banks = 0;
                for (int t = w; t < w + 32; ++t) {
                    const int x = elem_index_of(logn, s0, E, t, e);
                    banks |= 1u << (swz32<E>(x) & 31);
                    if (swz32<E>(x) != (swz32<E>(elem_index_of(logn, s0, E, t, 0)) ^ swz32<E>(elem_index_of(logn, s0, E, 0, e))))
                        ++bad;
                    if (swz32<E>(x) >> logn) ++bad;
                }
                if (banks != 0xffffffffu) ++bad;
            }
    }
    for (int s0 = (logn - 1) / le * le; s0 >= 0; s0 -= le) {
        const int s = logn - s0 < le ? logn - s0 : le;
        bi = inv32_bound(bi, s);
        if (bi > 16) ++bad;
    }
    return bad;
}
int main()
{
    int bad = 0;
    for (int logn = 10; logn <= 14; ++logn) bad += check<8>(logn) + check<16>(logn);
    printf("bad %d\n", bad);
    return bad != 0;
}
'''


def test_exchange_layout_and_bounds(tmp_path):
    cc = nvcc()
    if cc is None:
        pytest.skip("nvcc not found")
    src = tmp_path / "check32.cu"
    src.write_text(CHECK)
    exe = tmp_path / "check32"
    r = subprocess.run([cc, "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def primes_below(bits, logn, count):
    isprime = pytest.importorskip("sympy").isprime
    step = 2 << logn
    c = ((1 << bits) - 1) // step * step + 1
    out = []
    while len(out) < count and c > 1 << (bits - 1):
        if c < 1 << bits and isprime(c):
            out.append(c)
        c -= step
    return out


@pytest.mark.parametrize("logn", range(10, 15))
def test_reconstruction_modulo_the_limb(logn):
    n = 1 << logn
    aux = primes_below(28, logn, 3)
    assert len(aux) == 3 and (1 << 28) - aux[-1] <= 1 << 22
    for p in aux:   # the fold by the top bits ends below 2p; sixteen multiples of p fit a word
        assert (1 << 28) + 15 * ((1 << 28) - p) < 2 * p and 16 * p < 1 << 32
    rng = random.Random(logn)
    for bits in range(20, 61):
        for q in primes_below(bits, logn, 1):
            np_ = 2 if n * (q // 2) <= aux[0] * aux[1] // 4 else 3
            ps = aux[:np_]
            M = int(np.prod([int(p) for p in ps], dtype=object))
            assert n * (q // 2) <= M // 4
            t = bits - 33 if bits > 32 else bits - 1
            mu = (1 << (bits + 31)) // q
            assert mu < 1 << 32
            mi = [M // p % q for p in ps]
            c0 = 2 * q - 32 - 5 * ps[-1] * mi[-1] % q
            top = n * (q // 2)
            for x in [0, 1, -1, top, -top, q // 2, -(q // 2)] + [rng.randint(-top, top) for _ in range(40)]:
                y = [x * pow(M // p, -1, p) % p for p in ps]
                y = [v + p * rng.randint(0, 1) for v, p in zip(y, ps)]   # the lazy range [0, 2p)
                k = (sum(y) + (1 << 27)) >> 28
                d = y[:-1] + [y[-1] + (5 - k) * ps[-1]]                  # the last digit less k primes, offset
                assert 0 < d[-1] < 1 << 32 and sum(d) < 1 << 31
                for e in (-31, 0, 31):
                    lo = c0 + e + 32 + sum(v * (m & 0xffffffff) for v, m in zip(d, mi))
                    hi = sum(v * (m >> 32) for v, m in zip(d, mi))
                    assert lo < 1 << 64 and hi + (lo >> 32) < 1 << 64
                    T = (hi + (lo >> 32) if bits > 32 else lo) >> t
                    assert T < 1 << 32 and (bits > 32 or hi == 0)
                    r = lo + (hi << 32) - (T * mu >> 32) * q
                    assert 0 <= r < 3 * q
                    r = r - 2 * q if r >= 2 * q else r
                    r = r - q if r >= q else r
                    assert r == (x + e) % q


@pytest.mark.gpu
@pytest.mark.parametrize("ring", [
    dict(log_n=10, prime_bits=[20, 29, 45, 46, 60], log2_scale=15),    # two primes up to 45 bits at N = 2^10
    dict(log_n=11, prime_bits=[60, 30, 44, 45], log2_scale=25),
    dict(log_n=12, prime_bits=[43, 44], log2_scale=30),
    dict(log_n=13, prime_bits=[41, 42, 43], log2_scale=30),
    dict(log_n=14, prime_bits=[41, 40, 60, 42], log2_scale=30),        # the third prime's digits wait in the output
], ids=lambda r: "n%d" % (1 << r["log_n"]))
def test_fresh_against_the_oracle(ring):
    torch = pytest.importorskip("torch")
    from oracle import Oracle, Params
    from paper_2409_03568_gb300 import ichee
    ctx = ichee.Context(**ring)
    ctx.keygen(31)
    o = Oracle(Params(ring["log_n"], ring["prime_bits"], ring["log2_scale"])).keygen(31)
    px = np.array([0, 255, 1, 7, 128], dtype=np.uint8)
    ct, _ = ctx.encrypt(torch.from_numpy(px).cuda(), 1, 5, 1, 77)
    got = ct.cpu().numpy().view(np.uint64).reshape(5, 2, ctx.L, ctx.n)
    assert np.array_equal(got, o.encrypt_pixels(px, 77))
    # the batched kernel: the same ciphertexts for two one-row images
    dst = [ctx.empty_cts(3, ctx.L - 1), ctx.empty_cts(2, ctx.L - 1)]
    d = torch.from_numpy(px).cuda()
    ichee.ichee_encrypt_batch(ctx.handle, None, [d[:3].clone(), d[3:].clone()], [(1, 3, 1), (1, 2, 1)], [77, 78], dst,
                              ctx.stream())
    assert np.array_equal(dst[0].cpu().numpy().view(np.uint64).reshape(3, 2, ctx.L, ctx.n), got[:3])
    ref = o.encrypt_pixels(px[3:], 78)
    assert np.array_equal(dst[1].cpu().numpy().view(np.uint64).reshape(2, 2, ctx.L, ctx.n), ref)
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("ring", [
    dict(log_n=10, prime_bits=[30, 30], log2_scale=25),                # one and two groups
    dict(log_n=11, prime_bits=[30, 60, 44, 45, 29], log2_scale=25),    # groups with and without three primes
    dict(log_n=14, prime_bits=[60, 40, 40], log2_scale=30),
], ids=lambda r: "n%d" % (1 << r["log_n"]))
def test_few_ciphertexts_shared_out_by_limbs(ring):
    """A call of so few pixels that several blocks share a ciphertext gives the first ciphertexts of a
    larger call, for every number of groups and at both sides of each line."""
    torch = pytest.importorskip("torch")
    from paper_2409_03568_gb300 import ichee
    ctx = ichee.Context(**ring)
    ctx.keygen(8)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    px = torch.randint(0, 256, (sms,), dtype=torch.uint8, device="cuda")
    whole, _ = ctx.encrypt(px, 1, sms, 1, 5)
    for n in sorted({1} | {sms // g + d for g in range(2, ctx.L + 1) for d in (0, 1)}):
        part, _ = ctx.encrypt(px[:n].clone(), 1, n, 1, 5)
        assert torch.equal(part.view(torch.int64).flatten(), whole.view(torch.int64).flatten()[:part.numel()]), n
