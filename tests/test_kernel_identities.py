"""Checks of three shortcuts in the kernels' modular arithmetic on the prime chains of every workload
(primes from the oracle's generator):

* the per-pixel squared difference lifts a digit of t2 (Sec. 2.2.3, relinearisation by hybrid
  key switching; the digit is centered, its magnitude below half its prime q_j) into a
  modulus q >= q_j without a reduction: v if v <= (q_j - 1) / 2, else q - (q_j - v) (with exact Python
  integers);
* fresh encryption's reconstruction (Sec. 2.2.2; enc_crt, compiled from the kernel's source) gives
  the canonical residue of an integer product and the Gaussian noise (|e| <= 31) from the product's
  digits modulo the auxiliary primes, each anywhere in [0, 2p);
* the key-switching accumulators (halve and shoup3, from the kernels' source) stay in [0, 4q), the
  range that the inverse transform takes, and keep their sum modulo q, for primes up to 61 bits."""
import random

import pytest

from oracle.ckks import Oracle, Params
from paper_2409_03568_gb300 import workloads as W
from test_block_races_cpu import run_on_host

RINGS = [W.ENC8192, W.OPS8192, W.RING16384,
         dict(log_n=10, prime_bits=[60, 40, 40, 40], log2_scale=40, special_bits=61)]


def moduli(ring):
    o = Oracle(Params(ring["log_n"], ring["prime_bits"], ring["log2_scale"], ring["special_bits"]))
    return [int(q) for q in o.q], int(o.P)


@pytest.mark.parametrize("ring", RINGS, ids=lambda r: r.get("name", "n1024_4primes"))
def test_digit_lift_without_reduction(ring):
    qs, P = moduli(ring)
    rng = random.Random(5)
    pairs = 0
    for qj in qs:
        half = (qj - 1) // 2
        for q in qs + [P]:
            if q == qj or qj > q:
                continue   # these pairs keep the Barrett reduction
            pairs += 1
            for v in [0, 1, half - 1, half, half + 1, qj - 2, qj - 1] + [rng.randrange(qj) for _ in range(200)]:
                lifted = v if v <= half else q - (qj - v)
                centered = v if v <= half else v - qj
                assert 0 <= lifted < q
                assert lifted == centered % q
    assert pairs > 0   # at least the lifts into P take the shortcut


RECONSTRUCTION = r"""
#include "shim.h"
#include "host_math.h"
#include "kernels_enc_host.h"
#include <random>
namespace ichee { u64 smem[1], sm[1]; }
using namespace ichee;
namespace hm = ichee::host;
typedef __int128 i128;
static int check(int logn, u64 q, int bits)
{
    std::mt19937_64 rng(q);
    std::vector<u64> p;
    for (int i = 0; i < 3; ++i) p.push_back(hm::chain_prime(kAuxBits, logn, p));
    const i128 top = (i128)q / 2 << logn, m2 = (i128)p[0] * p[1];
    EncLimb lm = {};
    lm.q = q;
    lm.np = top <= m2 / 4 ? 2 : 3;
    lm.bits = bits;
    lm.t = bits > 32 ? bits - 33 : bits - 1;
    lm.mu = (u32)(((i128)1 << (bits + 31)) / q);
    lm.p_last = (u32)p[lm.np - 1];
    lm.nq_lo = (u32)(0 - q);
    lm.nq_hi = (u32)((0 - q) >> 32);
    u64 mi[3];
    for (int i = 0; i < lm.np; ++i) {
        mi[i] = 1;
        for (int j = 0; j < lm.np; ++j)
            if (j != i) mi[i] = hm::mulm(mi[i], p[j] % q, q);
        lm.ml[i] = (u32)mi[i];
        lm.mh[i] = (u32)(mi[i] >> 32);
    }
    lm.c0 = 2 * q - 32 - hm::mulm(5 * p[lm.np - 1] % q, mi[lm.np - 1], q);
    int bad = 0;
    for (int k = 0; k < 400; ++k) {
        const i128 r = (i128)(rng() >> 1) * (i128)(rng() >> 1) % top;
        const i128 x = k == 0 ? top : k == 1 ? -top : k == 2 ? 0 : k & 1 ? r : -r;
        u32 y[3] = {};
        for (int i = 0; i < lm.np; ++i) {
            u64 inv = 1;   // (M / p_i)^{-1} mod p_i
            for (int j = 0; j < lm.np; ++j)
                if (j != i) inv = inv * (p[j] % p[i]) % p[i];
            const i128 res = (x % (i128)p[i] + p[i]) % p[i];
            y[i] = (u32)((u64)res * hm::invm(inv, p[i]) % p[i] + (rng() & 1 ? p[i] : 0));
        }
        for (int e = -31; e <= 31; ++e) {
            const u32 eb = (u32)(e + 32);
            const u64 got = lm.np == 3 ? enc_crt<3, false>(lm, y[0], y[1], y[2], eb)
                          : bits > 32 ? enc_crt<2, false>(lm, y[0], y[1], 0, eb) : enc_crt<2, true>(lm, y[0], y[1], 0, eb);
            const i128 want = ((x + e) % (i128)q + q) % q;
            if (got != (u64)want) ++bad;
        }
    }
    return bad;
}
int main() { return (CHECKS) != 0; }
"""

ACCUMULATORS = r"""
#include "shim.h"
#include "host_math.h"
#include "ntt.cuh"
#include <random>
using namespace ichee;
static int check(u64 q)
{
    std::mt19937_64 rng(q);
    int bad = 0;
    u64 acc = 0, total = 0;
    for (int k = 0; k < 5000; ++k) {
        const u64 w = k % 3 ? rng() % q : q - 1, wp = host::shoup_of(w, q);
        const u64 x = k % 5 ? rng() % (8 * q) : 8 * q - 1;     // a transform's output, below 8 q
        const u64 p = shoup3(x, w, wp, q);
        acc = halve<8>(acc + p, q);
        total = (total + host::mulm(x % q, w, q)) % q;
        if (p >= 4 * q || acc >= 4 * q || acc % q != total) ++bad;
    }
    return bad;
}
int main() { return (CHECKS) != 0; }
"""


def test_reconstruction_with_noise(tmp_path):
    checks = []
    for ring in RINGS:
        qs, _ = moduli(ring)
        checks += ["check(%d, %dull, %d)" % (ring["log_n"], q, b) for q, b in zip(qs, ring["prime_bits"])]
    checks += ["check(10, %dull, 30)" % q for q in moduli(dict(log_n=10, prime_bits=[30], log2_scale=25, special_bits=61))[0]]
    run_on_host("kernels_enc", RECONSTRUCTION.replace("CHECKS", " + ".join(checks)), tmp_path)


def test_lazy_accumulators(tmp_path):
    primes = sorted({q for qs, special in map(moduli, RINGS) for q in qs + [special]})
    run_on_host("kernels_match", ACCUMULATORS.replace("CHECKS", " + ".join("check(%dull)" % q for q in primes)), tmp_path)
