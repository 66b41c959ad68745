// host_math.h -- host-side number theory for libichee's set-up: prime chain, roots of unity,
// twiddle tables with Shoup companions, the discrete-Gaussian table and CRT constants.
// Written for the CUDA library only (the CPU oracle has its own, separate code).
#pragma once
#include <cmath>
#include <cstdint>
#include <vector>

namespace ichee {
namespace host {

typedef unsigned __int128 u128;
typedef uint64_t u64;

inline u64 mulm(u64 a, u64 b, u64 m) { return (u64)((u128)a * b % m); }

// base^exp mod m for odd m below 2^63, by Montgomery products (a 128-bit division takes five times as
// long; finding a context's primes and roots takes some 10^4 products).
inline u64 powm(u64 base, u64 exp, u64 m)
{
    u64 inv = m;                          // m^{-1} mod 2^64, Newton
    for (int it = 0; it < 5; ++it) inv *= 2 - m * inv;
    auto mul = [&](u64 a, u64 b) {        // a b 2^{-64} mod m for a, b < m
        const u128 t = (u128)a * b;
        const u64 hi = (u64)(t >> 64), sub = (u64)((u128)((u64)t * inv) * m >> 64);
        return hi >= sub ? hi - sub : hi - sub + m;
    };
    const u64 one = (u64)(((u128)1 << 64) % m);
    u64 acc = one, b = mulm(base % m, one, m);
    for (; exp; exp >>= 1, b = mul(b, b))
        if (exp & 1) acc = mul(acc, b);
    return mul(acc, 1);
}

// a^{-1} mod p for a prime to p < 2^62 (extended Euclid: some 35 divisions; operations take several
// inverses per call, and a power by square and multiply took ten times as long).
inline u64 invm(u64 a, u64 p)
{
    u64 r0 = p, r1 = a % p;
    int64_t t0 = 0, t1 = 1;
    while (r1 != 0) {
        const u64 quo = r0 / r1, r2 = r0 - quo * r1;
        const int64_t t2 = t0 - (int64_t)quo * t1;
        r0 = r1;
        r1 = r2;
        t0 = t1;
        t1 = t2;
    }
    return t0 < 0 ? (u64)(t0 + (int64_t)p) : (u64)t0;
}

// Strong-probable-prime test to the first twelve prime bases (exact below 2^64).
inline bool is_prime64(u64 n)
{
    if (n < 2) return false;
    const u64 small[] = {2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31, 37};
    for (u64 p : small)
        if (n % p == 0) return n == p;
    u64 odd = n - 1;
    unsigned twos = 0;
    while (!(odd & 1)) { odd >>= 1; ++twos; }
    for (u64 a : small) {
        u64 x = powm(a, odd, n);
        bool witness = (x != 1 && x != n - 1);
        for (unsigned r = 1; witness && r < twos; ++r) {
            x = mulm(x, x, n);
            if (x == n - 1) witness = false;
        }
        if (witness) return false;
    }
    return true;
}

// Largest prime below 2^bits, congruent to 1 mod 2N, not in `taken`; 0 if none.
inline u64 chain_prime(unsigned bits, unsigned logn, const std::vector<u64>& taken)
{
    const u64 step = 2ull << logn;
    const u64 limit = 1ull << bits;
    u64 c = (limit - 1) - ((limit - 1) % step) + 1;
    if (c >= limit) c -= step;
    for (; c > (limit >> 1); c -= step) {
        bool used = false;
        for (u64 t : taken) used = used || (t == c);
        if (!used && is_prime64(c)) return c;
        if (c <= step) break;
    }
    return 0;
}

// A primitive 2N-th root of unity: psi = g^((q-1)/2N) for the first odd g >= 3 with
// psi^N = -1 (any such root gives the same negacyclic products).
inline u64 root_2n(u64 q, unsigned logn)
{
    const u64 n = 1ull << logn;
    for (u64 g = 3;; g += 2) {
        u64 psi = powm(g, (q - 1) / (2 * n), q);
        if (powm(psi, n, q) == q - 1) return psi;
    }
}

inline u64 shoup_of(u64 w, u64 q) { return (u64)(((u128)w << 64) / q); }

// Transform tables of q: N pairs (tw, companion) with tw[k] = psi^{bitrev(k)}, then N pairs of the inverse
// powers. Every doubling of the table is its first half times one power of psi. The companion
// floor(w 2^64 / q) comes from the reciprocal floor(2^128 / q), at most two too small; the inverse
// of psi^e is -psi^{N-e}, at the mirrored place of its doubling, and its companion the complement of that
// one's (w 2^64 / q is never whole). No division per entry: a context of four moduli at N = 2^13 is set
// up in 0.36 ms (2.1 with 128-bit divisions), of six at 2^14 in 0.73 (5.3).
inline void twiddle_pairs(u64 q, unsigned logn, u64* out)
{
    const u64 psi = root_2n(q, logn);
    const u128 recip = ~(u128)0 / q;
    const u64 r0 = (u64)recip, r1 = (u64)(recip >> 64);
    u64* inv = out + (2ull << logn);
    out[0] = inv[0] = 1;
    out[1] = inv[1] = r1;
    for (unsigned j = 0; j < logn; ++j) {
        const unsigned h = 1u << j;
        const u64 c = powm(psi, 1ull << (logn - 1 - j), q), cp = shoup_of(c, q);
        for (unsigned i = 0; i < h; ++i) {
            const u64 v = out[2 * i], y = v * c - (u64)((u128)v * cp >> 64) * q;   // below 2q
            const u64 w = y >= q ? y - q : y;
            u64 quo = w * r1 + (u64)((u128)w * r0 >> 64), rem = 0 - quo * q;
            for (; rem >= q; rem -= q) ++quo;
            const unsigned k = h + i, m = 2 * h - 1 - i;
            out[2 * k] = w;
            out[2 * k + 1] = quo;
            inv[2 * m] = q - w;
            inv[2 * m + 1] = ~quo;
        }
    }
}

// Cumulative table of the folded discrete Gaussian on [0, bound]: weight 1 at 0 and
// 2 exp(-k^2 / (2 sigma^2)) beyond; entry k = floor(2^63 * CDF(k)) for k < bound, the last
// entry 2^63. Long double, partial sums in increasing k.
inline void gauss_cdt(double sigma, unsigned bound, u64* out)
{
    const long double denom = 2.0L * (long double)sigma * (long double)sigma;
    long double total = 1.0L;
    for (unsigned k = 1; k <= bound; ++k) total += 2.0L * expl(-(long double)((u64)k * k) / denom);
    long double run = 1.0L;
    for (unsigned k = 0; k < bound; ++k) {
        if (k > 0) run += 2.0L * expl(-(long double)((u64)k * k) / denom);
        out[k] = (u64)floorl(ldexpl(run / total, 63));
    }
    out[bound] = 1ull << 63;
}

// Residue of a signed 64-bit integer.
inline u64 signed_mod(int64_t v, u64 q)
{
    if (v >= 0) return (u64)v % q;
    const u64 mag = (u64)(-(v + 1)) + 1;  // |v| without overflow
    const u64 r = mag % q;
    return r == 0 ? 0 : q - r;
}

// Low three words of a * b for a 3-word a.
inline void mul3(const u64 a[3], u64 b, u64 out[3])
{
    u128 c = 0;
    for (int i = 0; i < 3; ++i) {
        c += (u128)a[i] * b;
        out[i] = (u64)c;
        c >>= 64;
    }
}

}  // namespace host
}  // namespace ichee
