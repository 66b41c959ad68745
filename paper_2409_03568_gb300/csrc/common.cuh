// common.cuh -- device-side building blocks of libichee: word-size modular arithmetic on
// residues below 2^61 (RNS limbs of the CKKS modulus Q, Sec. 2.2), Philox4x32-10 and the
// samplers of Sec. 2.2.1 / 2.2.2, and the launch-argument structures shared by the kernels.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace ichee {

typedef uint64_t u64;
typedef uint32_t u32;
typedef int64_t i64;

constexpr int kMaxPrimes = 8;          // ciphertext limbs
constexpr int kMaxModuli = kMaxPrimes + 1;  // plus the special prime P
constexpr int kMaxGaussBound = 31;

// --------------------------------------------------------------------------------------
// Modular arithmetic. Every modulus q is prime with q < 2^61, so 4q < 2^63 and the lazy
// ranges [0, 2q) and [0, 4q) of the NTT butterflies never overflow 64 bits.
// --------------------------------------------------------------------------------------

__device__ __forceinline__ u64 mulhi(u64 a, u64 b) { return __umul64hi(a, b); }

// Shoup product with a fixed multiplicand w < q and its companion wp = floor(w * 2^64 / q):
// returns x*w mod q in [0, 2q) for any 64-bit x.
__device__ __forceinline__ u64 shoup_lazy(u64 x, u64 w, u64 wp, u64 q)
{
    u64 hi = mulhi(x, wp);
    return x * w - hi * q;
}

// The same in [0, 4q) with three 32-bit products for the quotient instead of four: the low words'
// product and the fractions of the cross products are dropped, so the quotient is short by at most
// two.
__host__ __device__ __forceinline__ u64 shoup3(u64 x, u64 w, u64 wp, u64 q)
{
    const u32 xl = (u32)x, xh = (u32)(x >> 32), pl = (u32)wp, ph = (u32)(wp >> 32);
    const u64 hi = (u64)xh * ph + (((u64)xh * pl) >> 32) + (((u64)xl * ph) >> 32);
    return x * w - hi * q;
}

__device__ __forceinline__ u64 shoup(u64 x, u64 w, u64 wp, u64 q)
{
    u64 r = shoup_lazy(x, w, wp, q);
    return r >= q ? r - q : r;
}

__device__ __forceinline__ u64 csub(u64 x, u64 q) { return x >= q ? x - q : x; }

// The same for q <= 2^63 and x < q + 2^63: the sign of the difference decides (one comparison).
__device__ __forceinline__ u64 csub_s(u64 x, u64 q)
{
    const i64 d = (i64)(x - q);
    return d < 0 ? x : (u64)d;
}

__device__ __forceinline__ u64 add_mod(u64 a, u64 b, u64 q) { return csub(a + b, q); }

__device__ __forceinline__ u64 sub_mod(u64 a, u64 b, u64 q) { return a >= b ? a - b : a + q - b; }

// Barrett reduction of any 64-bit x with mu = floor(2^64 / q).
__device__ __forceinline__ u64 reduce64(u64 x, u64 q, u64 mu)
{
    u64 r = x - mulhi(x, mu) * q;
    return csub(r, q);
}

// Full product a*b mod q for a, b < q (Barrett on the 128-bit product with the 2-word
// constant m = floor(2^128 / q), m = m1*2^64 + m0).
__device__ __forceinline__ u64 mul_mod(u64 a, u64 b, u64 q, u64 m0, u64 m1)
{
    u64 lo = a * b;
    u64 hi = mulhi(a, b);
    // x = hi*2^64 + lo. Estimate floor(x*m / 2^128) from the partial products that reach
    // the 2^64 and 2^128 places, dropping lo*m0 / 2^128 (< 1).
    u64 p1 = lo * m1, p1h = mulhi(lo, m1);
    u64 p2 = hi * m0, p2h = mulhi(hi, m0);
    u64 mid = p1 + p2;
    u64 carry = (mid < p1) ? 1 : 0;
    u64 qhat = hi * m1 + p1h + p2h + carry;
    // qhat >= floor(x/q) - 3, so x - qhat*q is in [0, 4q) and fits 64 bits (4q < 2^63)
    u64 r = lo - qhat * q;
    r = csub(r, 2 * q);
    r = csub(r, q);
    return r;
}

// Montgomery product a*b*2^{-64} mod q, q odd, in two steps of 32 bits (Montgomery, Math. Comp. 44,
// 1985): adding m q with m = (t mod 2^32) (-q^{-1}) makes the low word of t vanish. The result is
// below a b / 2^64 + q: in [0, 2q) for a, b < 4q with q < 2^60, or for a, b < 62q with q < 2^50.
// qinv = -q^{-1} mod 2^64 (its low word is used). Callers fold the factor 2^64 into a constant
// applied later. Ten 32-bit products; with 64-bit words it took sixteen.
__host__ __device__ __forceinline__ u64 mont_lazy(u64 a, u64 b, u64 q, u64 qinv)
{
    const u32 a0 = (u32)a, a1 = (u32)(a >> 32), b0 = (u32)b, b1 = (u32)(b >> 32);
    const u32 q0 = (u32)q, q1 = (u32)(q >> 32), qi = (u32)qinv;
    const u64 p = (u64)a0 * b0;
    const u64 r = (u64)a0 * b1 + (p >> 32);
    const u64 s = (u64)a1 * b0 + (u32)r;
    const u64 u = (u64)a1 * b1 + (r >> 32) + (s >> 32);        // words 2 and 3 of a b; word 1 is s's low
    const u32 m = (u32)p * qi;
    const u64 v = (u64)m * q0 + (u32)p;
    const u64 w = (u64)m * q1 + (u32)s + (v >> 32);
    const u32 m2 = (u32)w * qi;
    const u64 v2 = (u64)m2 * q0 + (u32)w;
    return (u64)m2 * q1 + u + (w >> 32) + (v2 >> 32);
}

// --------------------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): key = per-call seed, counter =
// (block, stream, id lo, id hi). Every random draw of the library is a pure function of
// (seed, stream, ct id, coefficient), never of the launch shape.
// --------------------------------------------------------------------------------------

struct Words4 { u32 w[4]; };

__device__ __forceinline__ Words4 philox(u64 seed, u32 stream, u64 id, u32 block)
{
    u32 c0 = block, c1 = stream, c2 = (u32)id, c3 = (u32)(id >> 32);
    u32 k0 = (u32)seed, k1 = (u32)(seed >> 32);
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        if (round > 0) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
        const u64 p0 = (u64)0xD2511F53u * c0, p1 = (u64)0xCD9E8D57u * c2;   // one wide multiply each
        const u32 hi0 = (u32)(p0 >> 32), lo0 = (u32)p0, hi1 = (u32)(p1 >> 32), lo1 = (u32)p1;
        u32 n0 = hi1 ^ c1 ^ k0;
        u32 n2 = hi0 ^ c3 ^ k1;
        c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
    }
    Words4 r;
    r.w[0] = c0; r.w[1] = c1; r.w[2] = c2; r.w[3] = c3;
    return r;
}

// Streams (which draw of a ciphertext a Philox block belongs to).
enum Stream : u32 {
    kStreamV = 0, kStreamE0 = 1, kStreamE1 = 2, kStreamRadixBits = 3, kStreamPool = 4,
    kStreamKeyS = 8, kStreamKeyE = 9, kStreamKeyA = 16
};

// Uniform ternary from one 32-bit word: floor(3w / 2^32) - 1, by the two words where it steps.
__device__ __forceinline__ int ternary_of(u32 w) { return (w >= 0xAAAAAAABu ? 1 : 0) - (w < 0x55555556u ? 1 : 0); }

// Discrete Gaussian from one 64-bit value: top bit sign, magnitude = number of table
// entries the low 63 bits reach (table strictly increasing, last entry 2^63).
struct CdtTable { u64 t[kMaxGaussBound + 1]; u32 bound; };

__device__ __forceinline__ int gauss_of(u64 u, const CdtTable& cdt)
{
    u64 r = u & 0x7FFFFFFFFFFFFFFFull;
    int mag = 0;
    for (u32 k = 0; k < cdt.bound; ++k) mag += (r >= cdt.t[k]) ? 1 : 0;
    return (u >> 63) ? -mag : mag;
}

// The same magnitude by a branch-free binary search: t holds the table's first kCdtSearch
// entries, those from `bound` on replaced by 2^63 (which no 63-bit value reaches), in memory
// that lanes may index independently (shared memory). Five probes count the entries the value
// reaches instead of one comparison per entry.
constexpr int kCdtSearch = 31;
static_assert(kMaxGaussBound <= kCdtSearch, "a 31-entry search covers every table");

__device__ __forceinline__ int gauss_of_sorted(u64 u, const u64* t)
{
    const u64 r = u & 0x7FFFFFFFFFFFFFFFull;
    int pos = 0;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) pos += r >= t[pos + s - 1] ? s : 0;
    return (u >> 63) ? -pos : pos;
}

// Fill the search copy of the table (every thread of the block calls it).
__device__ __forceinline__ void cdt_for_search(const CdtTable& cdt, u64* t)
{
    for (int k = threadIdx.x; k < kCdtSearch; k += blockDim.x) t[k] = k < (int)cdt.bound ? cdt.t[k] : (1ull << 63);
}

// Residue of a small signed integer.
__device__ __forceinline__ u64 small_mod(int x, u64 q) { return x < 0 ? q - (u64)(-x) : (u64)x; }

// --------------------------------------------------------------------------------------
// Per-modulus constants and tables as the kernels see them.
// --------------------------------------------------------------------------------------

struct ModTables {
    const ulonglong2* tw;   // [N] (psi^{bitrev(k)}, Shoup companion): forward twiddles, bit-reversed order
    const ulonglong2* itw;  // [N] (psi^{-bitrev(k)}, Shoup companion): inverse twiddles
};

struct RnsArgs {
    int logn;
    int n_mod;                  // moduli described below
    u64 q[kMaxModuli];
    u64 mu[kMaxModuli];         // floor(2^64 / q)
    u64 m0[kMaxModuli], m1[kMaxModuli];  // floor(2^128 / q) as two words
    u64 qinv[kMaxModuli];       // -q^{-1} mod 2^64 (Montgomery)
    ModTables tab[kMaxModuli];
};

}  // namespace ichee
