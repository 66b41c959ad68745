// ntt32.cuh -- block-wide negacyclic transforms modulo 28-bit auxiliary primes, for products of a
// small polynomial by a public-key polynomial (Sec. 2.2.2) computed over the integers: with v
// ternary and pk centered modulo q, every coefficient of v * pk is an integer below N q / 2 in
// magnitude, so its residues modulo two or three 28-bit primes determine it, and the residue
// modulo q follows exactly. A 28-bit butterfly takes 3 multiply instructions on 32-bit words
// (the 64-bit Shoup butterfly takes 10), and the transforms of v serve every limb.
//
// Same pass structure, layouts and barriers as ntt.cuh (N/E threads, E residues per thread and
// polynomial, radix-E passes, warp barriers where an exchange stays inside every warp). NP
// polynomials over one prime run in lockstep; a pair travels through shared memory as one 64-bit
// word, a single polynomial as 32-bit words with a swizzle of its own (conflict-free for every
// pass of N = 2^10 .. 2^14, as the 64-bit one; checked by the host-compiled layout test).
//
// Ranges: p < 2^28, so sixteen multiples of p fit a word and most butterflies need no reduction.
// The code knows every register's bound (a multiple of p) at compile time and folds a value below 2p
// only when the next sum would pass 16 p.
//
// z is a zero that the compiler does not know. A sum of two words may be issued as a multiply-add on the
// multiply pipe, which bounds these transforms; a sum of three takes the adder, half idle here. 4096
// fresh encryptions at N = 2^13 2.50 -> 2.43 ms (the inverse alone 2.48), at 2^14 7.72 -> 7.53, at 2^12
// 1.22 -> 1.21; the same in the reconstruction modulo q was slower (2.49), and the 64-bit transforms
// gain nothing from it.
#pragma once
#include "internal.h"
#include "ntt.cuh"

namespace ichee {


// x * w mod p in [0, 2p) for any 32-bit x; wp = floor(w 2^32 / p).
__device__ __forceinline__ u32 shoup32(u32 x, u32 w, u32 wp, u32 p) { return x * w - __umulhi(x, wp) * p; }

// x * w * 2^-32 mod p in (0, 2p) for any 32-bit x and w < p (Montgomery); pinv = p^-1 mod 2^32.
__device__ __forceinline__ u32 mont32(u32 x, u32 w, u32 p, u32 pinv)
{
    const u64 t = (u64)x * w;
    return (u32)(t >> 32) - __umulhi((u32)t * pinv, p) + p;
}

// x below B p to below 2p, congruent: x - 2p if that is no underflow (one fused add-and-minimum) up to
// 4p, else by the top bits, x - floor(x / 2^28) p < 2^28 + 15 (2^28 - p) < 2p.
template <int B>
__device__ __forceinline__ u32 fold32(u32 x, u32 p, u32 neg_p2)
{
    if constexpr (B > 4) return x - (x >> kAuxBits) * p;
    else if constexpr (B > 2) return __viaddmin_u32(x, neg_p2, x);
    else return x;
}

// The 2^k twiddles of one butterfly group in stage s of a pass, entries 2^s + (h << k) + b: pairs of
// neighbours in one 16-byte load.
template <int K, int ST>
__device__ __forceinline__ void twiddles32(const uint2* __restrict__ t, int h, uint2 (&w)[1 << K])
{
    const char* at = reinterpret_cast<const char*>(t) + ((u32)h << (K + 3));
    if constexpr (K == 0) {
        w[0] = __ldg(reinterpret_cast<const uint2*>(at) + (1 << ST));
    } else {
#pragma unroll
        for (int b = 0; b < (1 << K); b += 2) {
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(at) + ((1 << ST) + b) / 2);
            w[b] = make_uint2(v.x, v.y);
            w[b + 1] = make_uint2(v.z, v.w);
        }
    }
}

// Swizzle of 32-bit words: 32 lanes of every pass layout touch 32 banks.
template <int E>
__host__ __device__ constexpr int swz32(int x)
{
    if constexpr (E == 16) return x ^ ((x >> 5) & 15) ^ ((x >> 4) & 30);
    else return x ^ ((x >> 5) & 7) ^ ((x >> 3) & 28) ^ ((x >> 6) & 2);
}

// Stores / loads of an exchange; `sm` holds N words of 4 * NP bytes.
template <int LOGN, int S0, int NP, int E>
__device__ __forceinline__ void store_sm32(u32* sm, const u32 (&r)[NP][E], int tid)
{
    if constexpr (NP == 2) {
        const int base = slot_base<LOGN, S0, E>(tid);
#pragma unroll
        for (int e = 0; e < E; ++e)
            reinterpret_cast<uint2*>(sm)[slot_of<LOGN, S0, E>(base, e)] = make_uint2(r[0][e], r[1][e]);
    } else {
        const int base = swz32<E>(elem_index<LOGN, S0, E>(tid, 0));
#pragma unroll
        for (int e = 0; e < E; ++e) sm[base ^ swz32<E>(elem_index<LOGN, S0, E>(0, e))] = r[0][e];
    }
}

template <int LOGN, int S0, int NP, int E>
__device__ __forceinline__ void load_sm32(const u32* sm, u32 (&r)[NP][E], int tid)
{
    if constexpr (NP == 2) {
        const int base = slot_base<LOGN, S0, E>(tid);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint2 v = reinterpret_cast<const uint2*>(sm)[slot_of<LOGN, S0, E>(base, e)];
            r[0][e] = v.x;
            r[1][e] = v.y;
        }
    } else {
        const int base = swz32<E>(elem_index<LOGN, S0, E>(tid, 0));
#pragma unroll
        for (int e = 0; e < E; ++e) r[0][e] = sm[base ^ swz32<E>(elem_index<LOGN, S0, E>(0, e))];
    }
}

// ---- forward ------------------------------------------------------------------------------
// Bound (in multiples of p) after S forward stages that start from bound b: a stage adds 2, and
// folds its first operands to 2 when the sum would pass 16.
__host__ __device__ constexpr int fwd32_bound(int b, int S)
{
    for (int k = 0; k < S; ++k) b = (b + 2 > 16 ? 2 : b) + 2;
    return b;
}

// Forward stages S0 .. S0+S-1 on registers below B p. With TERNARY0 the registers of pass 0 hold
// the integers -1, 0, 1 (as signed words).
template <int LOGN, int S0, int NP, int E, int B, bool TERNARY0>
__device__ __forceinline__ void fwd32_regs(u32 (&r)[NP][E], int tid, const uint2* __restrict__ tw, u32 p, u32 z)
{
    using P = Pass<LOGN, S0, E>;
    const u32 p2 = p + p;
    static_for<P::G>([&](auto gc) {
        constexpr int g = decltype(gc)::v;
        const int h = pass_gid(P::T, P::G, tid, g) >> P::LO;
        static_for<P::S>([&](auto kc) {
            constexpr int k = decltype(kc)::v, half = 1 << (P::S - 1 - k);
            constexpr bool ternary = TERNARY0 && S0 == 0 && k == 0;
            constexpr int bound = fwd32_bound(B, k);
            uint2 w[1 << k];
            twiddles32<k, S0 + k>(tw, h, w);
            static_for<P::R / P::G / 2>([&](auto jc) {
                constexpr int j = decltype(jc)::v, b = j / half, i0 = g * (1 << P::S) + b * 2 * half + j % half, i1 = i0 + half;
#pragma unroll
                for (int n = 0; n < NP; ++n) {
                    u32 X = r[n][i0];
                    if constexpr (!ternary && bound + 2 > 16) X = fold32<bound>(X, p, 0u - p2);
                    // ternary: the product is the signed integer 0 or +-w, and the sums with
                    // 2p lie in (0, 4p)
                    const u32 T = ternary ? r[n][i1] * w[b].x : shoup32(r[n][i1], w[b].x, w[b].y, p);
                    r[n][i0] = ternary ? X + T + p2 : X + T + z;
                    r[n][i1] = X - T + p2;
                }
            });
        });
    });
}

template <int LOGN, int S0, int NP, int E, int B>
__device__ __forceinline__ void fwd32_rest(u32* sm, u32 (&r)[NP][E], int tid, const uint2* __restrict__ tw, u32 p, u32 z)
{
    constexpr int LE = Radix<E>::LE;
    if constexpr (S0 <= NttShape<LOGN, E>::LAST) {
        store_sm32<LOGN, S0 - LE, NP, E>(sm, r, tid);
        exchange_barrier<LOGN, S0, E>();
        load_sm32<LOGN, S0, NP, E>(sm, r, tid);
        fwd32_regs<LOGN, S0, NP, E, B, false>(r, tid, tw, p, z);
        fwd32_rest<LOGN, S0 + LE, NP, E, fwd32_bound(B, Pass<LOGN, S0, E>::S)>(sm, r, tid, tw, p, z);
    }
}

// Bound of a forward transform's outputs.
template <int LOGN, int E, bool TERNARY0>
__host__ __device__ constexpr int fwd32_out()
{
    return TERNARY0 ? fwd32_bound(4, LOGN - 1) : fwd32_bound(1, LOGN);
}

// Whole forward transform: input in the layout of pass 0 (ternary integers with TERNARY0, else
// residues below p), output in the layout of the last pass, bit-reversed order, below 16 p.
template <int LOGN, int NP, int E, bool TERNARY0>
__device__ __forceinline__ void ntt32_fwd(u32* sm, u32 (&r)[NP][E], int tid, const uint2* __restrict__ tw, u32 p, u32 z)
{
    constexpr int LE = Radix<E>::LE;
    // bound entering pass 0: the ternary stage leaves 4, as a stage from 2 would
    constexpr int B0 = TERNARY0 ? 2 : 1;
    fwd32_regs<LOGN, 0, NP, E, B0, TERNARY0>(r, tid, tw, p, z);
    fwd32_rest<LOGN, LE, NP, E, fwd32_bound(B0, LE)>(sm, r, tid, tw, p, z);
}

// ---- inverse ------------------------------------------------------------------------------
// A stage takes X and Y, both below b p, to X + Y (below 2b p) and a product below 2p; both are folded
// below 2p first when b is 16. Bound of register i before step t of a pass that starts from B (i's
// partner, which differs in bit t, has the same): the sums since its last product, bit t-1 down.
__host__ __device__ constexpr int inv32_before(int B, int t, int i)
{
    int b = B;
    for (int u = 0; u < t; ++u) b = ((i >> u) & 1) ? 2 : (b == 16 ? 4 : 2 * b);
    return b;
}

// Largest bound after S steps from b.
__host__ __device__ constexpr int inv32_bound(int b, int S)
{
    int m = 2;
    for (int i = 0; i < (1 << S); ++i) m = inv32_before(b, S, i) > m ? inv32_before(b, S, i) : m;
    return m;
}

// Inverse stages S0+S-1 .. S0 on registers below B p; the outputs of pass 0 are folded below 2p.
template <int LOGN, int S0, int NP, int E, int B>
__device__ __forceinline__ void inv32_regs(u32 (&r)[NP][E], int tid, const uint2* __restrict__ itw, u32 p, u32 z)
{
    using P = Pass<LOGN, S0, E>;
    const u32 p2 = p + p, neg_p2 = 0u - p2;
    static_for<P::G>([&](auto gc) {
        constexpr int g = decltype(gc)::v;
        const int h = pass_gid(P::T, P::G, tid, g) >> P::LO;
        static_for<P::S>([&](auto tc) {
            constexpr int t = decltype(tc)::v, k = P::S - 1 - t, half = 1 << t;
            uint2 w[1 << k];
            twiddles32<k, S0 + k>(itw, h, w);
            static_for<P::R / P::G / 2>([&](auto jc) {
                constexpr int j = decltype(jc)::v, b = j / half, j0 = b * 2 * half + j % half;
                constexpr int i0 = g * (1 << P::S) + j0, i1 = i0 + half;
                constexpr int bound = inv32_before(B, t, j0), kept = bound == 16 ? 2 : bound;
                const u32 add = kept == 8 ? p2 << 2 : kept == 4 ? p2 << 1 : p2;   // a multiple of p, at least Y
#pragma unroll
                for (int n = 0; n < NP; ++n) {
                    u32 X = r[n][i0], Y = r[n][i1];
                    if constexpr (bound == 16) {
                        X = fold32<bound>(X, p, neg_p2);
                        Y = fold32<bound>(Y, p, neg_p2);
                    }
                    r[n][i0] = X + Y + z;
                    r[n][i1] = shoup32(X - Y + add, w[b].x, w[b].y, p);
                }
            });
        });
    });
    if constexpr (S0 == 0)
        static_for<E>([&](auto ec) {
            constexpr int e = decltype(ec)::v;
#pragma unroll
            for (int n = 0; n < NP; ++n) r[n][e] = fold32<inv32_before(B, P::S, e % (1 << P::S))>(r[n][e], p, neg_p2);
        });
}

template <int LOGN, int S0, int NP, int E, int B>
__device__ __forceinline__ void inv32_rest(u32* sm, u32 (&r)[NP][E], int tid, const uint2* __restrict__ itw, u32 p, u32 z)
{
    constexpr int LE = Radix<E>::LE;
    inv32_regs<LOGN, S0, NP, E, B>(r, tid, itw, p, z);
    if constexpr (S0 > 0) {
        store_sm32<LOGN, S0, NP, E>(sm, r, tid);
        exchange_barrier<LOGN, S0, E>();
        load_sm32<LOGN, S0 - LE, NP, E>(sm, r, tid);
        inv32_rest<LOGN, S0 - LE, NP, E, inv32_bound(B, Pass<LOGN, S0, E>::S)>(sm, r, tid, itw, p, z);
    }
}

// Whole inverse transform (without 1/N): input in the layout of the last pass, below 2p; output
// in the layout of pass 0, natural order, below 2p.
template <int LOGN, int NP, int E>
__device__ __forceinline__ void ntt32_inv(u32* sm, u32 (&r)[NP][E], int tid, const uint2* __restrict__ itw, u32 p, u32 z)
{
    inv32_rest<LOGN, NttShape<LOGN, E>::LAST, NP, E, 2>(sm, r, tid, itw, p, z);
}

}  // namespace ichee
