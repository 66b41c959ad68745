// ntt.cuh -- block-wide negacyclic NTT / inverse NTT over one RNS limb, for the products in
// R_q = Z_q[X]/(X^N + 1) that CKKS encryption, key generation and ct x ct multiplication
// need (Sec. 2.2, 2.2.2, 2.2.3).
//
// Layout: N = 2^LOGN residues, one thread block of N/E threads, every thread holding E
// residues (E = 16 or 8) in registers. The log2(N) butterfly stages run in
// passes of up to log2(E) stages (a radix-E step entirely in registers); between passes the
// block exchanges data through one shared-memory buffer of N words,
// XOR-swizzled so that every pass reads and writes without bank conflicts (the host-compiled
// layout test checks every pass of N = 2^10 .. 2^14): x ^ ((x >> 4) & 15) for E = 16,
// x ^ ((x >> 2) & 7) ^ ((x >> 3) & 15) for E = 8. E = 8 halves the registers a polynomial
// takes, so twice the threads fit on an SM, at the price of one more exchange per transform.
// An exchange whose two layouts give every warp the same residues takes a warp barrier
// instead of a block barrier (the later passes of a transform).
//
// Between transforms on the same buffer: a forward transform's first exchange stores to its
// thread's pass-0 slots and its last exchange loads the thread's last-pass slots; an inverse
// does the reverse. So a forward after an inverse (or an inverse after a forward) overwrites
// only slots its own thread loaded last and needs no block barrier before it; two transforms
// of the same direction in a row do.
//
// Forward: Cooley-Tukey with the negacyclic twist merged into the twiddles, natural-order
// input, bit-reversed output. Inverse: Gentleman-Sande, bit-reversed input, natural-order output,
// without the 1/N factor (callers fold 1/N into a constant operand).
// Ranges: a product by a twiddle is left in [0, 4q) (shoup3), and CAP multiples of q fit a word:
// CAP = 16 for ciphertext primes (below 2^60), 8 where the modulus may be the special prime (below
// 2^61), kNoFold for moduli below 2^50, whose values never need one. Every register's bound is
// known at compile time, and a conditional subtraction is spent only where the next sum would
// pass CAP q: with CAP = 16 on 5 of the 13 stages at N = 2^13 instead of on every butterfly
// (Harvey's [0, 4q)). Register-only butterflies: 887 G/s with the exact quotient and a subtraction
// each, 1005 without the subtraction, 1132 with the three-product quotient as well.
// Twiddles: tw[k] = psi^{bitrev(k)}, itw[k] = psi^{-bitrev(k)}, psi a primitive 2N-th root,
// each stored next to its Shoup companion (one 16-byte load per twiddle).
#pragma once
#include "common.cuh"

namespace ichee {

template <int E>
struct Radix {
    static_assert(E == 8 || E == 16, "8 or 16 residues per thread");
    static constexpr int LE = E == 16 ? 4 : 3;   // stages of a full pass
};

template <int E = 16>
__host__ __device__ constexpr int swz(int x)
{
    if constexpr (E == 16) return x ^ ((x >> 4) & 15);
    else return x ^ ((x >> 2) & 7) ^ ((x >> 3) & 15);
}

template <int LOGN, int S0, int E = 16>
struct Pass {
    static constexpr int LE = Radix<E>::LE;
    static constexpr int R = E;                                      // residues per thread
    static constexpr int N = 1 << LOGN;
    static constexpr int T = N / E;
    static constexpr int S = (LOGN - S0) < LE ? (LOGN - S0) : LE;  // stages in this pass
    static constexpr int G = E >> S;                                 // groups per thread
    static constexpr int LO = LOGN - S0 - S;                         // lowest varying index bit
};

template <int LOGN, int E = 16>
struct NttShape {
    static constexpr int LE = Radix<E>::LE;
    static constexpr int N = 1 << LOGN;
    static constexpr int T = N / E;
    static constexpr int LAST = ((LOGN - 1) / LE) * LE;  // first stage of the last pass
};

__host__ __device__ constexpr int ilog2(int x) { return x > 1 ? 1 + ilog2(x >> 1) : 0; }

// Butterfly-group id of register group g of thread tid in a pass: a full pass has one group
// per thread; a partial last pass (fewer than LE stages, G > 1 groups per thread) keeps a
// warp's G x 32 groups adjacent (lane fastest, then g, then the warp), so that each warp holds
// the same 2^(LE+5) consecutive indices as in the full pass before it -- the exchange into the
// last pass stays inside the warp -- while a register's 32 lanes still touch consecutive
// butterflies (the coalescing and the bank pattern of global and shared accesses unchanged).
__host__ __device__ constexpr int pass_gid(int T, int G, int tid, int g, bool wt = true)
{
    return G > 1 && wt ? (((tid >> 5) << (5 + ilog2(G))) | (g << 5) | (tid & 31)) : g * T + tid;
}

// Natural index of register e of thread tid in the pass starting at stage S0 (values of the
// template parameters as arguments, for the compile-time checks below). WT = false keeps the
// groups of a partial last pass strided by the thread count (g * T + tid): the layout of the
// compact transform form.
__host__ __device__ constexpr int elem_index_of(int logn, int s0, int E, int tid, int e, bool wt = true)
{
    const int le = E == 16 ? 4 : 3;
    const int T = (1 << logn) / E;
    const int S = (logn - s0) < le ? (logn - s0) : le;
    const int G = E >> S, LO = logn - s0 - S;
    const int g = e >> S, j = e & ((1 << S) - 1);
    const int gid = pass_gid(T, G, tid, g, wt);
    return ((gid >> LO) << (LO + S)) | (j << LO) | (gid & ((1 << LO) - 1));
}

template <int LOGN, int S0, int E = 16, bool WT = true>
__device__ __forceinline__ int elem_index(int tid, int e) { return elem_index_of(LOGN, S0, E, tid, e, WT); }

// Whether the exchange between the layouts of the passes starting at SA and SB stays inside
// every warp: both layouts are bit permutations of (tid, e), so it does when the index bits
// driven by a warp's lane bits and the register bits are the same set in both, and every
// higher thread bit lands on the same index bit in both. Such an exchange needs only a warp
// barrier: a thread stores to the slots it loaded in the exchange before (the same layout),
// so no other warp's loads can be overtaken.
__host__ __device__ constexpr bool exchange_in_warp(int logn, int sa, int sb, int E)
{
    const int T = (1 << logn) / E;
    int va = 0, vb = 0;
    for (int i = 0; i < 5; ++i) {
        va |= elem_index_of(logn, sa, E, 1 << i, 0);
        vb |= elem_index_of(logn, sb, E, 1 << i, 0);
    }
    for (int k = 1; k < E; k <<= 1) {
        va |= elem_index_of(logn, sa, E, 0, k);
        vb |= elem_index_of(logn, sb, E, 0, k);
    }
    if (va != vb) return false;
    for (int i = 5; (1 << i) < T; ++i)
        if (elem_index_of(logn, sa, E, 1 << i, 0) != elem_index_of(logn, sb, E, 1 << i, 0)) return false;
    return true;
}

// Bit p set: the exchange between full passes p - 1 and p stays inside every warp (full passes
// have the same layout in both forms of the transform; the exchange is the same in the inverse
// direction).
__host__ __device__ constexpr unsigned full_exchanges_in_warp(int logn, int E)
{
    const int le = E == 16 ? 4 : 3;
    unsigned m = 0;
    for (int p = 1; p < logn / le; ++p)
        if (exchange_in_warp(logn, le * (p - 1), le * p, E)) m |= 1u << p;
    return m;
}

// An exchange that leaves the warp need not be a barrier of the block: only warps whose numbers
// differ in bits that the exchange moves trade data. Mask of the warp-number bits (thread bits from 5
// up) that stay on the same index bit in both layouts, at most the three highest. The groups drift
// apart, so that one computes while another exchanges: matching at N = 2^13 2.31 -> 2.27 ms, at 2^14
// 6.60 -> 6.44 ms.
__host__ __device__ constexpr int exchange_fixed_bits(int logn, int sa, int sb, int E)
{
    const int T = (1 << logn) / E;
    int fixed = 0, count = 0;
    for (int i = ilog2(T) - 1; i >= 5 && count < 3; --i)
        if (elem_index_of(logn, sa, E, 1 << i, 0) == elem_index_of(logn, sb, E, 1 << i, 0)) {
            fixed |= 1 << (i - 5);
            ++count;
        }
    return fixed;
}

__host__ __device__ constexpr int bits_of(int m) { return m ? (m & 1) + bits_of(m >> 1) : 0; }

// First named barrier of the exchange into the pass at s (barrier 0 is the block's): the exchanges of
// a transform that need one take consecutive numbers, one per group of warps.
__host__ __device__ constexpr int exchange_first_id(int logn, int s, int E)
{
    const int le = E == 16 ? 4 : 3;
    int id = 1;
    for (int p = le; p < s; p += le)
        if (!exchange_in_warp(logn, p - le, p, E) && exchange_fixed_bits(logn, p - le, p, E))
            id += 1 << bits_of(exchange_fixed_bits(logn, p - le, p, E));
    return id;
}

// The barrier of the exchange between the pass at S - LE and the pass at S (either direction).
template <int LOGN, int S, int E>
__device__ __forceinline__ void exchange_barrier()
{
    constexpr int LE = Radix<E>::LE, T = NttShape<LOGN, E>::T;
    constexpr int fixed = exchange_fixed_bits(LOGN, S - LE, S, E);
    if constexpr (exchange_in_warp(LOGN, S - LE, S, E)) {
        __syncwarp();
    } else if constexpr (fixed == 0) {
        __syncthreads();
    } else {
        constexpr int first = exchange_first_id(LOGN, S, E), groups = 1 << bits_of(fixed);
        static_assert(first + groups <= 16, "sixteen named barriers");
        const int warp = threadIdx.x >> 5;
        int group = 0, bit = 0;
#pragma unroll
        for (int i = 0; i < 5; ++i)
            if ((fixed >> i) & 1) group |= ((warp >> i) & 1) << bit++;
        asm volatile("bar.sync %0, %1;" ::"r"(first + group), "n"(T / groups) : "memory");
    }
}

// Without the swizzle the split is additive: elem_index(tid, e) = elem_index(tid, 0) +
// elem_index(0, e) (disjoint bits), so global accesses take a per-thread base pointer and
// compile-time offsets.
template <int LOGN, int S0, int E = 16, bool WT = true>
__device__ __forceinline__ int elem_offset(int e) { return elem_index<LOGN, S0, E, WT>(0, e); }

// Shared-memory slot of register e of thread tid in the pass starting at S0. elem_index is a
// permutation of the bits of (tid, e) and the swizzle is linear over GF(2), so the slot is
// swz(elem_index(tid, 0)) ^ swz(elem_index(0, e)): a per-thread base XOR a compile-time
// constant, one instruction per access (checked for every pass of N = 2^10 .. 2^14).
template <int LOGN, int S0, int E = 16, bool WT = true>
__device__ __forceinline__ int slot_base(int tid) { return swz<E>(elem_index<LOGN, S0, E, WT>(tid, 0)); }

template <int LOGN, int S0, int E = 16, bool WT = true>
__device__ __forceinline__ int slot_of(int base, int e) { return base ^ swz<E>(elem_index<LOGN, S0, E, WT>(0, e)); }

template <int LOGN, int S0, int E = 16, bool WT = true>
__device__ __forceinline__ void load_sm(const u64* sm, u64 (&r)[E], int tid)
{
    const int base = slot_base<LOGN, S0, E, WT>(tid);
#pragma unroll
    for (int e = 0; e < E; ++e) r[e] = sm[slot_of<LOGN, S0, E, WT>(base, e)];
}

template <int LOGN, int S0, int E = 16, bool WT = true>
__device__ __forceinline__ void store_sm(u64* sm, const u64 (&r)[E], int tid)
{
    const int base = slot_base<LOGN, S0, E, WT>(tid);
#pragma unroll
    for (int e = 0; e < E; ++e) sm[slot_of<LOGN, S0, E, WT>(base, e)] = r[e];
}

// f(Index<0>()), ..., f(Index<N - 1>()): a loop whose index is a compile-time constant.
template <int I>
struct Index {
    static constexpr int v = I;
};

template <int N, int I = 0, class F>
__device__ __forceinline__ void static_for(F&& f)
{
    if constexpr (I < N) {
        f(Index<I>());
        static_for<N, I + 1>(f);
    }
}

constexpr int kNoFold = 1 << 12;   // CAP of moduli below 2^50

// x below CAP q to below CAP/2 q: one conditional subtraction.
template <int CAP>
__device__ __forceinline__ u64 halve(u64 x, u64 q) { return csub_s(x, (CAP / 2) * q); }

// x below B q (B at most 16) to below 4q.
template <int B>
__device__ __forceinline__ u64 below4(u64 x, u64 q)
{
    static_assert(B <= 16, "one subtraction of 8q and one of 4q");
    if constexpr (B > 8) x = csub_s(x, 8 * q);
    if constexpr (B > 4) x = csub_s(x, 4 * q);
    return x;
}

// x below B q to [0, q).
template <int B>
__device__ __forceinline__ u64 below1(u64 x, u64 q) { return csub_s(csub_s(below4<B>(x, q), 2 * q), q); }

// Bound after S forward stages from b: a stage adds 4, its first operands halved below CAP/2 when the
// sum would pass CAP.
__host__ __device__ constexpr int fwd_bound(int cap, int b, int S)
{
    for (int k = 0; k < S; ++k) b = (b + 4 > cap ? cap / 2 : b) + 4;
    return b;
}

// Forward stages S0 .. S0+S-1 on registers below B q. Stage s pairs x with x + N/2^{s+1} and uses
// twiddle index root 2^s + (x >> (LOGN - s)): root = 1 for a whole transform; for part h of the 2^r
// equal parts that the first r stages of a longer transform leave, root = 2^r + h and the longer
// transform's table.
template <int LOGN, int S0, int E, bool WT, int CAP, int B, int NP>
__device__ __forceinline__ void fwd_regs(u64 (&r)[NP][E], int tid, const ulonglong2* __restrict__ tw, u64 q, int root)
{
    using P = Pass<LOGN, S0, E>;
    static_for<P::G>([&](auto gc) {
        constexpr int g = decltype(gc)::v;
        const int h = pass_gid(P::T, P::G, tid, g, WT) >> P::LO;
        static_for<P::S>([&](auto kc) {
            constexpr int k = decltype(kc)::v, s = S0 + k, half = 1 << (P::S - 1 - k);
            constexpr bool fold = fwd_bound(CAP, B, k) + 4 > CAP;
            static_for<(1 << k)>([&](auto bc) {
                constexpr int b = decltype(bc)::v;
                const ulonglong2 w = __ldg(tw + (root << s) + (h << k) + b);
#pragma unroll
                for (int jj = b * 2 * half; jj < b * 2 * half + half; ++jj) {
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        const int i0 = g * (1 << P::S) + jj, i1 = i0 + half;
                        const u64 X = fold ? halve<CAP>(r[p][i0], q) : r[p][i0];
                        const u64 T = shoup3(r[p][i1], w.x, w.y, q);
                        r[p][i0] = X + T;
                        r[p][i1] = X - T + 4 * q;
                    }
                }
            });
        });
    });
}

// A stage takes X and Y, both below b q, to X + Y -- halved when it would pass CAP/2 -- and a product
// in [0, 4q). Bound of register i before step t of an inverse pass that starts from B: the sums since
// its last product.
__host__ __device__ constexpr int inv_before(int cap, int B, int t, int i)
{
    int b = B;
    for (int u = 0; u < t; ++u) b = ((i >> u) & 1) ? 4 : (2 * b > cap / 2 ? cap / 2 : 2 * b);
    return b;
}

__host__ __device__ constexpr int inv_bound(int cap, int b, int S)
{
    int m = 4;
    for (int i = 0; i < (1 << S); ++i) m = inv_before(cap, b, S, i) > m ? inv_before(cap, b, S, i) : m;
    return m;
}

// Inverse stages S0+S-1 .. S0 (reverse order) on registers below B q (B <= CAP/2).
template <int LOGN, int S0, int E, bool WT, int CAP, int B>
__device__ __forceinline__ void inv_regs(u64 (&r)[E], int tid, const ulonglong2* __restrict__ itw, u64 q, int root)
{
    using P = Pass<LOGN, S0, E>;
    static_for<P::G>([&](auto gc) {
        constexpr int g = decltype(gc)::v;
        const int h = pass_gid(P::T, P::G, tid, g, WT) >> P::LO;
        static_for<P::S>([&](auto tc) {
            constexpr int t = decltype(tc)::v, k = P::S - 1 - t, s = S0 + k, half = 1 << t;
            static_for<(1 << k)>([&](auto bc) {
                constexpr int b = decltype(bc)::v;
                const ulonglong2 w = __ldg(itw + (root << s) + (h << k) + b);
                static_for<half>([&](auto jc) {
                    constexpr int j0 = b * 2 * half + decltype(jc)::v;
                    constexpr int i0 = g * (1 << P::S) + j0, i1 = i0 + half;
                    constexpr int bound = inv_before(CAP, B, t, j0);
                    const u64 X = r[i0], Y = r[i1];
                    r[i0] = 2 * bound > CAP / 2 ? halve<CAP>(X + Y, q) : X + Y;
                    r[i1] = shoup3(X - Y + bound * q, w.x, w.y, q);
                });
            });
        });
    });
}

// Forward passes after the first: on entry r holds the output of pass S0-LE (its layout), on
// exit the output of the last pass in the last pass's layout. Polynomial p exchanges through
// sm + p N; the polynomials share the barriers.
template <int LOGN, int S0, int E, int CAP, int B, int NP>
__device__ __forceinline__ void fwd_rest(u64* sm, u64 (&r)[NP][E], int tid, const ulonglong2* __restrict__ tw, u64 q, int root)
{
    constexpr int LE = Radix<E>::LE;
    if constexpr (S0 <= NttShape<LOGN, E>::LAST) {
#pragma unroll
        for (int p = 0; p < NP; ++p) store_sm<LOGN, S0 - LE, E>(sm + (p << LOGN), r[p], tid);
        exchange_barrier<LOGN, S0, E>();
#pragma unroll
        for (int p = 0; p < NP; ++p) load_sm<LOGN, S0, E>(sm + (p << LOGN), r[p], tid);
        fwd_regs<LOGN, S0, E, true, CAP, B>(r, tid, tw, q, root);
        fwd_rest<LOGN, S0 + LE, E, CAP, fwd_bound(CAP, B, Pass<LOGN, S0, E>::S)>(sm, r, tid, tw, q, root);
    }
}

// NP whole forward transforms, every pass unrolled.
template <int LOGN, int E, int CAP, int B, int NP>
__device__ __forceinline__ void ntt_fwd_polys(u64* sm, u64 (&r)[NP][E], int tid, const ModTables& t, u64 q, int root = 1)
{
    constexpr int LE = Radix<E>::LE;
    fwd_regs<LOGN, 0, E, true, CAP, B>(r, tid, t.tw, q, root);
    fwd_rest<LOGN, LE, E, CAP, fwd_bound(CAP, B, Pass<LOGN, 0, E>::S)>(sm, r, tid, t.tw, q, root);
}

// Inverse passes S0, S0-LE, ..., 0: on entry r holds bit-reversed data in the layout of pass
// S0 (no inverse stage applied yet), on exit natural-order data in the layout of pass 0.
template <int LOGN, int S0, int E, int CAP, int B>
__device__ __forceinline__ void inv_rest(u64* sm, u64 (&r)[E], int tid, const ulonglong2* __restrict__ itw, u64 q, int root)
{
    constexpr int LE = Radix<E>::LE;
    inv_regs<LOGN, S0, E, true, CAP, B>(r, tid, itw, q, root);
    if constexpr (S0 > 0) {
        store_sm<LOGN, S0, E>(sm, r, tid);
        exchange_barrier<LOGN, S0, E>();
        load_sm<LOGN, S0 - LE, E>(sm, r, tid);
        inv_rest<LOGN, S0 - LE, E, CAP, inv_bound(CAP, B, Pass<LOGN, S0, E>::S)>(sm, r, tid, itw, q, root);
    }
}

// The first LS stages of a forward transform on the R = 2^LS coefficients i + j N/R of one i (r[j] below
// q on entry, below fwd_bound(CAP, 1, LS) q on exit), and the last LS of an inverse one (below 4q on
// entry, below CAP/2 q on exit): what couples the R parts of a transform split over blocks.
template <int LS, int CAP>
__device__ __forceinline__ void fwd_head(u64 (&r)[1 << LS], const ulonglong2* __restrict__ tw, u64 q)
{
    static_for<LS>([&](auto kc) {
        constexpr int k = decltype(kc)::v, half = 1 << (LS - 1 - k);
        constexpr bool fold = fwd_bound(CAP, 1, k) + 4 > CAP;
#pragma unroll
        for (int i = 0; i < 1 << LS; ++i) {
            if (i & half) continue;
            const ulonglong2 w = __ldg(tw + (1 << k) + i / (2 * half));
            const u64 X = fold ? halve<CAP>(r[i], q) : r[i];
            const u64 T = shoup3(r[i + half], w.x, w.y, q);
            r[i] = X + T;
            r[i + half] = X - T + 4 * q;
        }
    });
}

template <int LS, int CAP>
__device__ __forceinline__ void inv_tail(u64 (&r)[1 << LS], const ulonglong2* __restrict__ itw, u64 q)
{
    static_for<LS>([&](auto tc) {
        constexpr int t = decltype(tc)::v, k = LS - 1 - t, half = 1 << t;
        static_for<(1 << LS)>([&](auto ic) {
            constexpr int i = decltype(ic)::v;
            if constexpr (!(i & half)) {
                constexpr int bound = inv_before(CAP, 4, t, i);
                const ulonglong2 w = __ldg(itw + (1 << k) + i / (2 * half));
                const u64 X = r[i], Y = r[i + half];
                r[i] = 2 * bound > CAP / 2 ? halve<CAP>(X + Y, q) : X + Y;
                r[i + half] = shoup3(X - Y + bound * q, w.x, w.y, q);
            }
        });
    });
}

// ---------------------------------------------------------------------------------------
// Full passes with the pass position as a runtime value. The register indexing is the same as
// in the compile-time form (S = LE, one group per thread); only the index bits of the
// shared-memory and twiddle addresses depend on the pass. Every full pass of a transform runs
// through one copy of this code, which keeps a kernel that chains many transforms small
// enough for the instruction cache.
// ---------------------------------------------------------------------------------------

// Natural index of register e of thread tid in the full pass whose lowest varying index bit
// is lo (= LOGN - S0 - LE): (tid >> lo) << (lo + LE) | e << lo | (tid & (2^lo - 1)).
template <int LE>
__device__ __forceinline__ int pass_base(int tid, int lo) { return ((tid >> lo) << (lo + LE)) | (tid & ((1 << lo) - 1)); }

// As in the compile-time form, slot = swz(base) ^ swz(e << lo); with lo known only at run time
// the E offsets swz(e << lo) are XOR combinations of the LE basis values swz(2^k << lo).
template <int E = 16>
__device__ __forceinline__ void rt_offsets(int lo, int (&c)[E])
{
    constexpr int LE = Radix<E>::LE;
    int b[LE];
#pragma unroll
    for (int k = 0; k < LE; ++k) b[k] = swz<E>(1 << (k + lo));
#pragma unroll
    for (int e = 0; e < E; ++e) {
        int v = 0;
#pragma unroll
        for (int k = 0; k < LE; ++k)
            if (e & (1 << k)) v ^= b[k];
        c[e] = v;
    }
}

template <int E = 16>
__device__ __forceinline__ void store_sm_rt(u64* sm, const u64 (&r)[E], int tid, int lo)
{
    const int base = swz<E>(pass_base<Radix<E>::LE>(tid, lo));
    int c[E];
    rt_offsets<E>(lo, c);
#pragma unroll
    for (int e = 0; e < E; ++e) sm[base ^ c[e]] = r[e];
}

template <int E = 16>
__device__ __forceinline__ void load_sm_rt(const u64* sm, u64 (&r)[E], int tid, int lo)
{
    const int base = swz<E>(pass_base<Radix<E>::LE>(tid, lo));
    int c[E];
    rt_offsets<E>(lo, c);
#pragma unroll
    for (int e = 0; e < E; ++e) r[e] = sm[base ^ c[e]];
}

// Forward stages S0 .. S0+LE-1 (lo = LOGN - S0 - LE): registers below CAP q on entry and exit (one
// code for every pass, so every stage halves its first operands). The runtime passes take the exact
// quotient: the three-product form spilled more there (312 against 184 bytes; per-pixel squared
// difference of 768 pairs at N = 2^14 16.9 against 13.3 ms).
template <int CAP, int E = 16>
__device__ __forceinline__ void fwd_regs_rt(u64 (&r)[E], int tid, int S0, int lo, const ulonglong2* __restrict__ tw, u64 q)
{
    constexpr int LE = Radix<E>::LE;
    const int h = tid >> lo;
#pragma unroll
    for (int k = 0; k < LE; ++k) {
        const int half = 1 << (LE - 1 - k);
#pragma unroll
        for (int b = 0; b < (1 << k); ++b) {
            const ulonglong2 w = __ldg(tw + (1 << (S0 + k)) + (h << k) + b);
#pragma unroll
            for (int jj = b * 2 * half; jj < b * 2 * half + half; ++jj) {
                const u64 X = halve<CAP>(r[jj], q);
                const u64 T = shoup_lazy(r[jj + half], w.x, w.y, q);
                r[jj] = X + T;
                r[jj + half] = X - T + 2 * q;
            }
        }
    }
}

// Inverse stages S0+LE-1 .. S0 (lo = LOGN - S0 - LE): registers below CAP/2 q on entry and exit.
template <int CAP, int E = 16>
__device__ __forceinline__ void inv_regs_rt(u64 (&r)[E], int tid, int S0, int lo, const ulonglong2* __restrict__ itw, u64 q)
{
    constexpr int LE = Radix<E>::LE;
    const int h = tid >> lo;
#pragma unroll
    for (int k = LE - 1; k >= 0; --k) {
        const int half = 1 << (LE - 1 - k);
#pragma unroll
        for (int b = 0; b < (1 << k); ++b) {
            const ulonglong2 w = __ldg(itw + (1 << (S0 + k)) + (h << k) + b);
#pragma unroll
            for (int jj = b * 2 * half; jj < b * 2 * half + half; ++jj) {
                const u64 X = r[jj], Y = r[jj + half];
                r[jj] = halve<CAP>(X + Y, q);
                r[jj + half] = shoup_lazy(X - Y + (CAP / 2) * q, w.x, w.y, q);
            }
        }
    }
}

// Whole forward transform, input already in registers in the layout of pass 0, below B q; output
// in registers in the layout of the last pass, below fwd_out q. `sm` holds N words. The caller
// must make sure no thread still reads `sm` from an earlier use other than an inverse transform's
// (a __syncthreads before the call; see the header comment).
// Passes: LOGN / LE full passes, then one pass of the remaining LOGN % LE stages.
// COMPACT runs the full passes through one runtime loop (one copy of the pass code); otherwise
// every pass is unrolled with its position known at compile time, which needs fewer address
// instructions but about LOGN / LE times the code. Both take a warp barrier for the exchanges
// that stay inside every warp (exchange_in_warp). The compact form, used by the per-pixel
// squared difference at N = 2^14 (where the unrolled passes spill), keeps the strided last-pass
// layout (WT = false; its callers index the last pass with it) and a block barrier into it:
// there the warp-adjacent layout took more registers (spills 8 -> 76 bytes) and time.
template <int LOGN, bool COMPACT, int CAP, int B>
__host__ __device__ constexpr int fwd_out() { return COMPACT ? CAP : fwd_bound(CAP, B, LOGN); }

template <int LOGN, bool COMPACT, int E, int CAP, int B>
__device__ __forceinline__ void ntt_fwd_regs(u64* sm, u64 (&r)[E], int tid, const ModTables& t, u64 q, int root = 1)
{
    constexpr int LE = Radix<E>::LE;
    if constexpr (!COMPACT) {
        ntt_fwd_polys<LOGN, E, CAP, B>(sm, reinterpret_cast<u64(&)[1][E]>(r), tid, t, q, root);
        return;
    }
    constexpr int NFULL = LOGN / LE, TAIL = LOGN % LE;
    constexpr unsigned in_warp = full_exchanges_in_warp(LOGN, E);
#pragma unroll 1
    for (int p = 0; p < NFULL; ++p) {
        const int lo = LOGN - LE * p - LE;
        if (p > 0) {
            store_sm_rt<E>(sm, r, tid, lo + LE);
            if ((in_warp >> p) & 1u) __syncwarp();   // uniform across the block
            else __syncthreads();
            load_sm_rt<E>(sm, r, tid, lo);
        }
        fwd_regs_rt<CAP, E>(r, tid, LE * p, lo, t.tw, q);
    }
    if constexpr (TAIL > 0) {
        store_sm_rt<E>(sm, r, tid, LOGN - LE * NFULL);
        __syncthreads();
        load_sm<LOGN, LE * NFULL, E, false>(sm, r, tid);
        fwd_regs<LOGN, LE * NFULL, E, false, CAP, CAP>(reinterpret_cast<u64(&)[1][E]>(r), tid, t.tw, q, 1);
    }
}

// Whole inverse transform, input in registers in the layout of the last pass, below 4q; output in
// registers in the layout of pass 0, natural order, below CAP/2 q.
template <int LOGN, bool COMPACT, int E, int CAP>
__device__ __forceinline__ void ntt_inv_regs(u64* sm, u64 (&r)[E], int tid, const ModTables& t, u64 q, int root = 1)
{
    constexpr int LE = Radix<E>::LE;
    if constexpr (!COMPACT) {
        inv_rest<LOGN, NttShape<LOGN, E>::LAST, E, CAP, 4>(sm, r, tid, t.itw, q, root);
        return;
    }
    constexpr int NFULL = LOGN / LE, TAIL = LOGN % LE;
    if constexpr (TAIL > 0) {
        inv_regs<LOGN, LE * NFULL, E, false, CAP, 4>(r, tid, t.itw, q, 1);
        store_sm<LOGN, LE * NFULL, E, false>(sm, r, tid);
        __syncthreads();
        load_sm_rt<E>(sm, r, tid, LOGN - LE * NFULL);
    }
    constexpr unsigned in_warp = full_exchanges_in_warp(LOGN, E);
#pragma unroll 1
    for (int p = NFULL - 1; p >= 0; --p) {
        const int lo = LOGN - LE * p - LE;
        inv_regs_rt<CAP, E>(r, tid, LE * p, lo, t.itw, q);
        if (p > 0) {
            store_sm_rt<E>(sm, r, tid, lo);
            if ((in_warp >> p) & 1u) __syncwarp();
            else __syncthreads();
            load_sm_rt<E>(sm, r, tid, lo + LE);
        }
    }
}

}  // namespace ichee
