// kernels_match.cu -- image matching (Sec. 4.4.3, as a squared L2 distance): the sum over all pixel
// ciphertexts of (a - b)^2 with ct x ct multiplication, then relinearisation with the
// evaluation key (Sec. 2.2.3; hybrid key switching with one special prime P).
#include "ops.h"
#include "ntt.cuh"

namespace ichee {

// Moduli below this run their transforms without any fold: outputs stay below (6 + 4 * 14) q, as the
// Montgomery products take them (mont_lazy).
constexpr u64 kNoFoldBelow = 1ull << 50;

// The tensor terms of two neighbouring positions added to the accumulators at acc, acc + n, acc + 2n
// (in [0, 2q)): d0^2, d0 d1, d1^2, each carrying 2^{-64}, undone after the inverse transform.
__device__ __forceinline__ void tensor_pair(u64* acc, int n, u64 d1x, u64 d1y, u64 d0x, u64 d0y, u64 q, u64 qinv)
{
    auto add = [&](u64* p, u64 tx, u64 ty) {
        ulonglong2* s = reinterpret_cast<ulonglong2*>(p);
        const ulonglong2 v = *s;
        *s = make_ulonglong2(csub_s(v.x + tx, 2 * q), csub_s(v.y + ty, 2 * q));
    };
    add(acc, mont_lazy(d0x, d0x, q, qinv), mont_lazy(d0y, d0y, q, qinv));
    add(acc + n, mont_lazy(d0x, d1x, q, qinv), mont_lazy(d0y, d1y, q, qinv));
    add(acc + 2 * n, mont_lazy(d1x, d1x, q, qinv), mont_lazy(d1y, d1y, q, qinv));
}

// A transform's output (below B q) as the products take it: below 4q, or any of a modulus below 2^50.
template <int B>
__device__ __forceinline__ u64 for_products(u64 x, u64 q)
{
    if constexpr (B > 16) return x;
    else return below4<B>(x, q);
}

// The tensor terms of all positions of a thread (last-pass layout) from the transforms of d0 (r[0]) and
// d1 (r[1]), below B q.
template <int LOGN, int E, int B>
__device__ __forceinline__ void tensor_terms(u64* acc, const u64 (&r)[2][E], int tid, u64 q, u64 qinv)
{
#pragma unroll
    for (int e = 0; e < E; e += 2)
        tensor_pair(acc + elem_index<LOGN, NttShape<LOGN, E>::LAST, E>(tid, e), 1 << LOGN, for_products<B>(r[1][e], q),
                    for_products<B>(r[1][e + 1], q), for_products<B>(r[0][e], q), for_products<B>(r[0][e + 1], q), q,
                    qinv);
}

// One block per SM-sized share of the work: block j owns limb l = j % limbs and every
// (n_blocks/limbs)-th ciphertext. Per ciphertext it forms d = a - b for its limb, transforms
// d0 and d1, and accumulates (d0^2, d0 d1, d1^2) position by position into its own slice of
// the scratch buffer (each position is owned by one thread, so no atomics are needed; the middle
// term is doubled when the slices are added up). From N = 2^12 a thread holds its 8 residues of both
// polynomials in registers: they share the twiddle loads and the exchange barriers, give every warp two
// independent chains, and reach the tensor terms without a detour through shared memory. Below, d0 is
// transformed first and waits in its own slots of the second buffer: with many small blocks on an SM
// that is as fast or faster (900 pairs at N = 2^10 139 us, both at once 147; 3600 at 2^11 487 and 489).
// Values stay lazily reduced throughout (ntt.cuh): the difference in [0, 2q), the
// transforms' outputs below 4q as the Montgomery products take them, the accumulators in [0, 2q).
// Moduli below 2^50 (NOFOLD) need no reduction inside a transform at all.
// Whole matching calls, 4096 pairs at N = 2^13 with primes 60/40/60: 2.59 ms with a conditional
// subtraction per butterfly, exact quotients and canonical values, 2.31 lazily reduced, 2.27 with the
// exchange barriers of ntt.cuh, 2.24 with the short relinearisation below, 2.15 with both polynomials at
// once; 1600 pairs at N = 2^12 0.74 ms at first, 0.52 with the short relinearisation, 0.50 now. What bounds it: the multiply pipe, three quarters busy; the rest of the time goes
// to exchanges and to the tensor terms' accumulators (in L2).
template <int LOGN, int E, int CAP>
__device__ __forceinline__ void sqdiff_accumulate(const SqDiffArgs& a, u64* buf)
{
    constexpr int N = 1 << LOGN;
    constexpr int LAST = NttShape<LOGN, E>::LAST;
    constexpr int OUT = fwd_out<LOGN, false, CAP, 2>();
    u64* acc = a.partial + (size_t)blockIdx.x * 4 * N;
    const int tid = threadIdx.x;
    const int limbs = a.limbs;
    const int l = blockIdx.x % limbs;
    const u64 stride = a.n_blocks / limbs;
    const u64 start = blockIdx.x / limbs;
    const u64 q = a.rns.q[l];
    const u64 qinv = a.rns.qinv[l];
    const ModTables t = a.rns.tab[l];
    // In the last pass registers e and e + 1 (e even) hold positions x and x + 1 (its lowest
    // index bit is the stage bit), so the accumulators are read and written in 16-byte pairs.
#pragma unroll
    for (int e = 0; e < E; e += 2) {
        const int x = elem_index<LOGN, LAST, E>(tid, e);
        *reinterpret_cast<ulonglong2*>(acc + x) = make_ulonglong2(0, 0);
        *reinterpret_cast<ulonglong2*>(acc + N + x) = make_ulonglong2(0, 0);
        *reinterpret_cast<ulonglong2*>(acc + 2 * N + x) = make_ulonglong2(0, 0);
    }
    for (u64 k = start; k < a.n_ct; k += stride) {
        const u64* A = a.a + k * 2 * (u64)limbs * N;
        const u64* B = a.b + k * 2 * (u64)limbs * N;
        const int x0 = elem_index<LOGN, 0, E>(tid, 0);   // first-pass layout: x0 + elem_offset(e)
        if constexpr (LOGN >= 12) {
            u64 r[2][E];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const u64* pa = A + ((u64)p * limbs + l) * N + x0;
                const u64* pb = B + ((u64)p * limbs + l) * N + x0;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int x = elem_offset<LOGN, 0, E>(e);
                    r[p][e] = __ldcs(pa + x) + q - __ldcs(pb + x);
                }
            }
            __syncthreads();   // the last exchange's loads of the previous pixel are over
            ntt_fwd_polys<LOGN, E, CAP, 2>(buf, r, tid, t, q);
            tensor_terms<LOGN, E, OUT>(acc, r, tid, q, qinv);
        } else {
            u64* d0buf = buf + N;
#pragma unroll 1
            for (int p = 0; p < 2; ++p) {
                const u64* pa = A + ((u64)p * limbs + l) * N + x0;
                const u64* pb = B + ((u64)p * limbs + l) * N + x0;
                u64 r[E];
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int x = elem_offset<LOGN, 0, E>(e);
                    r[e] = __ldcs(pa + x) + q - __ldcs(pb + x);
                }
                // d0 is transformed in its parking buffer and d1 in the other one: the barrier before d0's
                // transform is past every thread's reads of the previous pixel from either buffer, so
                // d1's transform needs none of its own. Every thread parks
                // and reads back only the slots of its own last-pass registers -- the slots it loaded
                // in the transform's last exchange -- so no barrier follows the transform.
                if (p == 0) __syncthreads();
                u64* dst = p == 0 ? d0buf : buf;
                ntt_fwd_regs<LOGN, false, E, CAP, 2>(dst, r, tid, t, q);
                const int sb = slot_base<LOGN, LAST, E>(tid);
#pragma unroll
                for (int e = 0; e < E; ++e) dst[slot_of<LOGN, LAST, E>(sb, e)] = for_products<OUT>(r[e], q);
            }
#pragma unroll
            for (int e = 0; e < E; e += 2) {
                const int x = elem_index<LOGN, LAST, E>(tid, e);
                tensor_pair(acc + x, N, buf[swz<E>(x)], buf[swz<E>(x + 1)], d0buf[swz<E>(x)], d0buf[swz<E>(x + 1)], q,
                            qinv);
            }
        }
    }
}

template <int LOGN, int E>
__global__ void __launch_bounds__(NttShape<LOGN, E>::T, sqdiff_blocks_per_sm(LOGN)) k_sqdiff_accumulate(const __grid_constant__ SqDiffArgs a)
{
    extern __shared__ u64 buf[];
    if (a.rns.q[blockIdx.x % a.limbs] < kNoFoldBelow) sqdiff_accumulate<LOGN, E, kNoFold>(a, buf);
    else sqdiff_accumulate<LOGN, E, 16>(a, buf);
}

// N = 2^14, split: the first stage of the forward transform pairs x with x + N/2 and leaves two
// independent 2^13-point transforms (outputs with the top index bit clear, and set). Block j
// takes limb j % limbs and half h = (j / limbs) % 2: it loads both halves of d = a - b, applies
// the first-stage butterfly for its half only (the product W d_hi is made by both halves'
// blocks: 1/14 more products), and runs the other 13 stages with the 2^13-point code -- 8
// residues of both polynomials per thread, 1024 threads -- from root 2 + h of the table. Its tensor terms
// go to a [4][N/2] slice. The two blocks of a half pair read the same ciphertexts at about the same
// time (one HBM read, one L2 hit). 992 pairs of five limbs: 2.14 ms with the polynomials in turn, 2.08
// with both at once (2.21 while the slot and twiddle addresses of every pass were kept, spilled, across
// pixels: the opaque thread number below makes them anew).
template <int CAP>
__device__ __forceinline__ void sqdiff_accumulate_split(const SqDiffArgs& a, u64* buf)
{
    constexpr int LOGH = 13, NH = 1 << LOGH, N = 2 * NH, E = 8;
    constexpr int LAST = NttShape<LOGH, E>::LAST;
    constexpr int IN = 6, OUT = fwd_out<LOGH, false, CAP, IN>();
    const int tid = threadIdx.x;
    const int limbs = a.limbs;
    const int l = blockIdx.x % limbs;
    const int h = (blockIdx.x / limbs) & 1;
    const u64 stride = a.n_blocks / (2 * limbs);
    const u64 start = blockIdx.x / (2 * limbs);
    u64* acc = a.partial + (size_t)blockIdx.x * 4 * NH;
    const u64 q = a.rns.q[l];
    const u64 qinv = a.rns.qinv[l];
    const ModTables t = a.rns.tab[l];   // the halves' roots are 2 and 3
    const ulonglong2 w1 = a.rns.tab[l].tw[1];   // the first stage's twiddle and its companion
#pragma unroll
    for (int e = 0; e < E; e += 2) {
        const int x = elem_index<LOGH, LAST, E>(tid, e);
        *reinterpret_cast<ulonglong2*>(acc + x) = make_ulonglong2(0, 0);
        *reinterpret_cast<ulonglong2*>(acc + NH + x) = make_ulonglong2(0, 0);
        *reinterpret_cast<ulonglong2*>(acc + 2 * NH + x) = make_ulonglong2(0, 0);
    }
    for (u64 k = start; k < a.n_ct; k += stride) {
        const u64* A = a.a + k * 2 * (u64)limbs * N;
        const u64* B = a.b + k * 2 * (u64)limbs * N;
        int tid = threadIdx.x;
        asm volatile("" : "+r"(tid));
        const int x0 = elem_index<LOGH, 0, E>(tid, 0);
        u64 r[2][E];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const u64* pa = A + ((u64)p * limbs + l) * N + x0;
            const u64* pb = B + ((u64)p * limbs + l) * N + x0;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int x = elem_offset<LOGH, 0, E>(e);
                const u64 lo = pa[x] + q - pb[x];                                   // [0, 2q)
                const u64 tt = shoup3(pa[x + NH] + q - pb[x + NH], w1.x, w1.y, q);   // [0, 4q)
                r[p][e] = h ? lo + 4 * q - tt : lo + tt;                            // below IN q
            }
        }
        __syncthreads();   // the last exchange's loads of the previous pixel are over
        ntt_fwd_polys<LOGH, E, CAP, IN>(buf, r, tid, t, q, 2 + h);
        tensor_terms<LOGH, E, OUT>(acc, r, tid, q, qinv);
    }
}

__global__ void __launch_bounds__(1024, 1) k_sqdiff_accumulate_split(const __grid_constant__ SqDiffArgs a)
{
    extern __shared__ u64 buf[];
    if (a.rns.q[blockIdx.x % a.limbs] < kNoFoldBelow) sqdiff_accumulate_split<kNoFold>(a, buf);
    else sqdiff_accumulate_split<16>(a, buf);
}

// 8 residues per thread: 1024 threads in 64 registers per SM at every N, as one block or several.
template <int LOGN>
static cudaError_t sqdiff_launch(const SqDiffArgs& a, cudaStream_t st)
{
    constexpr int E = 8;
    const size_t smem = 2 * (sizeof(u64) << LOGN);
    cudaError_t e = cudaFuncSetAttribute(k_sqdiff_accumulate<LOGN, E>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    k_sqdiff_accumulate<LOGN, E><<<a.n_blocks, NttShape<LOGN, E>::T, smem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_sqdiff_accumulate(const SqDiffArgs& a, cudaStream_t st)
{
    if (a.n_blocks <= 0 || a.n_blocks % a.limbs != 0) return cudaErrorInvalidValue;
    if (sqdiff_split(a.rns.logn)) {
        if (a.n_blocks % (2 * a.limbs) != 0) return cudaErrorInvalidValue;
        const size_t smem = 2 * (sizeof(u64) << 13);
        cudaError_t e = cudaFuncSetAttribute(k_sqdiff_accumulate_split, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        k_sqdiff_accumulate_split<<<a.n_blocks, NttShape<13, 8>::T, smem, st>>>(a);
        return cudaGetLastError();
    }
    switch (a.rns.logn) {
    case 10: return sqdiff_launch<10>(a, st);
    case 11: return sqdiff_launch<11>(a, st);
    case 12: return sqdiff_launch<12>(a, st);
    case 13: return sqdiff_launch<13>(a, st);
    default: return cudaErrorInvalidValue;
    }
}

__global__ void k_sqdiff_reduce(RnsArgs rns, int limbs, const u64* partial, int n_blocks, u64* tensor, int add)
{
    const int n = 1 << rns.logn;
    const int pl = blockIdx.y;                 // p * limbs + l
    const int p = pl / limbs, l = pl % limbs;
    const u64 q = rns.q[l];
    const bool split = sqdiff_split(rns.logn);
    const int row = split ? n / 2 : n;         // slice row length
    const int step = split ? 2 * limbs : limbs;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < n; x += gridDim.x * blockDim.x) {
        u64 s = 0;
        const int h = split ? x / row : 0, xx = split ? x % row : x;
        for (int j = l + h * limbs; j < n_blocks; j += 8 * step) {   // slices in [0, 2q), the sum too
            u64 v[8];   // eight loads in flight
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int ju = j + u * step;
                v[u] = ju < n_blocks ? partial[((size_t)ju * 4 + p) * row + xx] : 0;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) s = csub_s(s + v[u], 2 * q);
        }
        s = csub_s(s, q);
        if (p == 1) s = add_mod(s, s, q);                      // 2 d0 d1
        if (add) s = add_mod(s, reduce64(tensor[(size_t)pl * n + x], q, rns.mu[l]), q);
        tensor[(size_t)pl * n + x] = s;
    }
}

cudaError_t launch_sqdiff_reduce(const RnsArgs& rns, int limbs, const u64* partial, int n_blocks, u64* tensor,
                                 bool add, cudaStream_t st)
{
    dim3 grid((1u << rns.logn) / 256, 3 * limbs);
    k_sqdiff_reduce<<<grid, 256, 0, st>>>(rns, limbs, partial, n_blocks, tensor, add ? 1 : 0);
    return cudaGetLastError();
}

// out[r][x] = in[r][x] mod q_{r % limbs} for any 64-bit input word (sums of accumulators).
__global__ void k_reduce_rows(RnsArgs rns, int limbs, const u64* in, u64* out)
{
    const int n = 1 << rns.logn;
    const int r = blockIdx.y, l = r % limbs;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < n; x += gridDim.x * blockDim.x)
        out[(size_t)r * n + x] = reduce64(in[(size_t)r * n + x], rns.q[l], rns.mu[l]);
}

cudaError_t launch_reduce_rows(const RnsArgs& rns, int rows, int limbs, const u64* in, u64* out, cudaStream_t st)
{
    dim3 grid((1u << rns.logn) / 256, rows);
    k_reduce_rows<<<grid, 256, 0, st>>>(rns, limbs, in, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Per-pixel squared difference: out_k = Rescale(Relin((a_k - b_k) (x) (a_k - b_k))) for every
// ciphertext pair (the per-pixel form of Sec. 4.4.3; Relin by hybrid key switching, rescale
// with centered rounding). A persistent block takes one pixel at a time and runs the whole chain on it:
//   1. per limb l: d^ = NTT(a - b) for both polynomials; t0^ = d0^2, t1^ = 2 d0 d1 stay in the
//      NTT domain; t2 = INTT(d1^2) (N^{-1} folded into the product). The squares are
//      Montgomery products, so each carries 2^{-64}; the constants below carry 2^64. Digit l
//      of t2 lifted to its own modulus q_l is t2_l itself, whose transform d1^2 is at hand, so
//      the accumulators of modulus q_l start here: acc_b = (P N^{-1} 2^64) t_b^ + d1^2 evk^_l[b][l];
//   2. per modulus m (P first, then q_t, then q_0..q_{t-1}): acc_b += NTT([t2]_j lifted to m) *
//      evk^_j[b][m] for every digit j != m (all j for P), so INTT(acc_b) = P t_b + key-switched
//      part and (INTT(acc_b) - [acc_b mod P]) P^{-1} is the relinearised limb m;
//   3. the relinearised limb q_t is kept; every other limb is rescaled against it and stored.
// That is L^2 + 5L + 2 transforms per pixel (t2 is the only tensor limb inverse-transformed,
// and no digit is transformed back into its own modulus). They run in one loop over a per-pixel
// schedule (one word per transform, in shared memory) with one call site per direction, so the
// transform code with every pass unrolled appears twice and fits the instruction cache (four
// unrolled call sites did not; the compact pass loop in this schedule took 15.0 ms for 4096
// pixels at N = 2^13, the unrolled passes 12.6 ms, the compact loop at four call sites 13.9).
// A transform's first exchange stores to the slots of its thread in pass 0 (forward) or in the
// last pass (inverse), and its last exchange loads the slots of the other end, so a block
// barrier is needed only between two transforms of the same direction: after a forward, an
// inverse overwrites only slots its thread loaded last, and after an inverse a forward does.
// 4096 pairs at N = 2^13 and three limbs take 11.0 ms (11.9 with a subtraction per butterfly, exact
// quotients and canonical accumulators), 768 at N = 2^14 and five limbs 13.3 ms.
// Every intermediate word is produced and consumed by the same thread (the transforms move
// data between threads only through their own shared buffer), so the block's scratch
// ([3 limbs + 2][N] words: t0^, t1^, t2 per limb, then the two P accumulators) is stored
// thread-major -- element e of thread tid at e * T + tid -- which makes every scratch access
// coalesced and needs no barrier of its own. The key-switching accumulators of modulus q_m
// build up in the t0^ / t1^ slots of limb m (the P accumulators in their own slots); keeping
// them in shared memory instead was slower, because the larger carve-out leaves too little
// L1 for the twiddle tables.
// ---------------------------------------------------------------------------------------
// Transform kinds of the per-pixel schedule.
constexpr u32 kFwdDiff = 0, kInvT2 = 1, kFwdDigit = 2, kInvAcc = 3;

template <int LOGN, int E>
__global__ void __launch_bounds__(NttShape<LOGN, E>::T, sqdiff_blocks_per_sm(LOGN)) k_sqdiff_image(const __grid_constant__ SqImgArgs a)
{
    constexpr int N = 1 << LOGN;
    constexpr int T = NttShape<LOGN, E>::T;
    constexpr int LAST = NttShape<LOGN, E>::LAST;
    // transforms with every pass unrolled up to N = 2^13 (one call site per direction, so the
    // code fits the instruction cache), the compact pass loop at 2^14 (registers)
    constexpr bool CMP = LOGN >= 14;
    constexpr bool WT = !CMP;   // the last-pass layout of the unrolled form keeps a warp's groups adjacent
    extern __shared__ u64 sm[];
    u32* sched = reinterpret_cast<u32*>(sm + N);
    const int tid = threadIdx.x;
    const int limbs = a.limbs, L = a.L;
    const int t = limbs - 1;
    u64* S = a.scratch + (size_t)blockIdx.x * (3 * limbs + 2) * N + tid;   // thread-major slots
    u64* T0 = S;                          // [limbs] t0^, then the poly-0 accumulator / relinearised q_t limb
    u64* T1 = S + (size_t)limbs * N;      // [limbs] t1^, likewise for poly 1
    u64* T2 = S + (size_t)2 * limbs * N;  // [limbs] d1^, then t2 in the coefficient domain
    u64* AP = S + (size_t)3 * limbs * N;  // [2] accumulators modulo P, then their inverse transforms
    const u64 P = a.rns.q[L];
    const u64 halfP = (P - 1) / 2;
    // The transforms of one pixel in order, one word each: kind (bits 0-1), polynomial (2), limb
    // or digit (3-6), target modulus (7-10, 15 = P), barrier before the transform (11), first
    // term of the P accumulators (12). A barrier is needed only between two transforms of the
    // same direction (see above).
    if (tid == 0) {
        int n = 0;
        auto push = [&](u32 kind, u32 pb, u32 x, u32 mm, u32 bar, u32 first) {
            sched[n++] = kind | (pb << 2) | (x << 3) | (mm << 7) | (bar << 11) | (first << 12);
        };
        for (int l = 0; l < limbs; ++l) {
            push(kFwdDiff, 0, l, 0, 0, 0);
            push(kFwdDiff, 1, l, 0, 1, 0);
            push(kInvT2, 0, l, 0, 0, 0);
        }
        for (int step = 0; step <= limbs; ++step) {
            const int m = step == 0 ? -1 : (step == 1 ? t : step - 2);
            const u32 mm = m < 0 ? 15u : (u32)m;
            bool first = true;
            for (int j = 0; j < limbs; ++j) {
                if (j == m) continue;   // digit m's term went in with t_b^ in the first phase
                push(kFwdDigit, 0, j, mm, first ? 0 : 1, m < 0 && j == 0 ? 1 : 0);
                first = false;
            }
            push(kInvAcc, 0, 0, mm, 0, 0);
            push(kInvAcc, 1, 0, mm, 1, 0);
        }
    }
    __syncthreads();
    const int n_ops = limbs * limbs + 5 * limbs + 2;
    for (u64 k = blockIdx.x; k < a.n_ct; k += gridDim.x) {
        const u64* A = a.a + k * 2 * (u64)limbs * N;
        const u64* B = a.b + k * 2 * (u64)limbs * N;
        u64 r[E];
#pragma unroll 1
        for (int op = 0; op < n_ops; ++op) {
            const u32 code = sched[op];
            const u32 kind = code & 3u;
            const int pb = (int)((code >> 2) & 1u), x = (int)((code >> 3) & 15u);
            const int m = ((code >> 7) & 15u) == 15u ? -1 : (int)((code >> 7) & 15u);
            const int mod = kind == kFwdDiff || kind == kInvT2 ? x : (m < 0 ? L : m);
            const u64 q = a.rns.q[mod];
            if (kind == kFwdDiff || kind == kFwdDigit) {
                if (kind == kFwdDiff) {   // d = a - b, polynomial pb of limb x
                    const u64* pa = A + ((u64)pb * limbs + x) * N;
                    const u64* pq = B + ((u64)pb * limbs + x) * N;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const int xi = elem_index<LOGN, 0, E>(tid, e);
                        r[e] = __ldcs(pa + xi) + q - __ldcs(pq + xi);   // [0, 2q)
                    }
                } else {                  // digit x of t2, centered, lifted to the modulus
                    const u64 mu = a.rns.mu[mod];
                    const u64 qj = a.rns.q[x];
                    const u64 half = (qj - 1) / 2;
                    const u64* t2 = T2 + (size_t)x * N;
                    if (qj <= q) {        // |digit| < q_j / 2 < q: no reduction
#pragma unroll
                        for (int e = 0; e < E; ++e) {
                            const u64 v = t2[e * T];
                            r[e] = v <= half ? v : q - (qj - v);
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < E; ++e) {
                            const u64 v = t2[e * T];
                            if (v <= half) {
                                r[e] = reduce64(v, q, mu);
                            } else {
                                const u64 mag = reduce64(qj - v, q, mu);
                                r[e] = mag == 0 ? 0 : q - mag;
                            }
                        }
                    }
                }
                if ((code >> 11) & 1u) __syncthreads();
                ntt_fwd_regs<LOGN, CMP, E, 8, 2>(sm, r, tid, a.rns.tab[mod], q);   // below 8q
                if (kind == kFwdDiff) {
                    u64* dst = (pb == 0 ? T0 : T2) + (size_t)x * N;
#pragma unroll
                    for (int e = 0; e < E; ++e) dst[e * T] = below4<8>(r[e], q);   // as mont_lazy takes it
                } else {                  // acc_b(m) += NTT(digit) * evk^_x[b][m]
                    u64* acc0 = m < 0 ? AP : T0 + (size_t)m * N;
                    u64* acc1 = m < 0 ? AP + N : T1 + (size_t)m * N;
                    const bool init = (code >> 12) & 1u;
                    const u64* e0 = a.evk_hat + (((size_t)x * 2 + 0) * (L + 1) + mod) * N;
                    const u64* e0p = a.evk_hat_p + (((size_t)x * 2 + 0) * (L + 1) + mod) * N;
                    const u64* e1 = a.evk_hat + (((size_t)x * 2 + 1) * (L + 1) + mod) * N;
                    const u64* e1p = a.evk_hat_p + (((size_t)x * 2 + 1) * (L + 1) + mod) * N;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const int xi = elem_index<LOGN, LAST, E, WT>(tid, e);
                        // the accumulators stay in [0, 4q): the inverse transform takes that range
                        const u64 p0 = shoup3(r[e], __ldg(e0 + xi), __ldg(e0p + xi), q);
                        const u64 p1 = shoup3(r[e], __ldg(e1 + xi), __ldg(e1p + xi), q);
                        const u64 s0 = init ? 0 : acc0[e * T];
                        const u64 s1 = init ? 0 : acc1[e * T];
                        acc0[e * T] = halve<8>(s0 + p0, q);
                        acc1[e * T] = halve<8>(s1 + p1, q);
                    }
                }
            } else {
                if (kind == kInvT2) {     // the tensor of limb x; t2 = INTT(d1^2) next
                    u64* t0 = T0 + (size_t)x * N;
                    u64* t1 = T1 + (size_t)x * N;
                    const u64* t2 = T2 + (size_t)x * N;
                    const u64 qinv = a.rns.qinv[x];   // Montgomery products: 2^64 is folded into ninv, pn and r64
                    const u64* e0 = a.evk_hat + (((size_t)x * 2 + 0) * (L + 1) + x) * N;
                    const u64* e0p = a.evk_hat_p + (((size_t)x * 2 + 0) * (L + 1) + x) * N;
                    const u64* e1 = a.evk_hat + (((size_t)x * 2 + 1) * (L + 1) + x) * N;
                    const u64* e1p = a.evk_hat_p + (((size_t)x * 2 + 1) * (L + 1) + x) * N;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const int xi = elem_index<LOGN, LAST, E, WT>(tid, e);
                        const u64 d0 = t0[e * T], d1 = t2[e * T];
                        const u64 m2 = mont_lazy(d1, d1, q, qinv);
                        const u64 th = shoup3(m2, a.r64[x], a.r64_p[x], q);   // d1^2, the transform of digit x
                        const u64 c = mont_lazy(d0, d1, q, qinv);
                        t0[e * T] = halve<8>(shoup3(mont_lazy(d0, d0, q, qinv), a.pn[x], a.pn_p[x], q) +
                                             shoup3(th, __ldg(e0 + xi), __ldg(e0p + xi), q), q);
                        t1[e * T] = halve<8>(shoup3(c + c, a.pn[x], a.pn_p[x], q) +
                                             shoup3(th, __ldg(e1 + xi), __ldg(e1p + xi), q), q);
                        r[e] = shoup3(m2, a.ninv[x], a.ninv_p[x], q);
                    }
                } else {
                    const u64* acc = (m < 0 ? AP + (size_t)pb * N : (pb == 0 ? T0 : T1) + (size_t)m * N);
#pragma unroll
                    for (int e = 0; e < E; ++e) r[e] = acc[e * T];
                }
                if ((code >> 11) & 1u) __syncthreads();
                ntt_inv_regs<LOGN, CMP, E, 8>(sm, r, tid, a.rns.tab[mod], q);      // below 4q
                if (kind == kInvT2) {
                    u64* t2 = T2 + (size_t)x * N;
#pragma unroll
                    for (int e = 0; e < E; ++e) t2[e * T] = below1<4>(r[e], q);
                } else if (m < 0) {
                    u64* acc = AP + (size_t)pb * N;
#pragma unroll
                    for (int e = 0; e < E; ++e) acc[e * T] = below1<4>(r[e], q);
                } else {
                    const u64 mu = a.rns.mu[mod];
                    u64* acc = (pb == 0 ? T0 : T1) + (size_t)m * N;
                    const u64* last = (pb == 0 ? T0 : T1) + (size_t)t * N;
                    u64* o = a.out + ((k * 2 + pb) * (u64)t + m) * N;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const u64 ap = AP[(size_t)pb * N + e * T];
                        u64 lp = reduce64(ap, q, mu);
                        if (ap > halfP) lp = add_mod(lp, a.neg_p_mod[m], q);   // (ap - P) mod q_m
                        const u64 md = shoup(r[e] + q - lp, a.p_inv[m], a.p_inv_p[m], q);
                        if (m == t) {
                            acc[e * T] = md;              // relinearised limb q_t, the rescale's divisor
                        } else {
                            const u64 ct = last[e * T];
                            const u64 u = shoup_lazy(md, a.qt_inv[m], a.qt_inv_p[m], q);
                            const u64 w = shoup_lazy(ct, a.qt_inv[m], a.qt_inv_p[m], q);
                            u64 v = csub(csub(u + 2 * q - w, 2 * q), q);
                            if (ct > a.half_qt) v = add_mod(v, 1, q);
                            __stcs(o + elem_index<LOGN, 0, E>(tid, e), v);
                        }
                    }
                }
            }
        }
    }
}

size_t sqdiff_image_scratch_words(int logn, int limbs) { return (size_t)(3 * limbs + 2) << logn; }

// Residues per thread: 8 up to N = 2^13 (twice the warps of the 16-residue layout hide the
// latency of the scratch and key loads), 16 at N = 2^14 (thread limit).
template <int LOGN>
static constexpr int kSqImgE = LOGN <= 13 ? 8 : 16;

template <int LOGN>
static size_t sqimg_smem() { return (sizeof(u64) << LOGN) + 128 * sizeof(u32); }   // + the schedule

template <int LOGN>
static cudaError_t sqimg_prepare(int* blocks_per_sm)
{
    auto kern = k_sqdiff_image<LOGN, kSqImgE<LOGN>>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sqimg_smem<LOGN>());
    if (e != cudaSuccess) return e;
    if (blocks_per_sm)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kern, NttShape<LOGN, kSqImgE<LOGN>>::T,
                                                          sqimg_smem<LOGN>());
    return e;
}

static cudaError_t sqimg_prepare_any(int logn, int* blocks_per_sm)
{
    switch (logn) {
    case 10: return sqimg_prepare<10>(blocks_per_sm);
    case 11: return sqimg_prepare<11>(blocks_per_sm);
    case 12: return sqimg_prepare<12>(blocks_per_sm);
    case 13: return sqimg_prepare<13>(blocks_per_sm);
    case 14: return sqimg_prepare<14>(blocks_per_sm);
    default: return cudaErrorInvalidValue;
    }
}

int sqdiff_image_grid(int logn, u64 n_ct, int num_sms)
{
    int per_sm = 0;
    if (sqimg_prepare_any(logn, &per_sm) != cudaSuccess || per_sm < 1) per_sm = 1;
    const u64 cap = (u64)num_sms * per_sm;
    return (int)(n_ct < cap ? n_ct : cap);
}

template <int LOGN>
static void sqimg_launch(const SqImgArgs& a, int grid, cudaStream_t st)
{
    k_sqdiff_image<LOGN, kSqImgE<LOGN>><<<grid, NttShape<LOGN, kSqImgE<LOGN>>::T, sqimg_smem<LOGN>(), st>>>(a);
}

cudaError_t launch_sqdiff_image(const SqImgArgs& a, int grid, cudaStream_t st)
{
    if (grid <= 0 || a.n_ct == 0) return cudaSuccess;
    cudaError_t e = sqimg_prepare_any(a.rns.logn, nullptr);
    if (e != cudaSuccess) return e;
    switch (a.rns.logn) {
    case 10: sqimg_launch<10>(a, grid, st); break;
    case 11: sqimg_launch<11>(a, grid, st); break;
    case 12: sqimg_launch<12>(a, grid, st); break;
    case 13: sqimg_launch<13>(a, grid, st); break;
    case 14: sqimg_launch<14>(a, grid, st); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Relinearisation and rescale of one degree-2 ciphertext in the transform domain (matching's sum):
// hybrid key switching with one special prime P, one digit per ciphertext prime, mod-down and
// rescale with centered rounding, as the per-pixel kernel does them (t0^ and t1^ stay in the
// transform domain, times P; digit j needs no transform into its own modulus). One ciphertext has
// few transforms, so each is split over R = 2^LS blocks (R = 8; 4 at N = 2^10) -- the stages that
// couple the parts run in the elementwise kernels before and after -- and lifts, key products,
// mod-down and rescale ride along. Five short launches after the sum instead of eight with whole
// transforms in one block each: 43 instead of 67 us of kernels at N = 2^13 and three limbs, 52 instead
// of 119 at N = 2^14 and five; matching of one pair 116 -> 75 and 171 -> 89 us.
// ---------------------------------------------------------------------------------------
template <int LOGN>
static constexpr int kRelinLs = LOGN == 10 ? 2 : 3;

// t2: the parts of INTT(t2^ N^{-1} 2^64) of every limb, below 4q. Block (limb, part).
template <int LOGN>
__global__ void __launch_bounds__((1 << (LOGN - kRelinLs<LOGN>)) / 8) k_relin_t2(const __grid_constant__ SqImgArgs a,
                                                                               const u64* t2_hat, u64* t2)
{
    constexpr int LS = kRelinLs<LOGN>, LOGM = LOGN - LS, E = 8, LAST = NttShape<LOGM, E>::LAST;
    extern __shared__ u64 sm[];
    const int tid = threadIdx.x, l = blockIdx.x >> LS, h = blockIdx.x & ((1 << LS) - 1);
    const u64 q = a.rns.q[l];
    const size_t at = ((size_t)l << LOGN) + ((size_t)h << LOGM);
    u64 r[E];
#pragma unroll
    for (int e = 0; e < E; ++e)
        r[e] = shoup3(t2_hat[at + elem_index<LOGM, LAST, E>(tid, e)], a.ninv[l], a.ninv_p[l], q);
    ntt_inv_regs<LOGM, false, E, 8>(sm, r, tid, a.rns.tab[l], q, (1 << LS) + h);
#pragma unroll
    for (int e = 0; e < E; ++e) t2[at + elem_index<LOGM, 0, E>(tid, e)] = r[e];
}

// digits[j][m], m = 0 .. limbs (limbs: P), m != j: digit j of t2, centered, lifted to modulus m, through
// the stages that couple the parts of its transform (below 8q). One thread per (j, m) and R coefficients.
template <int LOGN>
__global__ void __launch_bounds__(128) k_relin_digits(const __grid_constant__ SqImgArgs a, const u64* t2, u64* digits)
{
    constexpr int LS = kRelinLs<LOGN>, R = 1 << LS, M = 1 << (LOGN - LS);
    const int nm = a.limbs + 1;
    const int j = blockIdx.y / a.limbs, mj = blockIdx.y % a.limbs, m = mj + (mj >= j ? 1 : 0);
    const int mod = m < a.limbs ? m : a.L;
    const u64 qj = a.rns.q[j], q = a.rns.q[mod], mu = a.rns.mu[mod], half = (qj - 1) / 2;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M) return;
    u64 r[R];
#pragma unroll
    for (int k = 0; k < R; ++k) r[k] = t2[((size_t)j << LOGN) + k * M + i];
    inv_tail<LS, 8>(r, a.rns.tab[j].itw, qj);
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const u64 v = below1<4>(r[k], qj), mag = reduce64(v <= half ? v : qj - v, q, mu);
        r[k] = v <= half || mag == 0 ? mag : q - mag;
    }
    fwd_head<LS, 8>(r, a.rns.tab[mod].tw, q);
#pragma unroll
    for (int k = 0; k < R; ++k) digits[((size_t)(j * nm + m) << LOGN) + k * M + i] = r[k];
}

// The parts of the digits' transforms, in place (below 8q). Block ((j, m != j), part).
template <int LOGN>
__global__ void __launch_bounds__((1 << (LOGN - kRelinLs<LOGN>)) / 8) k_relin_fwd(const __grid_constant__ SqImgArgs a,
                                                                                u64* digits)
{
    constexpr int LS = kRelinLs<LOGN>, LOGM = LOGN - LS, E = 8, LAST = NttShape<LOGM, E>::LAST;
    extern __shared__ u64 sm[];
    const int tid = threadIdx.x, jm = blockIdx.x >> LS, h = blockIdx.x & ((1 << LS) - 1);
    const int j = jm / a.limbs, mj = jm % a.limbs, m = mj + (mj >= j ? 1 : 0);
    const int mod = m < a.limbs ? m : a.L;
    const u64 q = a.rns.q[mod];
    u64* d = digits + ((size_t)(j * (a.limbs + 1) + m) << LOGN) + ((size_t)h << LOGM);
    u64 r[E];
#pragma unroll
    for (int e = 0; e < E; ++e) r[e] = d[elem_index<LOGM, 0, E>(tid, e)];
    ntt_fwd_regs<LOGM, false, E, 8, 8>(sm, r, tid, a.rns.tab[mod], q, (1 << LS) + h);
#pragma unroll
    for (int e = 0; e < E; ++e) d[elem_index<LOGM, LAST, E>(tid, e)] = r[e];
}

// acc[b][m] = the parts of INTT(sum_{j != m} digit_j^ evk_j^[b][m] + (P N^{-1} 2^64) t_b^ + t2^ 2^64 evk_m^[b][m])
// (the last two for m < limbs), below 4q. Block ((b, m), part).
template <int LOGN>
__global__ void __launch_bounds__((1 << (LOGN - kRelinLs<LOGN>)) / 8)
    k_relin_acc(const __grid_constant__ SqImgArgs a, const u64* tensor, const u64* digits, u64* acc)
{
    constexpr int LS = kRelinLs<LOGN>, LOGM = LOGN - LS, E = 8, LAST = NttShape<LOGM, E>::LAST;
    extern __shared__ u64 sm[];
    const int tid = threadIdx.x, bm = blockIdx.x >> LS, h = blockIdx.x & ((1 << LS) - 1);
    const int nm = a.limbs + 1, b = bm / nm, m = bm % nm;
    const int mod = m < a.limbs ? m : a.L;
    const u64 q = a.rns.q[mod];
    const size_t part = (size_t)h << LOGM;
    u64 r[E];
#pragma unroll
    for (int e = 0; e < E; ++e) r[e] = 0;
    for (int j = 0; j < a.limbs; ++j) {
        const size_t key = ((((size_t)j * 2 + b) * (a.L + 1) + mod) << LOGN) + part;
        const u64* d = (j == m ? tensor + ((size_t)(2 * a.limbs + m) << LOGN) : digits + ((size_t)(j * nm + m) << LOGN)) + part;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int x = elem_index<LOGM, LAST, E>(tid, e);
            u64 v = d[x];
            if (j == m) v = shoup3(v, a.r64[m], a.r64_p[m], q);
            r[e] = halve<8>(r[e] + shoup3(v, __ldg(a.evk_hat + key + x), __ldg(a.evk_hat_p + key + x), q), q);
        }
    }
    if (m < a.limbs) {
        const u64* t = tensor + ((size_t)(b * a.limbs + m) << LOGN) + part;
#pragma unroll
        for (int e = 0; e < E; ++e)
            r[e] = halve<8>(r[e] + shoup3(t[elem_index<LOGM, LAST, E>(tid, e)], a.pn[m], a.pn_p[m], q), q);
    }
    ntt_inv_regs<LOGM, false, E, 8>(sm, r, tid, a.rns.tab[mod], q, (1 << LS) + h);
    u64* o = acc + ((size_t)bm << LOGN) + part;
#pragma unroll
    for (int e = 0; e < E; ++e) o[elem_index<LOGM, 0, E>(tid, e)] = r[e];
}

// out_b[j], j < t = limbs - 1: the last coupling stages of acc[b][P], acc[b][t] and acc[b][j], mod-down by P,
// rescale by q_t. One thread per (b, j) and R coefficients.
template <int LOGN>
__global__ void __launch_bounds__(128) k_relin_out(const __grid_constant__ SqImgArgs a, const u64* acc)
{
    constexpr int LS = kRelinLs<LOGN>, R = 1 << LS, M = 1 << (LOGN - LS);
    const int nm = a.limbs + 1, t = a.limbs - 1;
    const int b = blockIdx.y / t, j = blockIdx.y % t;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M) return;
    const u64 P = a.rns.q[a.L], halfP = (P - 1) / 2;
    u64 ap[R], lt[R], r[R];
    auto load = [&](int m, int mod, u64 (&v)[R]) {
#pragma unroll
        for (int k = 0; k < R; ++k) v[k] = acc[((size_t)(b * nm + m) << LOGN) + k * M + i];
        inv_tail<LS, 8>(v, a.rns.tab[mod].itw, a.rns.q[mod]);
    };
    auto mod_down = [&](u64 v, u64 p, int m) {   // (v - [p]_centered) P^{-1} mod q_m, v below 4 q_m
        const u64 q = a.rns.q[m];
        u64 lp = reduce64(p, q, a.rns.mu[m]);
        if (p > halfP) lp = add_mod(lp, a.neg_p_mod[m], q);
        return shoup(v + q - lp, a.p_inv[m], a.p_inv_p[m], q);
    };
    load(a.limbs, a.L, ap);
#pragma unroll
    for (int k = 0; k < R; ++k) ap[k] = below1<4>(ap[k], P);
    load(t, t, lt);
    load(j, j, r);
    const u64 q = a.rns.q[j];
    u64* o = a.out + ((size_t)(b * t + j) << LOGN) + i;
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const u64 ct = mod_down(lt[k], ap[k], t), cj = mod_down(r[k], ap[k], j);
        const u64 u = shoup_lazy(cj, a.qt_inv[j], a.qt_inv_p[j], q);
        const u64 w = shoup_lazy(ct, a.qt_inv[j], a.qt_inv_p[j], q);
        u64 v = csub_s(csub_s(u + 2 * q - w, 2 * q), q);
        if (ct > a.half_qt) v = add_mod(v, 1, q);
        o[k * M] = v;
    }
}

template <int LOGN>
static cudaError_t relin_launch(const SqImgArgs& a, const u64* tensor, u64* t2, u64* digits, u64* acc, cudaStream_t st)
{
    constexpr int LS = kRelinLs<LOGN>, R = 1 << LS, M = 1 << (LOGN - LS), T = M / 8;
    const size_t smem = (size_t)M * 8;
    const int limbs = a.limbs;
    k_relin_t2<LOGN><<<limbs * R, T, smem, st>>>(a, tensor + ((size_t)2 * limbs << LOGN), t2);
    k_relin_digits<LOGN><<<dim3((M + 127) / 128, limbs * limbs), 128, 0, st>>>(a, t2, digits);
    k_relin_fwd<LOGN><<<limbs * limbs * R, T, smem, st>>>(a, digits);
    k_relin_acc<LOGN><<<2 * (limbs + 1) * R, T, smem, st>>>(a, tensor, digits, acc);
    k_relin_out<LOGN><<<dim3((M + 127) / 128, 2 * (limbs - 1)), 128, 0, st>>>(a, acc);
    return cudaGetLastError();
}

cudaError_t launch_relin_rescale(const SqImgArgs& a, const u64* tensor, u64* t2, u64* digits, u64* acc, cudaStream_t st)
{
    switch (a.rns.logn) {
    case 10: return relin_launch<10>(a, tensor, t2, digits, acc, st);
    case 11: return relin_launch<11>(a, tensor, t2, digits, acc, st);
    case 12: return relin_launch<12>(a, tensor, t2, digits, acc, st);
    case 13: return relin_launch<13>(a, tensor, t2, digits, acc, st);
    case 14: return relin_launch<14>(a, tensor, t2, digits, acc, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace ichee
