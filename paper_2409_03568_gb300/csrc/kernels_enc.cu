// kernels_enc.cu -- key generation helpers, fused fresh encryption (Sec. 2.2.2, 3.1) and the
// cached encryption kernels (radix combine and value lookup with the zero pool, Sec. 3.2, 3.3).
#include "internal.h"
#include "ntt32.cuh"

namespace ichee {

// Shape of the fresh-encryption kernel. Up to N = 2^13: 8 residues per thread, both polynomials
// of a limb in lockstep (each twiddle loaded once for the two, exchanges in 64-bit words); at
// N = 2^14 (1024 threads, 16 residues) one polynomial at a time, as two take more than the 64
// registers. Blocks of up to 1024 threads in 64 registers a thread, as many per SM as that allows.
// 16 residues in 128 registers were slower at N = 2^13 (102 against 96 us per ciphertext and SM) and
// at 2^12 (61 against 51), as was a second set of samples drawn ahead (96.4 against 95.9).
template <int LOGN>
struct EncShape {
    static constexpr int N = 1 << LOGN;
    static constexpr int E = LOGN <= 13 ? 8 : 16;
    static constexpr int T = N / E;
    static constexpr int NP = LOGN <= 13 ? 2 : 1;
    static constexpr int KEEP = 2;   // v^ modulo two primes at a time
    static constexpr int BUFS = LOGN <= 13 ? 2 : 1;   // exchange buffers, used in turn (two do not fit at 2^14)
    static constexpr int BLOCKS = 1024 / T;
    static constexpr size_t CDT_AT = (size_t)N * (4 * NP * BUFS + 4 * KEEP + 2);
    static constexpr size_t SMEM = CDT_AT + 32 * sizeof(u64);
    static_assert(SMEM <= 227 * 1024 && BLOCKS * (SMEM + 1024) <= 228 * 1024, "shared memory of an SM");
};

// Word of the key operands for unit u, polynomial b, transform position x: both polynomials of a
// position adjacent where they are transformed together.
template <int LOGN>
__host__ __device__ constexpr size_t enc_pk_at(int u, int b, int x)
{
    return EncShape<LOGN>::NP == 2 ? (((size_t)u << LOGN) + x) * 2 + b : (((size_t)u * 2 + b) << LOGN) + x;
}

// ---------------------------------------------------------------------------------------
// Samplers (Sec. 2.2.1 / 2.2.2). Coefficient i of a ternary polynomial uses word i%4 of
// Philox block i/4; of a Gaussian one, words 2(i%2), 2(i%2)+1 of block i/2; of a uniform
// one, the four words of block i as a 128-bit x giving floor(x*q / 2^128).
// ---------------------------------------------------------------------------------------

__global__ void k_sample_small(int8_t* out, int n, u64 seed, u32 stream_id, u64 id, int gaussian, CdtTable cdt)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (gaussian) {
        Words4 w = philox(seed, stream_id, id, (u32)(i >> 1));
        int h = 2 * (i & 1);
        u64 u = (u64)w.w[h] | ((u64)w.w[h + 1] << 32);
        out[i] = (int8_t)gauss_of(u, cdt);
    } else {
        Words4 w = philox(seed, stream_id, id, (u32)(i >> 2));
        out[i] = (int8_t)ternary_of(w.w[i & 3]);
    }
}

__global__ void k_sample_uniform(u64* out, int n, u64 q, u64 seed, u32 stream_id, u64 id)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    Words4 w = philox(seed, stream_id, id, (u32)i);
    u64 lo = (u64)w.w[0] | ((u64)w.w[1] << 32);
    u64 hi = (u64)w.w[2] | ((u64)w.w[3] << 32);
    // floor((hi*2^64 + lo) * q / 2^128) = floor((hi*q + floor(lo*q / 2^64)) / 2^64)
    u64 carry = mulhi(lo, q);
    u64 t_lo = hi * q;
    u64 t_hi = mulhi(hi, q);
    u64 s = t_lo + carry;
    t_hi += (s < t_lo) ? 1 : 0;
    out[i] = t_hi;
}

cudaError_t launch_sample_small(int8_t* out, int n, u64 seed, u32 stream_id, u64 id, int gaussian,
                                const CdtTable& cdt, cudaStream_t st)
{
    k_sample_small<<<(n + 255) / 256, 256, 0, st>>>(out, n, seed, stream_id, id, gaussian, cdt);
    return cudaGetLastError();
}

cudaError_t launch_sample_uniform(u64* out, int n, u64 q, u64 seed, u32 stream_id, u64 id, cudaStream_t st)
{
    k_sample_uniform<<<(n + 255) / 256, 256, 0, st>>>(out, n, q, seed, stream_id, id);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Batched transforms in global memory (set-up paths and key switching).
// ---------------------------------------------------------------------------------------

template <int LOGN>
__global__ void __launch_bounds__(NttShape<LOGN>::T) k_ntt_fwd(const __grid_constant__ RnsArgs rns, const __grid_constant__ PolyBatch b)
{
    extern __shared__ u64 sm[];
    const int tid = threadIdx.x;
    const int m = b.midx[blockIdx.x % b.nl];
    const u64 q = rns.q[m];
    u64* d = b.data + (size_t)blockIdx.x * (1 << LOGN);
    u64 r[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) r[e] = d[elem_index<LOGN, 0>(tid, e)];
    ntt_fwd_regs<LOGN, false, 16, 8, 1>(sm, r, tid, rns.tab[m], q);
#pragma unroll
    for (int e = 0; e < 16; ++e) d[elem_index<LOGN, NttShape<LOGN>::LAST>(tid, e)] = below1<8>(r[e], q);
}

template <int LOGN>
__global__ void __launch_bounds__(NttShape<LOGN>::T) k_ntt_inv(const __grid_constant__ RnsArgs rns, const __grid_constant__ PolyBatch b)
{
    extern __shared__ u64 sm[];
    const int tid = threadIdx.x;
    const int m = b.midx[blockIdx.x % b.nl];
    const u64 q = rns.q[m];
    u64* d = b.data + (size_t)blockIdx.x * (1 << LOGN);
    u64 r[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) r[e] = d[elem_index<LOGN, NttShape<LOGN>::LAST>(tid, e)];
    ntt_inv_regs<LOGN, false, 16, 8>(sm, r, tid, rns.tab[m], q);
#pragma unroll
    for (int e = 0; e < 16; ++e) d[elem_index<LOGN, 0>(tid, e)] = below1<4>(r[e], q);
}

template <int LOGN>
static cudaError_t ntt_launch(bool fwd, const RnsArgs& rns, const PolyBatch& b, cudaStream_t st)
{
    const int T = NttShape<LOGN>::T;
    const size_t smem = sizeof(u64) << LOGN;
    auto kern = fwd ? k_ntt_fwd<LOGN> : k_ntt_inv<LOGN>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<b.n_poly, T, smem, st>>>(rns, b);
    return cudaGetLastError();
}

static cudaError_t ntt_dispatch(bool fwd, const RnsArgs& rns, const PolyBatch& b, cudaStream_t st)
{
    if (b.n_poly <= 0) return cudaSuccess;
    switch (rns.logn) {
    case 10: return ntt_launch<10>(fwd, rns, b, st);
    case 11: return ntt_launch<11>(fwd, rns, b, st);
    case 12: return ntt_launch<12>(fwd, rns, b, st);
    case 13: return ntt_launch<13>(fwd, rns, b, st);
    case 14: return ntt_launch<14>(fwd, rns, b, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_ntt_fwd(const RnsArgs& rns, const PolyBatch& b, cudaStream_t st) { return ntt_dispatch(true, rns, b, st); }
cudaError_t launch_ntt_inv(const RnsArgs& rns, const PolyBatch& b, cudaStream_t st) { return ntt_dispatch(false, rns, b, st); }

__global__ void k_pointwise_mul(RnsArgs rns, PolyBatch out, const u64* a, const u64* b, int b_period)
{
    const int n = 1 << rns.logn;
    const int p = blockIdx.y;
    const int m = out.midx[p % out.nl];
    const u64 q = rns.q[m];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        u64 x = a[(size_t)p * n + i];
        u64 y = b[(size_t)(p % b_period) * n + i];
        out.data[(size_t)p * n + i] = mul_mod(x, y, q, rns.m0[m], rns.m1[m]);
    }
}

cudaError_t launch_pointwise_mul(const RnsArgs& rns, const PolyBatch& out, const u64* a, const u64* b, int b_period,
                                 cudaStream_t st)
{
    dim3 grid((1u << rns.logn) / 256, out.n_poly);
    k_pointwise_mul<<<grid, 256, 0, st>>>(rns, out, a, b, b_period);
    return cudaGetLastError();
}

__global__ void k_scale_const(RnsArgs rns, PolyBatch b, const u64* cst)
{
    const int n = 1 << rns.logn;
    const int p = blockIdx.y;
    const int m = b.midx[p % b.nl];
    const u64 q = rns.q[m], c = cst[m];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        u64* x = b.data + (size_t)p * n + i;
        *x = mul_mod(*x, c, q, rns.m0[m], rns.m1[m]);
    }
}

cudaError_t launch_scale_const(const RnsArgs& rns, const PolyBatch& b, const u64* cst_per_mod, cudaStream_t st)
{
    dim3 grid((1u << rns.logn) / 256, b.n_poly);
    k_scale_const<<<grid, 256, 0, st>>>(rns, b, cst_per_mod);
    return cudaGetLastError();
}

// floor(w * 2^64 / q) by binary long division (w < q < 2^61)
__device__ u64 shoup_companion(u64 w, u64 q)
{
    u64 rem = w, quo = 0;
    for (int i = 0; i < 64; ++i) {
        rem <<= 1;
        quo <<= 1;
        if (rem >= q) { rem -= q; quo |= 1; }
    }
    return quo;
}

__global__ void k_shoup_companions(RnsArgs rns, PolyBatch b, u64* out)
{
    const int n = 1 << rns.logn;
    const int p = blockIdx.y;
    const u64 q = rns.q[b.midx[p % b.nl]];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        out[(size_t)p * n + i] = shoup_companion(b.data[(size_t)p * n + i], q);
}

cudaError_t launch_shoup_companions(const RnsArgs& rns, const PolyBatch& b, u64* out, cudaStream_t st)
{
    dim3 grid((1u << rns.logn) / 256, b.n_poly);
    k_shoup_companions<<<grid, 256, 0, st>>>(rns, b, out);
    return cudaGetLastError();
}

__global__ void k_small_to_mod(const int8_t* x, int n, u64 q, u64* out)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = small_mod(x[i], q);
}

cudaError_t launch_small_to_mod(const int8_t* x, int n, u64 q, u64* out, cudaStream_t st)
{
    k_small_to_mod<<<(n + 255) / 256, 256, 0, st>>>(x, n, q, out);
    return cudaGetLastError();
}

__global__ void k_neg_add_small(const u64* x, const int8_t* e, int n, u64 q, u64* out)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = add_mod(x[i] == 0 ? 0 : q - x[i], small_mod(e[i], q), q);
}

cudaError_t launch_neg_add_small(const u64* x, const int8_t* e, int n, u64 q, u64* out, cudaStream_t st)
{
    k_neg_add_small<<<(n + 255) / 256, 256, 0, st>>>(x, e, n, q, out);
    return cudaGetLastError();
}

__global__ void k_axpy_const(u64* out, const u64* x, const u64* y, u64 c, int n, u64 q, u64 m0, u64 m1)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = add_mod(x[i], mul_mod(c, y[i], q, m0, m1), q);
}

cudaError_t launch_axpy_const(u64* out, const u64* x, const u64* y, u64 c, int n, u64 q, u64 m0, u64 m1,
                              cudaStream_t st)
{
    k_axpy_const<<<(n + 255) / 256, 256, 0, st>>>(out, x, y, c, n, q, m0, m1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Operands of fresh encryption: the public key modulo the auxiliary primes, transformed. Unit u
// is a (limb l, prime i) pair (EncLimb::unit + i); block u writes
//   NTT_{p_i}(pk_b, centered modulo q_l) * (N^{-1} (M_l / p_i)^{-1} 2^32) mod p_i
// for both polynomials b, so that the Montgomery product with NTT(v) and the inverse transform
// leave the CRT digit [v pk_b (M_l / p_i)^{-1}] mod p_i. Set-up code, one launch per key.
// ---------------------------------------------------------------------------------------
template <int LOGN>
__global__ void __launch_bounds__(EncShape<LOGN>::T) k_pk_aux(const __grid_constant__ PkAuxArgs a)
{
    constexpr int N = 1 << LOGN, E = EncShape<LOGN>::E, LAST = NttShape<LOGN, E>::LAST;
    extern __shared__ u64 smem[];
    const int tid = threadIdx.x;
    int l = 0;
    while (l + 1 < a.L && (int)blockIdx.x >= a.unit[l + 1]) ++l;
    const int u = blockIdx.x, i = u - a.unit[l];
    const u64 q = a.q[l];
    const u32 p = a.aux.p[i], k = a.k[u];
    for (int b = 0; b < 2; ++b) {
        const u64* src = a.pk + ((size_t)b * a.L + l) * N;
        u32 r[1][E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const u64 c = src[elem_index<LOGN, 0, E>(tid, e)];
            const u32 m = (u32)((c > q / 2 ? q - c : c) % p);
            r[0][e] = c > q / 2 && m != 0 ? p - m : m;
        }
        if (b > 0) __syncthreads();   // two forward transforms in a row: the first one's last loads are over
        ntt32_fwd<LOGN, 1, E, false>(reinterpret_cast<u32*>(smem), r, tid, a.aux.tw[i], p, a.aux.zero);
#pragma unroll
        for (int e = 0; e < E; ++e)
            a.out[enc_pk_at<LOGN>(u, b, elem_index<LOGN, LAST, E>(tid, e))] = (u32)((u64)(r[0][e] % p) * k % p);
    }
}

template <int LOGN>
static cudaError_t pk_aux_launch(const PkAuxArgs& a, int n_units, cudaStream_t st)
{
    const size_t smem = sizeof(u32) << LOGN;
    cudaError_t e = cudaFuncSetAttribute(k_pk_aux<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_pk_aux<LOGN><<<n_units, EncShape<LOGN>::T, smem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_pk_aux(const PkAuxArgs& a, int logn, int n_units, cudaStream_t st)
{
    switch (logn) {
    case 10: return pk_aux_launch<10>(a, n_units, st);
    case 11: return pk_aux_launch<11>(a, n_units, st);
    case 12: return pk_aux_launch<12>(a, n_units, st);
    case 13: return pk_aux_launch<13>(a, n_units, st);
    case 14: return pk_aux_launch<14>(a, n_units, st);
    default: return cudaErrorInvalidValue;
    }
}

// ---------------------------------------------------------------------------------------
// Fused fresh encryption (Sec. 2.2.2, with the library sign convention pk = (-a*s + e, a),
// since the printed formulas do not cancel): one thread block per ciphertext.
//   sample v (ternary), e0, e1 (Gaussian) once into shared memory; v^_i = NTT(v) modulo each
//   auxiliary prime p_i once; then per limb l: c_b = [v pk_b] mod q_l + e_b (+ Delta*p at
//   coefficient 0 of c0).
// The product v pk_b is taken over the integers (pk_b centered, |coefficient| <= N q_l / 2) from
// its residues modulo the limb's first np primes: y_i = INTT(v^_i . pk^_{b,i}) are the CRT digits
// (the key operands carry 1/N and (M/p_i)^{-1}), and x = sum_i y_i M/p_i - k M with
// k = round(sum_i y_i / p_i) is reduced modulo q_l by one 32-bit quotient estimate (enc_crt).
// Three 64-bit transforms per limb become three 28-bit ones per ciphertext and four or six per limb
// (19 at N = 2^13 with primes 60/40/60), at about a fifth of the multiply-pipe time each. Measured
// against the 64-bit form: 4096 pixels at N = 2^13 3.03 -> 2.43 ms, 851 pixels at N = 2^14 and five
// limbs 3.34 -> 1.69 ms, 1224 pixels at N = 2^12 0.66 -> 0.39 ms (there also more than one block per
// SM). Bound by the integer multiply pipe (76 % busy), then by the exchanges between the passes.
// ---------------------------------------------------------------------------------------

// The sample word of a coefficient: v + 1 (bits 0-1), e0 + 32 (bits 2-7), e1 + 32 (bits 8-13).
__device__ __forceinline__ u32 enc_sample(int v, int e0, int e1)
{
    return (u32)(v + 1) | ((u32)(e0 + 32) << 2) | ((u32)(e1 + 32) << 8);
}

// A limb's residue of one coefficient from its CRT digits (y[np - 1] the last prime's), noise added
// (e_biased = e + 32): in [0, q). With k = round(sum y_i / p_i) the last digit less k times its
// prime makes sum y_i M/p_i the product itself; it is offset by 5 primes to stay positive, which
// lm.c0 takes back. The digits then sum to less than 2^30.6, so their products with the low and high
// words of M/p_i mod q add up in 64 bits each. Primes of at most 32 bits (SMALL) have no high words.
template <int NPR, bool SMALL>
__device__ __forceinline__ u64 enc_crt(const EncLimb& lm, u32 y0, u32 y1, u32 y2, u32 e_biased)
{
    u32 sum = y0 + y1;
    if constexpr (NPR == 3) sum += y2;
    const u32 k = (sum + (1u << (kAuxBits - 1))) >> kAuxBits;
    const u32 last = (NPR == 3 ? y2 : y1) + (5u - k) * lm.p_last;
    u64 lo = (lm.c0 + e_biased) + (u64)y0 * lm.ml[0];
    if constexpr (NPR == 3) lo += (u64)y1 * lm.ml[1];
    lo += (u64)last * lm.ml[NPR - 1];
    u32 T;   // floor(V / 2^(bits - 1)) < 2^32; the estimated quotient is short by less than 2.75
    if constexpr (SMALL) {
        T = (u32)(lo >> lm.t);
    } else {
        u64 hi = (u64)y0 * lm.mh[0];
        if constexpr (NPR == 3) hi += (u64)y1 * lm.mh[1];
        hi += (u64)last * lm.mh[NPR - 1];
        T = (u32)((hi + (lo >> 32)) >> lm.t);
        lo += hi << 32;
    }
    const u32 qhat = __umulhi(T, lm.mu);
    lo += (u64)qhat * lm.nq_lo;             // less qhat q modulo 2^64: [0, 2.75 q)
    lo += (u64)(qhat * lm.nq_hi) << 32;
    return csub_s(csub_s(lo, 2 * lm.q), lm.q);
}

// The block's share of a ciphertext: all limbs or, with SPLIT, limbs group, group + groups, ...
template <int LOGN, bool SPLIT>
__device__ __forceinline__ void encrypt_ct(const EncArgs& a, int group, int p, u64 seed, u64 id, u64* ct, u64* smem)
{
    using S = EncShape<LOGN>;
    constexpr int N = 1 << LOGN, E = S::E, T = S::T, NP = S::NP, LAST = NttShape<LOGN, E>::LAST;
    u32* ex = reinterpret_cast<u32*>(smem);                       // exchange buffers, N words of 4 NP bytes
    u32* vh = ex + S::BUFS * NP * N;                                        // v^ modulo S::KEEP primes, thread-major
    uint16_t* smp = reinterpret_cast<uint16_t*>(vh + S::KEEP * N);
    const u64* tcdt = reinterpret_cast<const u64*>(reinterpret_cast<unsigned char*>(smem) + S::CDT_AT);
    const int tid = threadIdx.x;
    const int L = a.L;
    __syncthreads();   // the previous ciphertext's samples no longer read
    for (int b = tid; b < N / 4; b += T) {         // coefficients 4b .. 4b + 3
        const Words4 wv = philox(seed, kStreamV, id, (u32)b);
        u32 packed[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const Words4 w0 = philox(seed, kStreamE0, id, (u32)(2 * b + h));
            const Words4 w1 = philox(seed, kStreamE1, id, (u32)(2 * b + h));
            const u32 lo = enc_sample(ternary_of(wv.w[2 * h]), gauss_of_sorted((u64)w0.w[0] | ((u64)w0.w[1] << 32), tcdt),
                                      gauss_of_sorted((u64)w1.w[0] | ((u64)w1.w[1] << 32), tcdt));
            const u32 hi = enc_sample(ternary_of(wv.w[2 * h + 1]),
                                      gauss_of_sorted((u64)w0.w[2] | ((u64)w0.w[3] << 32), tcdt),
                                      gauss_of_sorted((u64)w1.w[2] | ((u64)w1.w[3] << 32), tcdt));
            packed[h] = lo | (hi << 16);
        }
        reinterpret_cast<uint2*>(smp)[b] = make_uint2(packed[0], packed[1]);
    }

    const int x0 = elem_index<LOGN, 0, E>(tid, 0);       // first-pass layout: x0 + elem_offset(e)
    const int xl = elem_index<LOGN, LAST, E>(tid, 0);    // last-pass layout
    // Up to N = 2^13 the transforms alternate two exchange buffers and need no barrier between them: a
    // transform's exchanges make every warp wait, through the groups that trade data, for all others,
    // so a buffer's earlier loads are over when it is written again (checked for every ring in the
    // host-compiled test of the groups). One buffer and a block barrier before each transform: 2.3 %
    // slower.
    // First the third prime, for the limbs that need it: its digits wait in the output's own words
    // (each thread's coefficients of the ciphertext, which it overwrites with the residues below),
    // so that at most two primes' digits are in registers. Then the first two primes of every limb.
    int turn = 0;
    const int first = SPLIT ? group : 0, step = SPLIT ? a.groups : 1;
#pragma unroll 1
    for (int phase = a.aux.n == 3 ? 0 : 1; phase < 2; ++phase) {
        if (SPLIT && phase == 0 && !((a.third >> group) & 1u)) continue;
        const int i0 = phase == 0 ? 2 : 0, i1 = phase == 0 ? 3 : 2;
#pragma unroll 1
        for (int i = i0; i < i1; ++i) {
            __syncthreads();   // samples drawn; the exchange buffer's last readers are done
            u32 r[1][E];
#pragma unroll
            for (int e = 0; e < E; ++e) r[0][e] = (u32)((int)(smp[x0 + elem_offset<LOGN, 0, E>(e)] & 3u) - 1);
            ntt32_fwd<LOGN, 1, E, true>(ex + (S::BUFS == 2 ? turn * NP * N : 0), r, tid, a.aux.tw[i], a.aux.p[i],
                                        a.aux.zero);
            turn ^= 1;
#pragma unroll
            for (int e = 0; e < E; ++e) vh[(i - i0) * N + e * T + tid] = r[0][e];
        }
#pragma unroll 1
        for (int l = first; l < L; l += step) {
            const EncLimb& lm = a.limb[l];
            if (i0 >= lm.np) continue;
#pragma unroll 1
            for (int pb = 0; pb < 2; pb += NP) {
                u32 ya[NP][E], y[NP][E];   // digits modulo the first prime, and the current one
#pragma unroll 1
                for (int i = i0; i < i1; ++i) {
                    const u32 pi = a.aux.p[i], pinv = a.aux.pinv[i];
                    const u32* pk = a.pk_aux + enc_pk_at<LOGN>(lm.unit + i, pb, xl);
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        if (i == 1) {
#pragma unroll
                            for (int n = 0; n < NP; ++n) ya[n][e] = y[n][e];
                        }
                        const u32 v = vh[(i - i0) * N + e * T + tid];
                        const int o = elem_offset<LOGN, LAST, E>(e);
                        if constexpr (NP == 2) {
                            const uint2 w = __ldg(reinterpret_cast<const uint2*>(pk) + o);
                            y[0][e] = mont32(v, w.x, pi, pinv);
                            y[NP - 1][e] = mont32(v, w.y, pi, pinv);
                        } else {
                            y[0][e] = mont32(v, __ldg(pk + o), pi, pinv);
                        }
                    }
                    if (S::BUFS == 1) __syncthreads();
                    ntt32_inv<LOGN, NP, E>(ex + (S::BUFS == 2 ? turn * NP * N : 0), y, tid, a.aux.itw[i], pi,
                                           a.aux.zero);
                    turn ^= 1;
                }
                u64* dst = ct + ((u64)pb * L + l) * N + x0;
                if (phase == 0) {
#pragma unroll
                    for (int n = 0; n < NP; ++n)
#pragma unroll
                        for (int e = 0; e < E; ++e)
                            dst[(u64)n * L * N + elem_offset<LOGN, 0, E>(e)] = y[n][e];
                    continue;
                }
                auto write = [&](auto residue) {
#pragma unroll
                    for (int n = 0; n < NP; ++n)
#pragma unroll
                        for (int e = 0; e < E; ++e) {
                            const int x = elem_offset<LOGN, 0, E>(e);
                            u64* o = dst + (u64)n * L * N + x;
                            const u32 s = smp[x0 + x];
                            u64 v = residue(n, e, o, pb + n == 0 ? (s >> 2) & 63u : s >> 8);
                            if (pb + n == 0 && x == 0 && x0 == 0) v = add_mod(v, a.dm[l * 256 + p], lm.q);   // coefficient 0
                            __stcs(o, v);
                        }
                };
                if (lm.np == 3)
                    write([&](int n, int e, const u64* o, u32 eb) {
                        return enc_crt<3, false>(lm, ya[n][e], y[n][e], (u32)*o, eb);
                    });
                else if (lm.bits > 32)
                    write([&](int n, int e, const u64*, u32 eb) { return enc_crt<2, false>(lm, ya[n][e], y[n][e], 0, eb); });
                else
                    write([&](int n, int e, const u64*, u32 eb) { return enc_crt<2, true>(lm, ya[n][e], y[n][e], 0, eb); });
            }
        }
    }
}

template <int LOGN>
__device__ __forceinline__ void encrypt_setup(const EncArgs& a, u64* smem)
{
    cdt_for_search(a.cdt, reinterpret_cast<u64*>(reinterpret_cast<unsigned char*>(smem) + EncShape<LOGN>::CDT_AT));
    __syncthreads();
}

template <int LOGN, bool SPLIT>
__global__ void __launch_bounds__(EncShape<LOGN>::T, EncShape<LOGN>::BLOCKS)
    k_encrypt_fresh(const __grid_constant__ EncArgs a)
{
    extern __shared__ u64 smem[];
    encrypt_setup<LOGN>(a, smem);
    const u64 ct_len = (u64)2 * a.L << LOGN;
    // all pixels, or a listed subset (the misses of a value cache) shared evenly; one call site,
    // so the kernel holds one copy of the transform code
    const u64 n = a.idx != nullptr ? (u64)*a.n_idx : a.n_ct;
    for (u64 u = blockIdx.x; u < (SPLIT ? n * a.groups : n); u += gridDim.x) {
        const u64 g = SPLIT ? u / a.groups : u;
        const u64 k = a.idx != nullptr ? (u64)a.idx[g] : g;
        const int p = a.pixels[k];
        if (a.skip_lut != nullptr && a.skip_lut[p] >= 0) continue;  // uniform across the block
        encrypt_ct<LOGN, SPLIT>(a, SPLIT ? (int)(u % a.groups) : 0, p, a.seed, a.id_base + k, a.out + k * ct_len, smem);
    }
}

template <int LOGN>
__global__ void __launch_bounds__(EncShape<LOGN>::T, EncShape<LOGN>::BLOCKS)
    k_encrypt_fresh_batch(const __grid_constant__ EncArgs a, const __grid_constant__ SegTable t)
{
    extern __shared__ u64 smem[];
    encrypt_setup<LOGN>(a, smem);
    const u64 ct_len = (u64)2 * a.L << LOGN;
    const u64 total = t.start[t.n];
    for (u64 g = blockIdx.x; g < total; g += gridDim.x) {
        const int s = seg_of(t, g);
        const u64 k = g - t.start[s];
        const int p = t.px[s][k];
        if (a.skip_lut != nullptr && a.skip_lut[p] >= 0) continue;
        encrypt_ct<LOGN, false>(a, 0, p, t.seed[s], k, t.out[s] + k * ct_len, smem);
    }
}

// Persistent grid: the blocks that fit on the GPU at once, each walking its share of the
// ciphertexts. With pixels to skip in-kernel the shares would be uneven, so there more blocks than
// fit are launched.
template <int LOGN>
static unsigned enc_grid(const EncArgs& a, u64 n, int num_sms)
{
    const u64 cap = (u64)num_sms * EncShape<LOGN>::BLOCKS * (a.skip_lut != nullptr ? 16 : 1);
    return (unsigned)(n < cap ? n : cap);
}

template <int LOGN, bool SPLIT>
static cudaError_t enc_launch_as(const EncArgs& a, u64 n, cudaStream_t st)
{
    using S = EncShape<LOGN>;
    cudaError_t e = cudaFuncSetAttribute(k_encrypt_fresh<LOGN, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)S::SMEM);
    if (e != cudaSuccess) return e;
    k_encrypt_fresh<LOGN, SPLIT><<<enc_grid<LOGN>(a, n, a.num_sms), S::T, S::SMEM, st>>>(a);
    return cudaGetLastError();
}

// Fewer than half as many ciphertexts as SMs (a cache's tables, a thumbnail): the limbs of each are
// shared out over blocks, as long as every block has an SM to itself. Each block draws the samples and
// transforms v again, but the limbs, most of the work, run side by side.
// Measured, 3 limbs at N = 2^13: 38 ciphertexts 96.8 -> 51.8 us, 64 in two groups 96.9 -> 78.5; 5 limbs
// at 2^14: 290 -> 113 and 204; 2 limbs at 2^10: 19.0 -> 14.7. With two blocks to an SM it gains little
// or loses (4 limbs at 2^10, 304 ciphertexts: 35.4 -> 45.9; 3 at 2^12, 110: 53.7 -> 74.2), so the line
// is one block to an SM. A kernel of its own: run-time groups in the general one cost it 1 %.
template <int LOGN>
static cudaError_t enc_launch(EncArgs a, cudaStream_t st)
{
    const u64 fit = (u64)a.num_sms / a.n_ct;
    a.groups = fit < (u64)a.L ? (int)fit : a.L;
    if (a.groups < 2) return enc_launch_as<LOGN, false>(a, a.n_ct, st);
    a.third = 0;
    for (int l = 0; l < a.L; ++l)
        if (a.limb[l].np == 3) a.third |= 1u << (l % a.groups);
    return enc_launch_as<LOGN, true>(a, a.n_ct * a.groups, st);
}

template <int LOGN>
static cudaError_t enc_batch_launch(EncArgs a, const SegTable& t, int num_sms, cudaStream_t st)
{
    using S = EncShape<LOGN>;
    cudaError_t e = cudaFuncSetAttribute(k_encrypt_fresh_batch<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)S::SMEM);
    if (e != cudaSuccess) return e;
    const unsigned grid = enc_grid<LOGN>(a, t.start[t.n], num_sms);
    k_encrypt_fresh_batch<LOGN><<<grid, S::T, S::SMEM, st>>>(a, t);
    return cudaGetLastError();
}

cudaError_t launch_encrypt_fresh_batch(const EncArgs& a, const SegTable& t, int num_sms, cudaStream_t st)
{
    if (t.n <= 0 || t.start[t.n] == 0) return cudaSuccess;
    switch (a.logn) {
    case 10: return enc_batch_launch<10>(a, t, num_sms, st);
    case 11: return enc_batch_launch<11>(a, t, num_sms, st);
    case 12: return enc_batch_launch<12>(a, t, num_sms, st);
    case 13: return enc_batch_launch<13>(a, t, num_sms, st);
    case 14: return enc_batch_launch<14>(a, t, num_sms, st);
    default: return cudaErrorInvalidValue;
    }
}

__global__ void k_miss_list(const uint8_t* px, u64 n, const int32_t* lut, u32* idx, u32* count)
{
    for (u64 k = blockIdx.x * (u64)blockDim.x + threadIdx.x; k < n; k += (u64)gridDim.x * blockDim.x)
        if (lut[px[k]] < 0) idx[atomicAdd(count, 1u)] = (u32)k;
}

cudaError_t launch_miss_list(const uint8_t* px, u64 n, const int32_t* lut, u32* idx, u32* count, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(count, 0, sizeof(u32), st);
    if (e != cudaSuccess || n == 0) return e;
    const u64 blocks = (n + 255) / 256;
    k_miss_list<<<(unsigned)(blocks < 1024 ? blocks : 1024), 256, 0, st>>>(px, n, lut, idx, count);
    return cudaGetLastError();
}

cudaError_t launch_encrypt_fresh(const EncArgs& a, cudaStream_t st)
{
    if (a.n_ct == 0) return cudaSuccess;
    switch (a.logn) {
    case 10: return enc_launch<10>(a, st);
    case 11: return enc_launch<11>(a, st);
    case 12: return enc_launch<12>(a, st);
    case 13: return enc_launch<13>(a, st);
    case 14: return enc_launch<14>(a, st);
    default: return cudaErrorInvalidValue;
    }
}

// ---------------------------------------------------------------------------------------
// Cached encryption.
// ---------------------------------------------------------------------------------------

// M[k][d + r] = d * Enc(r^k) mod q for d in [-r, r]: the multiples a radix combine can ask
// for. Repeated homomorphic addition of a ciphertext (Sec. 3.2) equals this scalar multiple
// residue for residue, so tabulating it once per cache changes no result.
__global__ void k_radix_multiples(const u64* cts, int n_pow, int r, RnsArgs rns, int L, u64* mult)
{
    const int n = 1 << rns.logn;
    const size_t ct_len = (size_t)2 * L * n;
    const int slot = blockIdx.y;            // kk * (2r+1) + (d + r)
    const int kk = slot / (2 * r + 1);
    const int d = slot % (2 * r + 1) - r;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < ct_len; i += (size_t)gridDim.x * blockDim.x) {
        const int l = (int)((i / n) % L);
        const u64 q = rns.q[l];
        const u64 c = cts[kk * ct_len + i];
        mult[slot * ct_len + i] = mul_mod(c, small_mod(d, q), q, rns.m0[l], rns.m1[l]);
    }
}

cudaError_t launch_radix_multiples(const u64* radix_cts, int n_pow, int r, const RnsArgs& rns, int L, u64* mult,
                                       cudaStream_t st)
{
    dim3 grid(64, n_pow * (2 * r + 1));
    k_radix_multiples<<<grid, 256, 0, st>>>(radix_cts, n_pow, r, rns, L, mult);
    return cudaGetLastError();
}

// P[i][j] = M[n-2][i] + M[n-1][j + r] mod q (i = d + r for d in [-r, r], j in [0, pair_w)): the
// top two positions' multiples summed once per cache, so a combine reads one cached ciphertext
// for both. Modular addition is exact, so every output residue is unchanged.
__global__ void k_radix_pairs(const u64* mult, int n_pow, int r, int pair_w, RnsArgs rns, int L, u64* pair)
{
    const int n = 1 << rns.logn;
    const size_t ct_len = (size_t)2 * L * n;
    const int width = 2 * r + 1;
    const int slot = blockIdx.y;            // i * pair_w + j
    const int i = slot / pair_w, j = slot % pair_w;
    const u64* lo = mult + ((size_t)(n_pow - 2) * width + i) * ct_len;
    const u64* hi = mult + ((size_t)(n_pow - 1) * width + j + r) * ct_len;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < ct_len; e += (size_t)gridDim.x * blockDim.x)
        pair[slot * ct_len + e] = add_mod(lo[e], hi[e], rns.q[(e / n) % L]);
}

cudaError_t launch_radix_pairs(const u64* mult, int n_pow, int r, int pair_w, const RnsArgs& rns, int L, u64* pair,
                               cudaStream_t st)
{
    dim3 grid(64, (2 * r + 1) * pair_w);
    k_radix_pairs<<<grid, 256, 0, st>>>(mult, n_pow, r, pair_w, rns, L, pair);
    return cudaGetLastError();
}

// Radix combine: one block per ciphertext. Signed digits d'_k = d_k + b_k - r*b_{k+1} with b
// from bit k of the pixel's randomness word (stream 3); c = sum_k M[k][d'_k], residue-wise
// modular sums of cached rows (the top two positions' from the pair table when the cache has
// one), 16-byte loads, streaming 16-byte stores.
__device__ __forceinline__ void radix_ct(const RadixArgs& a, int p, u64 seed, u64 id, u64* ct)
{
    const int n = 1 << a.logn;
    const size_t ct_len = (size_t)2 * a.L * n;
    const int width = 2 * a.r + 1;
    u32 bits = 0;
    if (a.randomize) bits = philox(seed, kStreamRadixBits, id, 0).w[0];
    const u64* src[8];
    int ns = 0;
    int rest = p;
    int dig[8];
    for (int kk = 0; kk < a.n_pow; ++kk) {
        int dk = rest % a.r;
        rest /= a.r;
        int bk = (a.randomize && kk >= 1) ? (int)((bits >> kk) & 1u) : 0;
        int bk1 = (a.randomize && kk + 1 < a.n_pow) ? (int)((bits >> (kk + 1)) & 1u) : 0;
        dig[kk] = dk + bk - a.r * bk1;
    }
    const int separate = a.pair_w ? a.n_pow - 2 : a.n_pow;
    for (int kk = 0; kk < separate; ++kk)
        if (dig[kk] != 0) src[ns++] = a.mult + ((size_t)kk * width + (dig[kk] + a.r)) * ct_len;
    if (a.pair_w && (dig[separate] != 0 || dig[separate + 1] != 0))
        src[ns++] = a.pair + ((size_t)(dig[separate] + a.r) * a.pair_w + dig[separate + 1]) * ct_len;
    // Row by row (one modulus per row); four coefficient pairs per thread and round, their
    // loads issued together.
    ulonglong2* dst = reinterpret_cast<ulonglong2*>(ct);
    const int half = n / 2;
    for (int row = 0; row < 2 * a.L; ++row) {
        const u64 q = a.q[row % a.L];
        const size_t base = (size_t)row * half;
        for (int i0 = threadIdx.x; i0 < half; i0 += 4 * blockDim.x) {
            ulonglong2 acc[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[u] = make_ulonglong2(0, 0);
            for (int s = 0; s < ns; ++s) {
                const ulonglong2* sp = reinterpret_cast<const ulonglong2*>(src[s]) + base;
                ulonglong2 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = i0 + u * blockDim.x;
                    v[u] = i < half ? __ldg(sp + i) : make_ulonglong2(0, 0);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    acc[u].x = add_mod(acc[u].x, v[u].x, q);
                    acc[u].y = add_mod(acc[u].y, v[u].y, q);
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + u * blockDim.x;
                if (i < half) __stcs(dst + base + i, acc[u]);
            }
        }
    }
}

__global__ void __launch_bounds__(256) k_radix_combine(const __grid_constant__ RadixArgs a)
{
    const size_t ct_len = (size_t)2 * a.L << a.logn;
    for (u64 k = blockIdx.x; k < a.n_ct; k += gridDim.x) {
        const int p = a.pixels[k];
        if (a.skip_lut != nullptr && a.skip_lut[p] >= 0) continue;
        radix_ct(a, p, a.seed, a.id_base + k, a.out + k * ct_len);
    }
}

__global__ void __launch_bounds__(1024) k_radix_combine_batch(const __grid_constant__ RadixArgs a,
                                                              const __grid_constant__ SegTable t)
{
    const size_t ct_len = (size_t)2 * a.L << a.logn;
    const u64 total = t.start[t.n];
    for (u64 g = blockIdx.x; g < total; g += gridDim.x) {
        const int s = seg_of(t, g);
        const u64 k = g - t.start[s];
        const int p = t.px[s][k];
        if (a.skip_lut != nullptr && a.skip_lut[p] >= 0) continue;
        radix_ct(a, p, t.seed[s], k, t.out[s] + k * ct_len);
    }
}

cudaError_t launch_radix_combine(const RadixArgs& a, cudaStream_t st)
{
    if (a.n_ct == 0) return cudaSuccess;
    unsigned grid = (unsigned)(a.n_ct < (1u << 30) ? a.n_ct : (1u << 30));
    k_radix_combine<<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

// Value lookup with the randomness pool: c = C[lut[p]] (+) Z[idx], idx = floor(w*M / 2^32)
// from stream 4. Pixels whose value is not cached are left to another kernel.
// One row (polynomial b, limb l: row = b L + l) of one pixel's ciphertext. The work is
// ordered row-major -- row 0 of every pixel, then row 1, ... -- so that while a row is being
// written only that row of the cached ciphertexts and of the pool is read: 256 x N x 8 bytes
// (16 MB at N = 8192) plus the pool's, which stays in L2 even when the whole cache does not.
__device__ __forceinline__ void lookup_row(const LookupArgs& a, int slot, u64 seed, u64 id, u64* ct, int row)
{
    const int n = 1 << a.logn;
    const int half = n / 2;
    const size_t ct_len = (size_t)2 * a.L * n;
    const size_t base = (size_t)row * half;
    const ulonglong2* c = reinterpret_cast<const ulonglong2*>(a.value_cts + (size_t)slot * ct_len) + base;
    const ulonglong2* z = nullptr;
    if (a.pool_size > 0) {
        u32 w = philox(seed, kStreamPool, id, 0).w[0];
        u32 idx = (u32)(((u64)w * a.pool_size) >> 32);
        z = reinterpret_cast<const ulonglong2*>(a.pool + (size_t)idx * ct_len) + base;
    }
    ulonglong2* dst = reinterpret_cast<ulonglong2*>(ct) + base;
    const u64 q = a.q[row % a.L];
    // four coefficient pairs per thread and round, their loads issued together
    for (int i0 = threadIdx.x; i0 < half; i0 += 4 * blockDim.x) {
        ulonglong2 v[4], w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * blockDim.x;
            v[u] = i < half ? __ldg(c + i) : make_ulonglong2(0, 0);
            w[u] = (i < half && z != nullptr) ? __ldg(z + i) : make_ulonglong2(0, 0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * blockDim.x;
            if (i >= half) continue;
            if (z != nullptr) {
                v[u].x = add_mod(v[u].x, w[u].x, q);
                v[u].y = add_mod(v[u].y, w[u].y, q);
            }
            __stcs(dst + i, v[u]);
        }
    }
}

// Work item g = row * n_ct + pixel.
__global__ void __launch_bounds__(256) k_lookup_combine(const __grid_constant__ LookupArgs a)
{
    const size_t ct_len = (size_t)2 * a.L << a.logn;
    const u64 items = a.n_ct * 2 * a.L;
    for (u64 g = blockIdx.x; g < items; g += gridDim.x) {
        const int row = (int)(g / a.n_ct);
        const u64 k = g % a.n_ct;
        const int slot = a.lut[a.pixels[k]];
        if (slot < 0) continue;
        lookup_row(a, slot, a.seed, a.id_base + k, a.out + k * ct_len, row);
    }
}

// Work item g = row * total + (pixel item of the batch), rows outermost across all segments.
__global__ void __launch_bounds__(1024) k_lookup_combine_batch(const __grid_constant__ LookupArgs a,
                                                               const __grid_constant__ SegTable t)
{
    const size_t ct_len = (size_t)2 * a.L << a.logn;
    const u64 total = t.start[t.n];
    const u64 items = total * 2 * a.L;
    for (u64 gg = blockIdx.x; gg < items; gg += gridDim.x) {
        const int row = (int)(gg / total);
        const u64 g = gg % total;
        const int s = seg_of(t, g);
        const u64 k = g - t.start[s];
        const int slot = a.lut[t.px[s][k]];
        if (slot < 0) continue;
        lookup_row(a, slot, t.seed[s], k, t.out[s] + k * ct_len, row);
    }
}

static unsigned persistent_grid(u64 total, LaunchShape ls, int num_sms)
{
    // blocks_per_sm = 0: one block per work item (no grid-stride loop), capped at 2^31 - 1
    const u64 cap = ls.blocks_per_sm > 0 ? (u64)num_sms * ls.blocks_per_sm : 0x7fffffffull;
    return (unsigned)(total < cap ? total : cap);
}

cudaError_t launch_radix_combine_batch(const RadixArgs& a, const SegTable& t, LaunchShape ls, int num_sms,
                                       cudaStream_t st)
{
    const u64 total = t.n > 0 ? t.start[t.n] : 0;
    if (total == 0) return cudaSuccess;
    k_radix_combine_batch<<<persistent_grid(total, ls, num_sms), ls.threads, 0, st>>>(a, t);
    return cudaGetLastError();
}

cudaError_t launch_lookup_combine_batch(const LookupArgs& a, const SegTable& t, LaunchShape ls, int num_sms,
                                        cudaStream_t st)
{
    const u64 total = t.n > 0 ? t.start[t.n] : 0;
    if (total == 0) return cudaSuccess;
    k_lookup_combine_batch<<<persistent_grid(total * 2 * a.L, ls, num_sms), ls.threads, 0, st>>>(a, t);
    return cudaGetLastError();
}

cudaError_t launch_lookup_combine(const LookupArgs& a, cudaStream_t st)
{
    if (a.n_ct == 0) return cudaSuccess;
    const u64 items = a.n_ct * 2 * a.L;
    unsigned grid = (unsigned)(items < (1u << 30) ? items : (1u << 30));
    k_lookup_combine<<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

__global__ void k_histogram(const uint8_t* px, u64 n, u32* counts)
{
    __shared__ u32 h[256];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) h[i] = 0;
    __syncthreads();
    for (u64 i = blockIdx.x * (u64)blockDim.x + threadIdx.x; i < n; i += (u64)gridDim.x * blockDim.x)
        atomicAdd(&h[px[i]], 1u);
    __syncthreads();
    for (int i = threadIdx.x; i < 256; i += blockDim.x)
        if (h[i]) atomicAdd(&counts[i], h[i]);
}

cudaError_t launch_histogram(const uint8_t* pixels, u64 n, u32* counts, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    unsigned grid = (unsigned)((n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024);
    k_histogram<<<grid, 256, 0, st>>>(pixels, n, counts);
    return cudaGetLastError();
}

}  // namespace ichee
