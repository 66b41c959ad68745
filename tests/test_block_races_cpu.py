"""Kernels that run several transforms through one shared buffer, run on the CPU from their own source
with every thread a fiber: block, group and warp barriers are the only places where a warp stops, and
the warp that runs on is the first one able to in a given order (ascending, descending, shuffled).
A word that a warp stores before another warp has loaded the one it replaces then changes the result,
which on the GPU happens only by chance. Covered, for every ring: the key operands of fresh encryption
(against a textbook transform), fresh encryption (whole ciphertexts, limbs shared out, batched),
matching's accumulation and the per-pixel squared difference (the same words for every order)."""
import os
import re
import shutil
import subprocess

import pytest

from test_ntt_layout import CSRC, ROOT, nvcc

# What the device code takes from the compiler and the hardware, and the scheduler.
SHIM = r'''
#pragma once
#include <cuda_runtime.h>
#include <ucontext.h>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <vector>
#undef __launch_bounds__
#define __launch_bounds__(...)
#undef __grid_constant__
#define __grid_constant__
#undef __forceinline__
#define __forceinline__ inline
namespace emu {
struct Fiber { ucontext_t at; int wait = -2; };   // waiting for: -2 nothing, -1 its warp, else a barrier
static std::vector<Fiber> fibers;
static std::vector<char> stacks;
static ucontext_t home;
static int current, n_threads;
static std::map<int, int> arrived;
static uint3 block;
static dim3 grid;
inline void stop(int what)
{
    fibers[current].wait = what;
    swapcontext(&fibers[current].at, &home);
}
inline void bar(int id, int count)
{
    const int me = current;
    if (++arrived[id] == count) {
        arrived[id] = 0;
        for (int t = 0; t < n_threads; ++t)
            if (t != me && fibers[t].wait == id) fibers[t].wait = -2;
    } else {
        stop(id);
    }
}
static void* body;
template <class F> static void enter()
{
    (*static_cast<F*>(body))();
    stop(1 << 20);   // done
}
// One block: `order` lists the warps, the first able to run runs until none of its lanes can.
template <class F> bool run_block(int threads, int b, int blocks, const std::vector<int>& order, F f)
{
    const size_t kStack = 1 << 16;
    n_threads = threads;
    block = make_uint3(b, 0, 0);
    grid = dim3(blocks);
    arrived.clear();
    fibers.assign(threads, Fiber());
    body = &f;
    stacks.resize(kStack * threads);
    for (int t = 0; t < threads; ++t) {
        getcontext(&fibers[t].at);
        fibers[t].at.uc_stack.ss_sp = stacks.data() + kStack * t;
        fibers[t].at.uc_stack.ss_size = kStack;
        fibers[t].at.uc_link = nullptr;
        makecontext(&fibers[t].at, enter<F>, 0);
    }
    for (;;) {
        bool ran = false, done = true;
        for (int w : order) {
            int at_warp = 0;
            for (int t = 32 * w; t < 32 * w + 32; ++t) {
                if (fibers[t].wait == -2) {
                    current = t;
                    swapcontext(&home, &fibers[t].at);
                    ran = true;
                }
                at_warp += fibers[t].wait == -1;
                done = done && fibers[t].wait == 1 << 20;
            }
            if (at_warp == 32) {
                for (int t = 32 * w; t < 32 * w + 32; ++t) fibers[t].wait = -2;
                ran = true;
            }
            if (ran) break;
        }
        if (done && !ran) return true;
        if (!ran) return false;   // every warp waits
    }
}
}  // namespace emu
#define threadIdx (make_uint3(emu::current, 0, 0))
#define blockIdx (emu::block)
#define blockDim (dim3(emu::n_threads))
#define gridDim (emu::grid)
inline void __syncthreads() { emu::bar(0, emu::n_threads); }
inline void __syncwarp() { emu::stop(-1); }
inline uint64_t __umul64hi(uint64_t a, uint64_t b) { return (uint64_t)((unsigned __int128)a * b >> 64); }
inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)((uint64_t)a * b >> 32); }
inline uint32_t __viaddmin_u32(uint32_t a, uint32_t b, uint32_t c) { const uint32_t s = a + b; return s < c ? s : c; }
template <class T> inline T __ldg(const T* p) { return *p; }
template <class T> inline T __ldcs(const T* p) { return *p; }
template <class T> inline void __stcs(T* p, T v) { *p = v; }
namespace ichee {
template <class F> cudaError_t cudaFuncSetAttribute(F*, cudaFuncAttribute, int) { return cudaSuccess; }
}
inline unsigned atomicAdd(unsigned* p, unsigned v) { const unsigned o = *p; *p += v; return o; }
'''

COMMON = r'''
#include "shim.h"
#include "host_math.h"
#include "internal.h"
#include <algorithm>
#include <random>
using namespace ichee;
namespace hm = ichee::host;
static std::mt19937_64 rng(1);
static std::vector<u64> random_words(size_t n, u64 q)
{
    std::vector<u64> v(n);
    for (u64& x : v) x = rng() % q;
    return v;
}
static std::vector<std::vector<int>> orders(int warps)
{
    std::vector<int> up(warps);
    for (int i = 0; i < warps; ++i) up[i] = i;
    std::vector<int> down(up.rbegin(), up.rend()), mixed = up;
    std::shuffle(mixed.begin(), mixed.end(), rng);
    return {up, down, mixed};
}
static void poison();   // other words into shared memory
// `go` runs every block of a launch in one order and fills in its result; all orders must agree.
template <class F> static int agree(int threads, const char* what, int logn, F go)
{
    std::vector<u64> first;
    for (const auto& o : orders(threads / 32)) {
        std::vector<u64> out;
        poison();
        if (!go(o, out)) return std::printf("%s N = 2^%d: every warp waits\n", what, logn), 1;
        if (first.empty()) first = out;
        if (out != first) return std::printf("%s N = 2^%d: depends on the order of the warps\n", what, logn), 1;
    }
    return 0;
}
'''

ENC = COMMON + r'''
#include "kernels_enc_host.h"
namespace ichee { u64 smem[1 << 15], sm[1 << 14]; }
static void poison() { for (u64& w : smem) w = rng(); }
static AuxPrimes aux;
static std::vector<uint2> aux_tables[3];
static std::vector<u64> dm(4 * 256);
template <int LOGN> static int check()
{
    constexpr u64 N = 1ull << LOGN;
    using S = EncShape<LOGN>;
    std::vector<u64> taken, pairs(4 * N);
    aux.n = 3;
    for (int i = 0; i < 3; ++i) {
        const u64 p = hm::chain_prime(kAuxBits, LOGN, taken);
        taken.push_back(p);
        aux.p[i] = aux.pinv[i] = (u32)p;
        for (int it = 0; it < 5; ++it) aux.pinv[i] *= 2u - (u32)p * aux.pinv[i];
        hm::twiddle_pairs(p, LOGN, pairs.data());
        aux_tables[i].resize(2 * N);
        for (u64 k = 0; k < 2 * N; ++k) aux_tables[i][k] = make_uint2((u32)pairs[2 * k], (u32)(pairs[2 * k + 1] >> 32));
        aux.tw[i] = aux_tables[i].data();
        aux.itw[i] = aux.tw[i] + N;
    }
    // key operands, one limb of three primes, against a textbook transform
    const u64 q = hm::chain_prime(60, LOGN, {});
    const std::vector<u64> pk = random_words(2 * N, q);
    PkAuxArgs a = {};
    a.aux = aux;
    a.L = 1;
    a.q[0] = q;
    a.pk = pk.data();
    for (int u = 0; u < 3; ++u) a.k[u] = 12345 + u;
    std::vector<u32> want(6 * N), got(6 * N);
    for (int u = 0; u < 3; ++u)
        for (int b = 0; b < 2; ++b) {
            const u64 p = aux.p[u];
            std::vector<u64> x(N);
            for (u64 i = 0; i < N; ++i) {
                const u64 c = pk[b * N + i];
                x[i] = c > q / 2 ? (p - (q - c) % p) % p : c % p;
            }
            for (u64 m = 1, t = N / 2; m < N; m *= 2, t /= 2)
                for (u64 i = 0; i < m; ++i)
                    for (u64 j = 2 * i * t; j < 2 * i * t + t; ++j) {
                        const u64 w = x[j + t] * aux.tw[u][m + i].x % p, v = x[j];
                        x[j] = (v + w) % p;
                        x[j + t] = (v + p - w) % p;
                    }
            for (u64 i = 0; i < N; ++i) want[enc_pk_at<LOGN>(u, b, (int)i)] = (u32)(x[i] * a.k[u] % p);
        }
    a.out = got.data();
    for (const auto& o : orders(S::T / 32))
        for (int u = 0; u < 3; ++u)
            if (!emu::run_block(S::T, u, 3, o, [&] { k_pk_aux<LOGN>(a); }) ||
                !std::equal(got.begin() + 2 * u * N, got.begin() + 2 * (u + 1) * N, want.begin() + 2 * u * N))
                return std::printf("key operands N = 2^%d, unit %d\n", LOGN, u), 1;
    // fresh encryption: limbs of two and three primes (any constants that depend on every digit)
    EncArgs e = {};
    e.logn = LOGN;
    e.L = 3;
    e.aux = aux;
    std::vector<u32> key(8 * 2 * N);
    for (u32& k : key) k = (u32)(rng() % aux.p[2]);
    for (int l = 0; l < 3; ++l) {
        EncLimb& lm = e.limb[l];
        lm.q = q;
        lm.np = l == 1 ? 3 : 2;
        lm.unit = l == 0 ? 0 : l == 1 ? 2 : 5;
        lm.bits = 60;
        lm.t = 27;
        lm.p_last = aux.p[lm.np - 1];
        for (int i = 0; i < lm.np; ++i) lm.ml[i] = (u32)rng() | 1, lm.mh[i] = (u32)rng() >> 5;
    }
    const uint8_t px[2] = {7, 200};
    e.n_ct = 2;
    e.pixels = px;
    e.dm = dm.data();
    e.pk_aux = key.data();
    e.seed = 5;
    hm::gauss_cdt(3.2, 19, e.cdt.t);
    e.cdt.bound = 19;
    int bad = 0;
    auto whole = [&](int kind) {
        return [&, kind](const std::vector<int>& o, std::vector<u64>& out) {
            out.assign(2 * 6 * N, 0);
            EncArgs x = e;
            x.out = out.data();
            x.groups = 2;
            x.third = 1u << 1;
            SegTable t = {};
            t.n = 1;
            t.start[1] = 2;
            t.px[0] = px;
            t.out[0] = out.data();
            const int blocks = kind == 1 ? 2 : 1;   // a block takes two ciphertexts (shared out: two shares)
            for (int b = 0; b < blocks; ++b)
                if (!emu::run_block(S::T, b, blocks, o, [&] {
                        if (kind == 0) k_encrypt_fresh<LOGN, false>(x);
                        else if (kind == 1) k_encrypt_fresh<LOGN, true>(x);
                        else k_encrypt_fresh_batch<LOGN>(x, t);
                    }))
                    return false;
            return true;
        };
    };
    const char* names[] = {"fresh", "fresh by limbs", "fresh batch"};
    for (int kind = 0; kind < 3; ++kind) bad += agree(S::T, names[kind], LOGN, whole(kind));
    return bad;
}
int main() { return check<10>() + check<11>() + check<12>() + check<13>() + check<14>() != 0; }
'''

MATCH = COMMON + r'''
#include "kernels_match_host.h"
namespace ichee { u64 buf[1 << 15], sm[1 << 15]; }
static void poison() { for (u64 i = 0; i < 1 << 15; ++i) buf[i] = rng(), sm[i] = rng(); }
template <int LOGN> static int check()
{
    constexpr u64 N = 1ull << LOGN;
    constexpr int limbs = 2;
    RnsArgs rns = {};
    rns.logn = LOGN;
    rns.n_mod = 3;
    std::vector<u64> taken, tables[3];
    for (int m = 0; m < 3; ++m) {
        const u64 q = hm::chain_prime(m == 0 ? 60 : m == 1 ? 40 : 61, LOGN, taken);
        taken.push_back(q);
        rns.q[m] = q;
        rns.mu[m] = (u64)(((hm::u128)1 << 64) / q);
        u64 inv = q;
        for (int it = 0; it < 6; ++it) inv *= 2 - q * inv;
        rns.qinv[m] = 0 - inv;
        tables[m].resize(4 * N);
        hm::twiddle_pairs(q, LOGN, tables[m].data());
        rns.tab[m].tw = reinterpret_cast<const ulonglong2*>(tables[m].data());
        rns.tab[m].itw = reinterpret_cast<const ulonglong2*>(tables[m].data() + 2 * N);
    }
    const std::vector<u64> x = random_words(2 * 2 * limbs * N, rns.q[1]), y = random_words(2 * 2 * limbs * N, rns.q[1]);
    SqDiffArgs s = {};
    s.rns = rns;
    s.limbs = limbs;
    s.n_ct = 2;
    s.a = x.data();
    s.b = y.data();
    s.n_blocks = sqdiff_split(LOGN) ? 2 * limbs : limbs;   // a block takes both pairs
    constexpr int TA = NttShape<LOGN == 14 ? 13 : LOGN, 8>::T;
    int bad = agree(TA, "matching", LOGN, [&](const std::vector<int>& o, std::vector<u64>& out) {
        out.assign((size_t)s.n_blocks * 4 * N, 0);
        s.partial = out.data();
        for (int b = 0; b < s.n_blocks; ++b)
            if (!emu::run_block(TA, b, s.n_blocks, o, [&] {
                    if constexpr (LOGN == 14) k_sqdiff_accumulate_split(s);
                    else k_sqdiff_accumulate<LOGN, 8>(s);
                }))
                return false;
        return true;
    });
    const std::vector<u64> key = random_words(2 * 2 * 3 * N, rns.q[1]);
    SqImgArgs g = {};
    g.rns = rns;
    g.L = g.limbs = limbs;
    g.n_ct = 2;
    g.a = x.data();
    g.b = y.data();
    g.evk_hat = g.evk_hat_p = key.data();
    for (int l = 0; l < limbs; ++l) {
        g.pn[l] = g.ninv[l] = g.r64[l] = g.p_inv[l] = g.qt_inv[l] = 12345 + l;
        g.pn_p[l] = g.ninv_p[l] = g.r64_p[l] = g.p_inv_p[l] = g.qt_inv_p[l] = hm::shoup_of(12345 + l, rns.q[l]);
    }
    std::vector<u64> scratch(sqdiff_image_scratch_words(LOGN, limbs));
    g.scratch = scratch.data();
    constexpr int E = kSqImgE<LOGN>, TI = NttShape<LOGN, E>::T;
    bad += agree(TI, "per pixel", LOGN, [&](const std::vector<int>& o, std::vector<u64>& out) {
        out.assign(2 * 2 * (limbs - 1) * N, 0);
        g.out = out.data();
        return emu::run_block(TI, 0, 1, o, [&] { k_sqdiff_image<LOGN, E>(g); });
    });
    return bad;
}
int main() { return check<10>() + check<11>() + check<12>() + check<13>() + check<14>() != 0; }
'''

BAR = 'asm volatile("bar.sync %0, %1;" ::"r"(first + group), "n"(T / groups) : "memory");'


def run_on_host(name, main, tmp_path):
    """Compile `main` for the CPU, with the shim and the source of csrc/<name>.cu (launches cut out) as
    <name>_host.h, and run it; a failure shows what it printed."""
    cxx, cc = shutil.which("g++"), nvcc()
    if cxx is None or cc is None:
        pytest.skip("g++ or the CUDA headers not found")
    for f in os.listdir(CSRC):
        if not f.endswith((".h", ".cuh")):
            continue
        text = open(os.path.join(CSRC, f)).read()
        if f == "ntt.cuh":
            assert text.count(BAR) == 1
            text = text.replace(BAR, "emu::bar(first + group, T / groups);")
        (tmp_path / f).write_text(text)
    kernels = open(os.path.join(CSRC, name + ".cu")).read()
    (tmp_path / (name + "_host.h")).write_text(re.sub(r"<<<.*?>>>", "", kernels, flags=re.S))
    (tmp_path / "shim.h").write_text(SHIM)
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(main)
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(cc))), "include")
    r = subprocess.run([cxx, "-O1", "-std=c++17", "-w", "-I", str(tmp_path), "-isystem", include, "-I",
                        os.path.join(ROOT, "include"), "-Wl,--unresolved-symbols=ignore-all", "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-4000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("name,main", [("kernels_enc", ENC), ("kernels_match", MATCH)], ids=["encryption", "matching"])
def test_results_do_not_depend_on_the_order_of_the_warps(name, main, tmp_path):
    run_on_host(name, main, tmp_path)
