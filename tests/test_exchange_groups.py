"""The barriers of the transforms' exchanges (csrc/ntt.cuh, exchange_barrier): host-compiled, for every
ring and both register widths. Every word a thread loads in an exchange was stored by a thread of
its own barrier group; a group has exactly the threads its barrier counts; groups of one transform
never share a barrier number, and all numbers are below 16. For the kernels that alternate two
exchange buffers without a barrier between transforms: after a transform's exchanges every warp has
(through the groups, step by step) waited for every other one."""
import os
import subprocess

import pytest

from test_ntt_layout import CSRC, ROOT, nvcc

CHECK = r'''
#include "ntt.cuh"
#include <cstdio>
#include <map>
#include <set>
#include <vector>
using namespace ichee;
static int group_of(int fixed, int warp)
{
    int g = 0, bit = 0;
    for (int i = 0; i < 5; ++i)
        if ((fixed >> i) & 1) g |= ((warp >> i) & 1) << bit++;
    return g;
}
template <int E> static int check(int logn)
{
    const int le = E == 16 ? 4 : 3, n = 1 << logn, T = n / E, W = T / 32;
    int bad = 0;
    std::map<int, std::set<int>> used;   // barrier number -> pass it serves
    // known[w]: the warps w has (transitively) waited for, forward order; the same set of groups in reverse
    std::vector<std::set<int>> fwd(W), inv(W);
    for (int w = 0; w < W; ++w) fwd[w] = inv[w] = {w};
    std::vector<std::vector<std::vector<int>>> steps;
    for (int s = le; s < logn; s += le) {
        const int a = s - le;
        if (exchange_in_warp(logn, a, s, E)) continue;
        const int fixed = exchange_fixed_bits(logn, a, s, E), groups = 1 << bits_of(fixed);
        std::vector<int> writer(n);
        for (int t = 0; t < T; ++t)
            for (int e = 0; e < E; ++e) writer[elem_index_of(logn, a, E, t, e)] = t;
        std::vector<std::vector<int>> members(groups);
        for (int w = 0; w < W; ++w) members[fixed ? group_of(fixed, w) : 0].push_back(w);
        for (auto& m : members)
            if ((int)m.size() * 32 != T / groups) ++bad;
        for (int t = 0; t < T; ++t)
            for (int e = 0; e < E; ++e) {
                const int wr = writer[elem_index_of(logn, s, E, t, e)];
                const int back = t;   // inverse direction: the thread that stores what wr loads
                if (fixed && group_of(fixed, wr >> 5) != group_of(fixed, back >> 5)) ++bad;
            }
        if (fixed)
            for (int g = 0; g < groups; ++g) {
                const int id = exchange_first_id(logn, s, E) + g;
                if (id < 1 || id > 15) ++bad;
                used[id].insert(s);
            }
        steps.push_back(members);
    }
    for (auto& u : used)
        if (u.second.size() != 1) ++bad;
    auto run = [&](std::vector<std::set<int>>& known, bool reverse) {
        for (size_t i = 0; i < steps.size(); ++i)
            for (auto& m : steps[reverse ? steps.size() - 1 - i : i]) {
                std::set<int> all;
                for (int w : m) all.insert(known[w].begin(), known[w].end());
                for (int w : m) known[w] = all;
            }
        for (int w = 0; w < W; ++w)
            if ((int)known[w].size() != W) ++bad;
    };
    run(fwd, false);
    run(inv, true);
    return bad;
}
int main()
{
    int bad = 0;
    for (int logn = 8; logn <= 13; ++logn) bad += check<8>(logn);   // from 8: the parts of relinearisation's transforms
    for (int logn = 10; logn <= 14; ++logn) bad += check<16>(logn);
    printf("bad %d\n", bad);
    return bad != 0;
}
'''


def test_exchange_groups(tmp_path):
    cc = nvcc()
    if cc is None:
        pytest.skip("nvcc not found")
    src = tmp_path / "groups.cu"
    src.write_text(CHECK)
    exe = tmp_path / "groups"
    r = subprocess.run([cc, "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
