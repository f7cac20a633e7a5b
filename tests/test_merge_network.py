"""The sorting network of the index's full buckets (csrc/merge_network.h),
compiled for the host: it sorts any number of places, and its steps end for
every 32-bit count (a genome with more than 2^29 bases that are not A, C, G or
T puts more than 2^30 entries into one bucket)."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_08052_gb300", "csrc")

SOURCE = r"""
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "merge_network.h"
struct TooMany {};
int main()
{
    uint32_t seed = 1;
    for (uint32_t n = 0; n < 1100; n += n < 70 ? 1 : 103)
        for (int rep = 0; rep < 3; ++rep) {
            std::vector<uint32_t> v(n), w;
            for (auto &x : v) x = (seed = seed * 1664525u + 1013904223u) >> (rep == 2 ? 29 : 4);
            w = v;
            std::sort(w.begin(), w.end());
            mpdp::network_steps(n, [&](uint32_t j) {
                for (uint32_t i = 0; i < n; ++i) {
                    const uint32_t l = i ^ j;
                    if (l > i && l < n && v[i] > v[l]) std::swap(v[i], v[l]);
                }
            });
            if (v != w) { std::printf("not sorted: %u\n", n); return 1; }
        }
    const uint32_t large[] = {513u, 1u << 20, (1u << 30) - 1, 1u << 30, (1u << 30) + 1, 1u << 31, (1u << 31) + 1, ~0u};
    for (uint32_t n : large) {
        uint64_t steps = 0, levels = 0;
        while ((1ull << levels) < n) ++levels;
        try {
            mpdp::network_steps(n, [&](uint32_t) { if (++steps > 1000) throw TooMany(); });
        } catch (TooMany &) {
        }
        if (steps != levels * (levels + 1) / 2) {
            std::printf("%u: %llu steps\n", n, static_cast<unsigned long long>(steps));
            return 1;
        }
    }
    return 0;
}
"""


def test_network_sorts_and_ends(tmp_path):
    src, exe = tmp_path / "network.cpp", tmp_path / "network"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
