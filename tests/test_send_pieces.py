"""Host pieces cut into windows and ranges for the device
(csrc/send_pieces.h), compiled for the host: no window is longer than the
pinned memory it may take, whatever the pieces' lengths, and the ranges of the
windows hold the pieces' bytes."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_08052_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include <string>
#include <vector>
#include "send_pieces.h"
using namespace mpdp;
int main()
{
    // one long piece among short ones (sizes alone)
    for (uint64_t total : {uint64_t{0}, uint64_t{1}, kSendWindow, kSendWindow + 1, uint64_t{5} << 30}) {
        uint64_t at = 0;
        const int rc = for_windows(total, kSendWindow, [&](uint64_t lo, uint64_t hi) {
            if (lo != at || hi <= lo || hi - lo > kSendWindow) return 1;
            at = hi;
            return 0;
        });
        if (rc || at != total) { std::printf("windows of %llu\n", static_cast<unsigned long long>(total)); return 1; }
    }
    if (for_windows(10, 3, [](uint64_t lo, uint64_t) { return lo == 3 ? 7 : 0; }) != 7) return 1;
    uint32_t seed = 3;
    auto next = [&](uint32_t m) { return (seed = seed * 1664525u + 1013904223u) / 65536u % m; };
    for (int rep = 0; rep < 300; ++rep) {
        std::vector<std::string> text(1 + next(9));
        std::vector<CopyPiece> p;
        std::string all;
        for (auto &t : text) {
            const uint32_t len = next(4) == 0 ? 0 : next(3) == 0 ? next(200) : next(5);      // empty, long, short
            for (uint32_t k = 0; k < len; ++k) t += static_cast<char>('a' + next(26));
            p.push_back(CopyPiece{t.data(), all.size(), t.size()});
            all += t;
            if (next(5) == 0) all += "..";                                                  // a gap
        }
        for (uint64_t limit : {uint64_t{1}, uint64_t{2}, uint64_t{7}, uint64_t{64}, uint64_t{1000}}) {
            std::string got(all.size(), '.');
            for_windows(all.size(), limit, [&](uint64_t lo, uint64_t hi) {
                const uint64_t mid = lo + (hi - lo) / 2;
                gather_range(p.data(), p.size(), lo, mid, &got[lo]);
                gather_range(p.data(), p.size(), mid, hi, &got[mid]);
                return 0;
            });
            if (got != all) { std::printf("rep %d limit %d\n", rep, static_cast<int>(limit)); return 1; }
        }
    }
    return 0;
}
"""


def test_windows_and_ranges(tmp_path):
    src, exe = tmp_path / "pieces.cpp", tmp_path / "pieces"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=address", "-I" + CSRC, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
