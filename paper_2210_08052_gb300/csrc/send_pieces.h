// Host pieces that lie one after the other on the device, cut into windows and
// ranges of bytes wherever their ends are (host code only; see ctx_send_pieces).
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <cstring>

namespace mpdp {

// bytes of pinned memory that one window takes at most
constexpr uint64_t kSendWindow = 256ull << 20;

// `len` bytes at src, for the bytes [at, at + len) of the destination; pieces
// come in ascending order and do not overlap (there may be gaps).
struct CopyPiece {
    const char *src;
    uint64_t at, len;
};

// window(lo, hi) for every window of at most `limit` bytes of [0, total); stops
// at the first that returns anything but 0, and returns that.
template <typename Window>
inline int for_windows(uint64_t total, uint64_t limit, Window window)
{
    for (uint64_t lo = 0; lo < total; lo += limit) {
        const int rc = window(lo, std::min(total, lo + limit));
        if (rc) return rc;
    }
    return 0;
}

// The bytes [lo, hi) of the destination from the pieces, to out[0 .. hi - lo).
inline void gather_range(const CopyPiece *pieces, size_t n, uint64_t lo, uint64_t hi, char *out)
{
    // the first piece that can reach past lo: the last one that starts at or
    // before it (one after it that starts at lo as well is longer than none)
    size_t k = static_cast<size_t>(
        std::upper_bound(pieces, pieces + n, lo, [](uint64_t v, const CopyPiece &p) { return v < p.at; }) - pieces);
    for (k = k ? k - 1 : 0; k < n && pieces[k].at < hi; ++k) {
        const uint64_t a = std::max(pieces[k].at, lo), e = std::min(pieces[k].at + pieces[k].len, hi);
        if (a < e) memcpy(out + (a - lo), pieces[k].src + (a - pieces[k].at), e - a);
    }
}

}  // namespace mpdp
