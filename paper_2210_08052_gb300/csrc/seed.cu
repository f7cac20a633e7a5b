// Seeding and chaining on the GPU (Li 2022, Methods: "Reduced alphabet",
// "Indexing the genome", "Chaining").  Hand-written for sm_103a.
//
// Index: both strands of the genome as independent sequences, each in three
// reading frames; every open reading frame (a maximal run of codons without
// a stop codon) of at least 30 amino acids; every 6-mer inside one whose
// hash psi(phi(6-mer)) has lowest bit 0 is stored as strand << 31 | bin,
// bin = floor(x / 256) with x the k-mer's first base on its strand.  The
// table is CSR over all 2^24 hash values, each value's entries ascending.
//
//   translate_kernel   reduced-alphabet code of every codon of the six frames
//   segment_kernel     per 1024-codon segment: its first and last stop codon
//   segment_scan       per frame: the nearest stop before and after each segment
//   kmer_kernel        per segment (one warp): run bounds of every codon from the
//                      stops, the sampled k-mers of long runs, counted (pass 0)
//                      or written at their bucket's cursor (pass 1)
//   scan kernels       exclusive prefix sums (bucket counts -> CSR offsets)
//   bucket_sort_kernel each bucket's entries in ascending order
//
// Chaining, per protein (a block each, four warps to a strand): its k-mers'
// hits as anchors (strand, x = bin, y = residue), sorted; the recurrence of Eq. 2 with the
// gap of Eq. 1 and the penalty of Eq. 3 (G = 200,000, beta = 0.75) in fixed
// point with 16 fractional bits (the log term from a table of every |g| < G),
// 32 anchors at a time, one per lane (see chain_dp); then the chains in order
// of decreasing score of their last anchor.
//
// Second round, per (protein, region) pair: every 5-mer of the protein
// (reduced alphabet, sorted in shared memory) against the 5-mer starting at
// every base of the region's aligned strand, by a filter and a binary search
// (one block per pair, the region in tiles, contiguous bases per thread, so the
// anchors come out in (x, y) order), counted then written; chained by one warp
// per pair, or eight, with g' = 3 dy - dx and Eq. 3.
#include <algorithm>
#include <climits>
#include <cstdint>
#include <cstring>
#include <vector>

#include "merge_network.h"
#include "mp_internal.cuh"

namespace mpdp {
namespace {

constexpr int kK = 6;                       // k-mer length (amino acids)
constexpr int kKeyBits = 4 * kK;            // 24-bit codes
constexpr uint32_t kNKeys = 1u << kKeyBits;
constexpr int kBin = 256;
constexpr int kMinOrf = 30;
constexpr int64_t kG = 200000;              // largest gap (bp) of a chain link
constexpr int64_t kScale = 65536;           // chaining scores in units of 2^-16
constexpr int kSeg = 1024;                  // codons per segment
constexpr uint8_t kStopCode = 14;           // phi of a stop codon
constexpr uint8_t kXCode = 15;

// The reduced alphabet ("Reduced alphabet"): A 0, ST 1, RK 2, H 3, ND 4,
// EQ 5, C 6, P 7, G 8, IV 10, LM 11, FY 12, W 13, stop 14, anything else 15.
constexpr uint8_t phi_letter(char c)
{
    return c == 'A' ? 0 : (c == 'S' || c == 'T') ? 1 : (c == 'R' || c == 'K') ? 2 : c == 'H' ? 3
         : (c == 'N' || c == 'D') ? 4 : (c == 'E' || c == 'Q') ? 5 : c == 'C' ? 6 : c == 'P' ? 7
         : c == 'G' ? 8 : (c == 'I' || c == 'V') ? 10 : (c == 'L' || c == 'M') ? 11
         : (c == 'F' || c == 'Y') ? 12 : c == 'W' ? 13 : c == '*' ? 14 : 15;
}

// NCBI table 1 with codons enumerated as A, C, G, T in each position.
constexpr char kCodonAA[] = "KNKNTTTTRSRSIIMIQHQHPPPPRRRRLLLLEDEDAAAAGGGGVVVV*Y*YSSSS*CWCLFLF";

struct Table64 {
    uint8_t v[64];
};
struct Table256 {
    uint8_t v[256];
};
constexpr Table64 make_codon_phi()
{
    Table64 t{};
    for (int k = 0; k < 64; ++k) t.v[k] = phi_letter(kCodonAA[k]);
    return t;
}
constexpr Table256 make_aa_phi()
{
    Table256 t{};
    for (int c = 0; c < 256; ++c) t.v[c] = phi_letter(static_cast<char>(c >= 'a' && c <= 'z' ? c - 32 : c));
    return t;
}

// phi of each codon (bases in A, C, G, T order) and of each protein letter
__constant__ Table64 c_codon_phi = make_codon_phi();
__constant__ Table256 c_aa_phi = make_aa_phi();

__device__ __forceinline__ int base_code(unsigned char c)
{
    switch (c | 0x20) {
    case 'a': return 0;
    case 'c': return 1;
    case 'g': return 2;
    case 't': return 3;
    default: return -1;
    }
}

// psi: Thomas Wang's integer mix with every step modulo 2^24 (a bijection
// of [0, 2^24), the invertible hash the paper cites from minimap)
__device__ __forceinline__ uint32_t psi24(uint32_t key)
{
    const uint64_t mask = (1ull << kKeyBits) - 1;
    uint64_t k = key & mask;
    k = (~k + (k << 21)) & mask;
    k = k ^ k >> 24;
    k = (k + (k << 3) + (k << 8)) & mask;
    k = k ^ k >> 14;
    k = (k + (k << 2) + (k << 4)) & mask;
    k = k ^ k >> 28;
    k = (k + (k << 31)) & mask;
    return static_cast<uint32_t>(k);
}

// frame fr = 3 * strand + frame of the index's six frames
struct Frames {
    uint8_t *code[6];          // phi of codon t of each frame
    uint64_t len[6];           // codons per frame
    uint64_t seg0[7];          // first segment index of each frame (segments are numbered across frames)
};

// Reduced-alphabet code of every codon of every frame.  Codon t of frame f
// of strand 1 is the reverse complement's bases f + 3t .. f + 3t + 2, i.e.
// the complements of genome[n-1-(f+3t)], genome[n-2-(f+3t)], genome[n-3-(f+3t)].
//
// A block takes kTransTile codons of all three frames of one strand
// (blockIdx.y): the bases are read and coded once into shared memory, and four
// neighbouring codons of a frame leave in one store (the frames' arrays start
// on 16 bytes).  A thread per codon, with three byte loads, a search of its
// frame and a table in constant memory read at 32 places, took 0.83 ms on 50
// Mb; this 0.25.
constexpr int kTransThreads = 256, kTransTile = 4 * kTransThreads;
__global__ void __launch_bounds__(kTransThreads) translate_kernel(const char *g, uint64_t n, Frames fr)
{
    __shared__ uint8_t base[3 * kTransTile + 4];
    __shared__ uint8_t s_phi[64];
    const int strand = blockIdx.y;
    for (int k = threadIdx.x; k < 64; k += blockDim.x) s_phi[k] = c_codon_phi.v[k];
    for (uint64_t t0 = blockIdx.x * static_cast<uint64_t>(kTransTile); t0 < fr.len[3 * strand];
         t0 += gridDim.x * static_cast<uint64_t>(kTransTile)) {
        __syncthreads();
        for (int i = threadIdx.x; i < 3 * kTransTile + 2; i += blockDim.x) {
            const uint64_t x = 3 * t0 + i;
            const int c = x < n ? base_code(static_cast<unsigned char>(strand ? g[n - 1 - x] : g[x])) : -1;
            base[i] = static_cast<uint8_t>(c < 0 ? 4 : strand ? 3 - c : c);
        }
        __syncthreads();
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            const uint64_t t = t0 + 4 * threadIdx.x, len = fr.len[3 * strand + f];
            const uint8_t *b = base + f + 12 * threadIdx.x;
            uint32_t w = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int b0 = b[3 * k], b1 = b[3 * k + 1], b2 = b[3 * k + 2];
                w |= static_cast<uint32_t>((b0 | b1 | b2) & 4 ? kXCode : s_phi[b0 * 16 + b1 * 4 + b2]) << (8 * k);
            }
            uint8_t *out = fr.code[3 * strand + f] + t;
            if (t + 4 <= len) *reinterpret_cast<uint32_t *>(out) = w;
            else
                for (int k = 0; t + k < len && k < 4; ++k) out[k] = static_cast<uint8_t>(w >> (8 * k));
        }
    }
}

// per segment: first and last stop codon (frame-relative index), or -1
__global__ void segment_kernel(Frames fr, int64_t *first, int64_t *last, uint64_t nseg)
{
    const int lane = threadIdx.x & 31;
    for (uint64_t s = (blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x) >> 5; s < nseg;
         s += (static_cast<uint64_t>(gridDim.x) * blockDim.x) >> 5) {
        int f = 0;
        while (s >= fr.seg0[f + 1]) ++f;
        const uint64_t t0 = (s - fr.seg0[f]) * kSeg, len = fr.len[f];
        int64_t lo = -1, hi = -1;
        for (int c = 0; c < kSeg; c += 32) {
            const uint64_t t = t0 + c + lane;
            const bool stop = t < len && fr.code[f][t] == kStopCode;
            const unsigned bal = __ballot_sync(0xffffffffu, stop);
            if (bal) {
                if (lo < 0) lo = static_cast<int64_t>(t0 + c + __ffs(bal) - 1);
                hi = static_cast<int64_t>(t0 + c + 31 - __clz(bal));
            }
        }
        if (lane == 0) {
            first[s] = lo;
            last[s] = hi;
        }
    }
}

// per frame (one block of kScanThreads each): for every segment, the last
// stop codon before it (-1 if none) and the first after it (the frame's
// length if none): each thread reduces a contiguous range of segments, the
// block scans the thread totals, each thread then walks its range again
constexpr int kScanThreads = 1024;

__global__ void __launch_bounds__(kScanThreads) segment_scan(Frames fr, const int64_t *first, const int64_t *last,
                                                              int64_t *before, int64_t *after)
{
    __shared__ int64_t red[kScanThreads];
    const int f = blockIdx.x;
    const uint64_t s0 = fr.seg0[f], s1 = fr.seg0[f + 1], ns = s1 - s0;
    const uint64_t per = (ns + kScanThreads - 1) / kScanThreads;
    const uint64_t ta = threadIdx.x * per, tb = (threadIdx.x + 1) * per;
    const uint64_t a = s0 + (ta < ns ? ta : ns), b = s0 + (tb < ns ? tb : ns);
    // forward: the last stop of the ranges before this thread's
    int64_t mx = -1;
    for (uint64_t s = a; s < b; ++s) mx = last[s] > mx ? last[s] : mx;
    red[threadIdx.x] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t run = -1;
        for (int t = 0; t < kScanThreads; ++t) {
            const int64_t v = red[t];
            red[t] = run;
            run = v > run ? v : run;
        }
    }
    __syncthreads();
    int64_t cur = red[threadIdx.x];
    for (uint64_t s = a; s < b; ++s) {
        before[s] = cur;
        if (last[s] >= 0) cur = last[s];
    }
    __syncthreads();
    // backward: the first stop of the ranges after this thread's
    const int64_t none = static_cast<int64_t>(fr.len[f]);
    int64_t mn = none;
    for (uint64_t s = a; s < b; ++s)
        if (first[s] >= 0 && first[s] < mn) mn = first[s];
    red[threadIdx.x] = mn;
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t run = none;
        for (int t = kScanThreads - 1; t >= 0; --t) {
            const int64_t v = red[t];
            red[t] = run;
            run = v < run ? v : run;
        }
    }
    __syncthreads();
    cur = red[threadIdx.x];
    for (uint64_t s = b; s > a; --s) {
        after[s - 1] = cur;
        if (first[s - 1] >= 0) cur = first[s - 1];
    }
}

// One warp per segment.  For codon t of a run [a, b) (a after a stop or at
// the frame's start, b at the next stop or the frame's end) with b - a >=
// kMinOrf and t + kK <= b, the k-mer code of codons t .. t+5 is hashed; a
// sampled one (lowest bit 0) is counted in its bucket (pass 0) or written at
// its bucket's cursor (pass 1).  The segment's codes are read once into shared
// memory; lane c keeps the stops of the segment's codons 32c .. 32c + 31 as a
// bit mask and the last stop before and the first after them, from which the
// run of any codon follows (a table of both per codon, filled in two sweeps,
// left room for 28 warps per SM: 0.75 and 1.17 ms on 50 Mb; this 0.20 and
// 0.49).
constexpr int kKmerWarps = 8;

__global__ void __launch_bounds__(kKmerWarps * 32) kmer_kernel(Frames fr, const int64_t *before, const int64_t *after,
                                                               uint64_t nseg, int pass, uint32_t *count,
                                                               uint32_t *cursor, uint32_t *entries)
{
    __shared__ alignas(16) uint8_t seg[kKmerWarps][kSeg + 16];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    static_assert(kSeg == 32 * 32, "a word of stops per lane");
    for (uint64_t s = blockIdx.x * static_cast<uint64_t>(kKmerWarps) + w; s < nseg;
         s += static_cast<uint64_t>(gridDim.x) * kKmerWarps) {
        int f = 0;
        while (s >= fr.seg0[f + 1]) ++f;
        const uint64_t t0 = (s - fr.seg0[f]) * kSeg, len = fr.len[f];
        const uint8_t *code = fr.code[f] + t0;
        const int cnt = static_cast<int>(len - t0 < kSeg ? len - t0 : kSeg);               // codons of the segment
        // and what its k-mers touch
        const int more = static_cast<int>(len - t0 < kSeg + kK - 1 ? len - t0 : kSeg + kK - 1);
        __syncwarp();
        if (cnt == kSeg) {
            // (the frames' arrays start on 16 bytes and a segment is a multiple of them)
            const uint4 *src = reinterpret_cast<const uint4 *>(code);
            reinterpret_cast<uint4 *>(seg[w])[lane] = src[lane];
            reinterpret_cast<uint4 *>(seg[w])[lane + 32] = src[lane + 32];
            if (kSeg + lane < more) seg[w][kSeg + lane] = code[kSeg + lane];
        } else {
            for (int t = lane; t < more; t += 32) seg[w][t] = code[t];
        }
        __syncwarp();
        // stops of this lane's 32 codons
        uint32_t mine = 0;
        for (int c = 0; c < 32; ++c) {
            const int t = c * 32 + lane;
            const unsigned bal = __ballot_sync(0xffffffffu, t < cnt && seg[w][t] == kStopCode);
            if (c == lane) mine = bal;
        }
        // the last stop before them and the first after (codons of the segment;
        // -1 and kSeg: none in it)
        int last = mine ? lane * 32 + 31 - __clz(mine) : -1, first = mine ? lane * 32 + __ffs(mine) - 1 : kSeg;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, last, o), z = __shfl_down_sync(0xffffffffu, first, o);
            if (lane >= o) last = max(last, y);
            if (lane + o < 32) first = min(first, z);
        }
        last = __shfl_up_sync(0xffffffffu, last, 1);
        first = __shfl_down_sync(0xffffffffu, first, 1);
        if (lane == 0) last = -1;
        if (lane == 31) first = kSeg;
        // as distances from the segment's first codon, clamped to what decides
        // (a run that leaves the segment by kMinOrf is long enough, by kK goes on)
        const int64_t far_b = before[s] - static_cast<int64_t>(t0), far_a = after[s] - static_cast<int64_t>(t0);
        const int out_b = static_cast<int>(far_b < -1 - kMinOrf ? -1 - kMinOrf : far_b);
        const int out_a = static_cast<int>(far_a > kSeg + kMinOrf ? kSeg + kMinOrf : far_a);
        if (last < 0) last = out_b;
        if (first >= kSeg) first = out_a;
        const uint32_t strand = f / 3, frame = f % 3;
        for (int c = 0; c < 32; ++c) {
            const uint32_t m = __shfl_sync(0xffffffffu, mine, c);
            const int lc = __shfl_sync(0xffffffffu, last, c), fc = __shfl_sync(0xffffffffu, first, c);
            const int t = c * 32 + lane;
            if (t >= cnt || (m >> lane & 1)) continue;
            const uint32_t below = m & ((1u << lane) - 1), above = lane == 31 ? 0u : m & ~((2u << lane) - 1);
            const int a = (below ? c * 32 + 31 - __clz(below) : lc) + 1, b = above ? c * 32 + __ffs(above) - 1 : fc;
            if (b - a < kMinOrf || t + kK > b) continue;
            uint32_t key = 0;
#pragma unroll
            for (int u = 0; u < kK; ++u) key = key * 16 + seg[w][t + u];
            const uint32_t h = psi24(key);
            if (h & 1u) continue;
            if (pass == 0) {
                atomicAdd(count + h, 1u);
            } else {
                const uint32_t at = atomicAdd(cursor + h, 1u);
                entries[at] = (strand << 31) | static_cast<uint32_t>((frame + 3 * (t0 + t)) / kBin);
            }
        }
    }
}

// ---- exclusive prefix sum of n uint32 counts into n + 1 uint32 offsets
constexpr int kScanBlock = 1024;

__global__ void scan_blocks(const uint32_t *in, uint64_t n, uint32_t *out, uint32_t *block_sums)
{
    __shared__ uint32_t warp_tot[32];
    const uint64_t base = static_cast<uint64_t>(blockIdx.x) * kScanBlock * 4;
    uint32_t v[4], s = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const uint64_t i = base + threadIdx.x * 4 + u;
        v[u] = i < n ? in[i] : 0u;
        s += v[u];
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t incl = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    if (w == 0) {
        uint32_t t = warp_tot[lane], ti = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, ti, o);
            if (lane >= o) ti += y;
        }
        warp_tot[lane] = ti - t;
        if (lane == 31) block_sums[blockIdx.x] = ti;
    }
    __syncthreads();
    uint32_t run = warp_tot[w] + incl - s;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const uint64_t i = base + threadIdx.x * 4 + u;
        if (i < n) out[i] = run;
        run += v[u];
    }
}

__global__ void scan_sums(uint32_t *block_sums, uint32_t nb, uint32_t *total)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        uint32_t run = 0;
        for (uint32_t b = 0; b < nb; ++b) {
            const uint32_t v = block_sums[b];
            block_sums[b] = run;
            run += v;
        }
        *total = run;
    }
}

__global__ void scan_add(uint32_t *out, uint64_t n, const uint32_t *block_sums, const uint32_t *total)
{
    const uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x;
    if (i < n) out[i] += block_sums[i / (kScanBlock * 4)];
    if (i == 0) out[n] = *total;
}

// Each bucket's entries in ascending order.  A warp takes 32 neighbouring
// buckets, whose entries are contiguous: in shared memory, each entry's place
// is the number of its bucket's entries before it (one lane per entry; 32
// buckets hold 34 on average on the 50 Mb genome, 340 on 500 Mb, where a fifth
// of them, with 57% of the entries, have more than fit).
// Where they do not fit, the warp sorts bucket by bucket in place (the network
// of merge_network.h).  One thread per bucket, by insertion in global memory,
// took 2.4 ms on the 50 Mb genome; this 0.46 (the whole index of 50 Mb 6.5 ->
// 2.8 ms, of 120 Mb 21.5 -> 6.3, of 500 Mb 230 -> 26).
constexpr int kBucketWarps = 8, kBucketStage = 512;

__global__ void __launch_bounds__(kBucketWarps * 32) bucket_sort_kernel(const uint32_t *off, uint32_t *entries)
{
    __shared__ uint32_t stage[kBucketWarps][kBucketStage];
    __shared__ uint32_t first[kBucketWarps][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (uint32_t h0 = (blockIdx.x * kBucketWarps + w) * 32; h0 < kNKeys; h0 += gridDim.x * kBucketWarps * 32) {
        const uint32_t mine = off[h0 + lane], end = off[h0 + 32];
        const uint32_t a = __shfl_sync(0xffffffffu, mine, 0), cnt = end - a;
        __syncwarp();
        first[w][lane] = mine - a;
        if (lane == 0) first[w][32] = cnt;
        if (cnt <= kBucketStage) {
            for (uint32_t i = lane; i < cnt; i += 32) stage[w][i] = entries[a + i];
            __syncwarp();
            for (uint32_t i = lane; i < cnt; i += 32) {
                int b = 0;                                 // the bucket: the last one that starts at or before i
#pragma unroll
                for (int step = 16; step > 0; step >>= 1)
                    if (first[w][b + step] <= i) b += step;
                const uint32_t s = first[w][b], e = first[w][b + 1], v = stage[w][i];
                uint32_t at = s;
                for (uint32_t j = s; j < e; ++j) {
                    const uint32_t u = stage[w][j];
                    at += u < v || (u == v && j < i) ? 1u : 0u;
                }
                entries[a + at] = v;
            }
        } else {
            __syncwarp();
            for (int b = 0; b < 32; ++b) {
                uint32_t *e = entries + a + first[w][b];
                const uint32_t n = first[w][b + 1] - first[w][b];
                network_steps(n, [&](uint32_t j) {
                    for (uint64_t i = lane; i < n; i += 32) {
                        const uint32_t l = static_cast<uint32_t>(i) ^ j;
                        if (l > i && l < n && e[i] > e[l]) {
                            const uint32_t t = e[i];
                            e[i] = e[l];
                            e[l] = t;
                        }
                    }
                    __syncwarp();
                });
            }
        }
    }
}

// ------------------------------------------------------------- chaining
// floor(S beta log2(v)) for v = |g| + 1: an integer log2 for a power of two
// (the device log2 need not be exact there), the double log2 otherwise
// (each such value lies at least 6.8e-6 from an integer for |g| < G)
__device__ __forceinline__ int64_t log_term(uint64_t v)
{
    return (v & (v - 1)) == 0
               ? static_cast<int64_t>(63 - __clzll(static_cast<long long>(v))) * (3 * kScale / 4)
               : static_cast<int64_t>(floor(0.75 * static_cast<double>(kScale) * log2(static_cast<double>(v))));
}

// the log term of every |g| < G, computed once per chaining call
__global__ void log_table_kernel(int32_t *tab)
{
    for (int64_t a = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; a < kG;
         a += static_cast<int64_t>(gridDim.x) * blockDim.x)
        tab[a] = static_cast<int32_t>(log_term(static_cast<uint64_t>(a + 1)));
}

// Eq. 3 in units of 2^-16: floor(S |g| / 3) and floor(S beta log2(|g| + 1))
// (their sum for g > 0, the smaller for g < 0); -1 if |g| >= G.  lt: the
// log terms of log_table_kernel.
__device__ __forceinline__ int64_t penalty_eq3(int64_t g, const int32_t *lt)
{
    if (g == 0) return 0;
    const int64_t a = g < 0 ? -g : g;
    if (a >= kG) return -1;
    const int64_t lin = (a * kScale) / 3;
    const int64_t lg = __ldg(lt + a);
    if (g > 0) return lin + lg;
    return lin < lg ? lin : lg;
}

// anchors of protein p: (strand << 63) | (x << 20) | y, x = bin, y = residue
__device__ __forceinline__ uint32_t kmer_hash(const char *P, int t)
{
    uint32_t key = 0;
#pragma unroll
    for (int u = 0; u < kK; ++u) key = key * 16 + c_aa_phi.v[static_cast<unsigned char>(P[t + u])];
    return psi24(key);
}

struct ChainArgs {
    const char *prot;
    const uint64_t *prot_off;
    const uint32_t *prot_len;
    uint32_t n_prot;
    const uint32_t *off;          // index CSR
    const uint32_t *entries;
    uint64_t *anc_off;            // per protein: first anchor (n_prot + 1)
    uint64_t *anc;                // anchors
    int64_t *f;                   // chaining score per anchor
    int32_t *pred;                // predecessor per anchor (-1: none)
    uint8_t *mark;                // kNoStart, kTaken
    int64_t *tmax;                // per 32 anchors of a protein: the largest f of one that may start a chain
    int top;
    mp_chain *chains;             // n_prot * top
    uint32_t *n_chains;
    const int32_t *log_tab;       // log terms of Eq. 3 for |g| < G
    const uint32_t *order;        // proteins, those with most anchors first
};

__global__ void anchor_count_kernel(ChainArgs a, uint64_t *count)
{
    const int lane = threadIdx.x & 31;
    for (uint32_t p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; p < a.n_prot; p += (gridDim.x * blockDim.x) >> 5) {
        const char *P = a.prot + a.prot_off[p];
        const int m = static_cast<int>(a.prot_len[p]);
        uint64_t c = 0;
        for (int t = lane; t + kK <= m; t += 32) {
            const uint32_t h = kmer_hash(P, t);
            c += a.off[h + 1] - a.off[h];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
        if (lane == 0) count[p] = c;
    }
}

__global__ void anchor_fill_kernel(ChainArgs a)
{
    const int lane = threadIdx.x & 31;
    for (uint32_t p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; p < a.n_prot; p += (gridDim.x * blockDim.x) >> 5) {
        const char *P = a.prot + a.prot_off[p];
        const int m = static_cast<int>(a.prot_len[p]);
        uint64_t at = a.anc_off[p];
        for (int t0 = 0; t0 + kK <= m; t0 += 32) {
            const int t = t0 + lane;
            uint32_t lo = 0, hi = 0;
            if (t + kK <= m) {
                const uint32_t h = kmer_hash(P, t);
                lo = a.off[h];
                hi = a.off[h + 1];
            }
            // each lane's hits go after the earlier lanes' hits
            uint64_t cnt = hi - lo, incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint64_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            // one hit per lane at a time (a lane per k-mer wrote its hits in runs of
            // its own): the hit's k-mer is the first lane whose count passes it
            const uint32_t total = static_cast<uint32_t>(__shfl_sync(0xffffffffu, incl, 31));
            for (uint32_t o0 = 0; o0 < total; o0 += 32) {
                const uint32_t o = o0 + lane;
                int k = 0;
#pragma unroll
                for (int step = 16; step > 0; step >>= 1) {
                    const uint32_t below = static_cast<uint32_t>(__shfl_sync(0xffffffffu, incl, k + step - 1));
                    if (o >= below) k += step;
                }
                const uint32_t first = __shfl_sync(0xffffffffu, lo, k);
                const uint32_t before = static_cast<uint32_t>(__shfl_sync(0xffffffffu, incl - cnt, k));
                if (o < total) {
                    const uint32_t v = a.entries[first + (o - before)];
                    a.anc[at + o] = (static_cast<uint64_t>(v >> 31) << 63) |
                                    (static_cast<uint64_t>(v & 0x7fffffffu) << 20) | static_cast<uint64_t>(t0 + k);
                }
            }
            at += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
}

// One block per protein, the ones with most anchors first: its anchors sorted
// by (strand, x), eight bits at a time from the lowest, stably; they come in
// ascending y, so that the order is (strand, x, y).  Each warp takes a
// contiguous part: it counts its digits, the counts are summed over digits and
// warps, and it writes its anchors 32 at a time, each behind the equal digits
// before it (a warp match gives its place among the 32).  The passes go to and
// fro between a.anc and tmp; after an odd number of passes the result is in
// tmp.  (A bitonic network over 64-bit keys in shared memory, 91 to 105 steps
// for a protein, took 5.2 ms for 4,000 proteins; this 0.75.)
constexpr int kSortThreads = 256;
constexpr int kDigitBits = 8, kDigits = 1 << kDigitBits;

__host__ __device__ constexpr int sort_passes(int xbits) { return (xbits + 1 + kDigitBits - 1) / kDigitBits; }

__global__ void __launch_bounds__(kSortThreads) anchor_sort_kernel(ChainArgs a, uint64_t *tmp, int xbits)
{
    constexpr int kWarps = kSortThreads / 32;
    static_assert(kSortThreads == kDigits, "a thread per digit sums the warps' counts");
    __shared__ uint32_t hist[kWarps][kDigits];
    __shared__ uint32_t warp_sum[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t xmask = (1ull << xbits) - 1;
    for (uint32_t k = blockIdx.x; k < a.n_prot; k += gridDim.x) {
        const uint32_t p = a.order[k];
        const uint64_t b0 = a.anc_off[p], n = a.anc_off[p + 1] - b0;
        uint64_t *src = a.anc + b0, *dst = tmp + b0;
        const uint64_t per = (n + kSortThreads - 1) / kSortThreads * 32;
        const uint64_t i0 = per * warp < n ? per * warp : n, i1 = i0 + per < n ? i0 + per : n;
        for (int shift = 0; shift <= xbits; shift += kDigitBits) {
            auto digit = [&](uint64_t v) {
                const uint64_t key = ((v >> 20) & xmask) | (v >> 63) << xbits;
                return static_cast<uint32_t>(key >> shift) & (kDigits - 1);
            };
            for (int d = lane; d < kDigits; d += 32) hist[warp][d] = 0;
            __syncwarp();
            for (uint64_t i = i0 + lane; i < i1; i += 32) atomicAdd(&hist[warp][digit(src[i])], 1u);
            __syncthreads();
            // thread d: digit d's count, the sum of the digits below, then each warp's start
            uint32_t sum = 0;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) sum += hist[w][threadIdx.x];
            uint32_t incl = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (lane == 31) warp_sum[warp] = incl;
            __syncthreads();
            uint32_t run = incl - sum;
            for (int w = 0; w < warp; ++w) run += warp_sum[w];
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const uint32_t c = hist[w][threadIdx.x];
                hist[w][threadIdx.x] = run;
                run += c;
            }
            __syncthreads();
            for (uint64_t i = i0; i < i1; i += 32) {
                const bool have = i + lane < i1;
                const uint64_t v = have ? src[i + lane] : 0;
                const uint32_t d = have ? digit(v) : kDigits;        // (no digit: a group of its own)
                const unsigned same = __match_any_sync(0xffffffffu, d);
                const int before = __popc(same & ((1u << lane) - 1));
                if (have) dst[hist[warp][d] + before] = v;
                __syncwarp();
                if (have && before == 0) hist[warp][d] += __popc(same);
                __syncwarp();
            }
            __syncthreads();
            uint64_t *t = src;
            src = dst;
            dst = t;
        }
    }
}

// an anchor that starts no chain (no predecessor, or one of no smaller f); one
// that a chain has taken
constexpr uint8_t kNoStart = 1, kTaken = 2;

__device__ __forceinline__ int anc_strand(uint64_t v) { return static_cast<int>(v >> 63); }
__device__ __forceinline__ int64_t anc_x(uint64_t v) { return static_cast<int64_t>((v >> 20) & 0x7fffffffffull); }
__device__ __forceinline__ int64_t anc_y(uint64_t v) { return static_cast<int64_t>(v & 0xfffffu); }

// Eq. 2 over sorted anchors, 32 anchors at a time (a tile), one per lane.  A
// lane keeps its anchor's best predecessor; every predecessor is read once per
// tile and tried by all lanes (in ascending order, a later one only if
// strictly better, so that the first of equal best ones stays).  Most tries
// end at a bound that takes the penalty's log2(|g| + 1) down to its integer
// part and so needs no table; only a link that may win looks its log term up.
// Inside a tile the anchors depend on one another: the same bound with the
// scores found so far shows which anchors of the tile any other can follow, a
// few of the 32; only these are tried one by one.
//
// What bounds it: the tries' integer instructions (about 20 a try, some 50
// tries per anchor on the 50 Mb workload) and, for the longest protein, the
// tiles' chain of dependent loads.  With the predecessors spread over the
// lanes and a 64-bit warp maximum per anchor (five rounds of four shuffles, in
// series) 4,000 proteins took 80 ms.
//
// T: int32_t for proteins up to kMax32 residues (f is at most (m + 6) * 2^16;
// links whose linear term alone passes every f are left out by the clamp of
// |g|), else int64_t.
constexpr int64_t kMax32 = 32000;
constexpr int32_t kClamp32 = 98000;          // kClamp32 * 21845 is just below 2^31, above every 32-bit f
constexpr int32_t kBits = 3 * static_cast<int32_t>(kScale) / 4;      // beta in units of 2^-16: one bit of |g| + 1

struct TileAnchor {
    uint32_t x;
    int32_t y;
};

// First round: x a bin, the strand in bit 30; the gap of Eq. 1.  reach: from
// this many bins on |g| >= G (dx is clamped to it; the other strand's anchors
// are further).
struct BinGeo {
    static constexpr int K = kK;
    uint32_t reach;
    __device__ __forceinline__ explicit BinGeo(int64_t m) : reach(static_cast<uint32_t>((kG + 3 * m) / kBin + 2)) {}
    static __device__ __forceinline__ TileAnchor anchor(uint64_t v)
    {
        return TileAnchor{static_cast<uint32_t>((v >> 20) & 0x3fffffffu) | static_cast<uint32_t>(v >> 63) << 30,
                          static_cast<int32_t>(v & 0xfffffu)};
    }
    __device__ __forceinline__ int32_t gap(uint32_t dx, int32_t dy) const
    {
        const int32_t d = static_cast<int32_t>(dx < reach ? dx : reach) * kBin, py = 3 * dy;
        return py - min(max(py, d - kBin), d + kBin);
    }
};

// Second round: x a base of the region; g' = 3 dy - dx.
struct BaseGeo {
    static constexpr int K = 5;
    uint32_t reach;
    __device__ __forceinline__ explicit BaseGeo(int64_t m) : reach(static_cast<uint32_t>(kG + 3 * m)) {}
    static __device__ __forceinline__ TileAnchor anchor(uint64_t v)
    {
        return TileAnchor{static_cast<uint32_t>(v >> 20), static_cast<int32_t>(v & 0xfffffu)};
    }
    __device__ __forceinline__ int32_t gap(uint32_t dx, int32_t dy) const
    {
        return 3 * dy - static_cast<int32_t>(dx < reach ? dx : reach);
    }
};

// the largest value of the lanes
__device__ __forceinline__ int32_t warp_max(int32_t v) { return __reduce_max_sync(0xffffffffu, v); }
__device__ __forceinline__ int64_t warp_max(int64_t v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const int64_t ov = __shfl_xor_sync(0xffffffffu, v, o);
        v = ov > v ? ov : v;
    }
    return v;
}

// the largest value of the lanes, the first index among equals
__device__ __forceinline__ void warp_first_max(int64_t &v, int64_t &i)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const int64_t ov = __shfl_xor_sync(0xffffffffu, v, o);
        const int64_t oi = __shfl_xor_sync(0xffffffffu, i, o);
        if (ov > v || (ov == v && oi < i)) {
            v = ov;
            i = oi;
        }
    }
}

// One lane's anchor and its best predecessor so far.
template <typename T, typename Geo>
struct Seeker {
    Geo geo;
    TileAnchor t;
    T best;
    int32_t arg = -1;
    bool gains = false;                      // best is above the predecessor's f
    static constexpr T kFirst = static_cast<T>(Geo::K) * static_cast<T>(kScale);

    __device__ __forceinline__ Seeker(const Geo &g, const TileAnchor &a) : geo(g), t(a), best(kFirst) {}

    // Whether an anchor at (x, y) with score f may be a better predecessor.
    // A link is worth at most K less the penalty, and the penalty at least
    // one kBits per bit of |g| + 1 above the first (less only for |g| <= 6, by
    // the linear term, which always passes here).
    __device__ __forceinline__ bool may(uint32_t x, int32_t y, T f, int32_t &g, int32_t &dy) const
    {
        dy = t.y - y;
        g = geo.gap(t.x - x, dy);
        const T slack = f + kFirst - best, top = static_cast<T>(INT_MAX);
        const uint32_t s = static_cast<uint32_t>(max(min(slack, top), static_cast<T>(0)));
        const uint32_t bits = max(__umulhi(s, 87382u) + 1u, 3u);             // floor(s / kBits) + 1, or one more
        return dy > 0 && __funnelshift_rc(static_cast<uint32_t>(abs(g)) + 1u, 0u, bits) == 0;
    }
    // The same with the linear term: the link's worth is at most `up`
    __device__ __forceinline__ bool may_win(T f, int32_t g, int32_t dy) const
    {
        const int32_t a = abs(g);
        const int32_t l2 = (31 - __clz(a + 1)) * kBits;
        const T lin = static_cast<T>(sizeof(T) == 4 ? min(a, kClamp32) : a) * 21845;        // 65536 = 3 * 21845 + 1
        const T low = g < 0 ? (lin < static_cast<T>(l2) ? lin : static_cast<T>(l2)) : lin + static_cast<T>(l2);
        // (32 bits: f is positive and the rest above -2^31)
        return a < static_cast<int32_t>(kG) &&
               f + (static_cast<T>(min(dy, Geo::K)) * static_cast<T>(kScale) - low) > best;
    }
    __device__ __forceinline__ void try_link(uint32_t x, int32_t y, T f, int32_t i, const int32_t *lt)
    {
        int32_t g, dy;
        if (may(x, y, f, g, dy) && may_win(f, g, dy)) {
            const int64_t c =
                static_cast<int64_t>(f) + static_cast<int64_t>(min(dy, Geo::K)) * kScale - penalty_eq3(g, lt);
            if (c > static_cast<int64_t>(best)) {
                best = static_cast<T>(c);
                arg = i;
                gains = c > static_cast<int64_t>(f);
            }
        }
    }
};

// Shared memory of chain_dp: the predecessors at hand, per warp, and what the
// other warps found for the tile's anchors.
template <int NW>
struct ChainSmem {
    int4 stage[NW][32];
    int64_t best[NW][32];
    int32_t arg[NW][32];                     // predecessor, its bit 31 flipped if best is above its f
    unsigned from[NW][32];
};

// The anchors [0, n) of A by NW warps of a block (0 .. NW-1, which meet at
// barrier `bar`; with one, nothing but that warp takes part), which share out
// a tile's tries.  done(j0, j, have, seeker): called by warp 0 for every tile.
template <typename T, typename Geo, int NW, typename Done>
__device__ void chain_dp(const uint64_t *A, int64_t n, const Geo &geo, const int32_t *lt, int64_t *F, int32_t *Pr,
                         ChainSmem<NW> &sm, int bar, int warp, int lane, Done done)
{
    auto meet = [&] {
        if (NW == 1) __syncwarp();
        else asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(NW * 32) : "memory");
    };
    int4 *stage = sm.stage[warp];
    auto put = [&](const TileAnchor &u, int64_t f) {
        stage[lane] = make_int4(static_cast<int>(u.x), u.y, static_cast<int>(f), static_cast<int>(f >> 32));
    };
    auto f_of = [](const int4 &u) {
        return sizeof(T) == 4 ? static_cast<T>(u.z)
                              : static_cast<T>(static_cast<int64_t>(u.w) << 32 | static_cast<uint32_t>(u.z));
    };
    int64_t lo = 0;
    uint64_t next = A[lane < n ? lane : n - 1];
    for (int64_t j0 = 0; j0 < n; j0 += 32) {
        const int64_t j = j0 + lane;
        const bool have = j < n;
        Seeker<T, Geo> me(geo, Geo::anchor(next));
        next = A[j + 32 < n ? j + 32 : n - 1];         // the next tile's, on its way
        // the window of the tile's first anchor holds every lane's
        const uint32_t x0 = __shfl_sync(0xffffffffu, me.t.x, 0);
        for (;;) {
            const int64_t i = lo + lane;
            const bool far = i < j0 && x0 - Geo::anchor(A[i]).x > geo.reach;
            const unsigned near = __ballot_sync(0xffffffffu, !far);
            lo += near ? __ffs(near) - 1 : 32;
            if (near) break;
        }
        for (int64_t i0 = lo + 32 * warp; i0 < j0; i0 += 32 * NW) {
            const int cnt = static_cast<int>(j0 - i0 < 32 ? j0 - i0 : 32);
            __syncwarp();
            if (lane < cnt) put(Geo::anchor(A[i0 + lane]), F[i0 + lane]);
            __syncwarp();
#pragma unroll 4
            for (int k = 0; k < cnt; ++k) {
                const int4 u = stage[k];
                me.try_link(static_cast<uint32_t>(u.x), u.y, f_of(u), static_cast<int32_t>(i0) + k, lt);
            }
        }
        if (NW > 1) {
            // the largest of the warps, the first predecessor among equals
            sm.best[warp][lane] = static_cast<int64_t>(me.best);
            sm.arg[warp][lane] = me.gains ? me.arg ^ INT_MIN : me.arg;
            meet();
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                const T b = static_cast<T>(sm.best[w][lane]);
                const int32_t r = sm.arg[w][lane];
                const bool gains = r < -1;
                const int32_t i = gains ? r ^ INT_MIN : r;
                if (b > me.best || (b == me.best && i >= 0 && me.arg >= 0 && i < me.arg)) {
                    me.best = b;
                    me.arg = i;
                    me.gains = gains;
                }
            }
        }
        // inside the tile: which anchors can any other follow?
        __syncwarp();
        put(me.t, static_cast<int64_t>(me.best));
        __syncwarp();
        const int cnt = static_cast<int>(n - j0 < 32 ? n - j0 : 32);
        unsigned from = 0;                                 // anchors this lane's may follow
#pragma unroll 4
        for (int k = warp; k < cnt - 1; k += NW) {
            const int4 u = stage[k];
            int32_t g, dy;
            if (me.may(static_cast<uint32_t>(u.x), u.y, f_of(u), g, dy) && k < lane && me.may_win(f_of(u), g, dy))
                from |= 1u << k;
        }
        if (NW > 1) {
            sm.from[warp][lane] = from;
            meet();
        }
        if (warp == 0) {
#pragma unroll
            for (int w = 1; w < NW; ++w) from |= sm.from[w][lane];
            // the anchors that any other may follow, in ascending order; one that
            // gains joins them (a test that failed with a lower score and an
            // unchanged one of the other anchor keeps failing)
            unsigned todo = __reduce_or_sync(0xffffffffu, have ? from : 0u);
            while (todo) {
                const int k = __ffs(todo) - 1;
                todo &= todo - 1;
                const uint32_t xi = __shfl_sync(0xffffffffu, me.t.x, k);
                const int32_t yi = __shfl_sync(0xffffffffu, me.t.y, k);
                const T fi = __shfl_sync(0xffffffffu, me.best, k);
                const T was = me.best;
                if (lane > k) me.try_link(xi, yi, fi, static_cast<int32_t>(j0) + k, lt);
                todo |= __ballot_sync(0xffffffffu, have && me.best != was);
            }
            if (have) {
                F[j] = static_cast<int64_t>(me.best);
                Pr[j] = me.arg;
            }
            done(j0, j, have, me);
        }
        meet();                                            // F is read by the next tiles
    }
}

// where a protein's tiles start in ChainArgs::tmax
__device__ __forceinline__ uint64_t tile_base(uint64_t b0, uint32_t p) { return b0 / 32 + 2ull * p; }

// One block per protein, the ones with most anchors first: Eq. 2 over its
// sorted anchors, kStrandWarps warps per strand (chains stay on one; the
// longest protein's tiles are a chain of their own), then its chains.
//
// Chains are taken in order of decreasing f of the last anchor (ties: the
// earlier anchor), each cut at an anchor already taken, and single anchors
// are dropped, which takes them too.  An anchor whose predecessor has no
// smaller f comes after it in that order and so is always alone; the walk of a
// chain from b stops at an anchor of an earlier chain or one that precedes b
// in the order.  So only anchors above their predecessor's f are looked at,
// and no single one is ever taken by itself: near a long chain thousands
// follow it at a loss, and with a look at every anchor before each of them one
// protein of 4,000 took 20 ms.  The best is found from the largest f of each
// tile; a tile whose largest is out of date is seen when it is looked at.
constexpr int kStrandWarps = 4;
__global__ void __launch_bounds__(kStrandWarps * 64) chain_kernel(ChainArgs a)
{
    __shared__ ChainSmem<kStrandWarps> sm[2];
    const int lane = threadIdx.x & 31, strand = threadIdx.x / (kStrandWarps * 32);
    const int warp = (threadIdx.x >> 5) % kStrandWarps;
    for (uint32_t k = blockIdx.x; k < a.n_prot; k += gridDim.x) {
        const uint32_t p = a.order[k];
        const uint64_t b0 = a.anc_off[p];
        const int64_t n = static_cast<int64_t>(a.anc_off[p + 1] - b0);
        const uint64_t *A = a.anc + b0;
        int64_t *F = a.f + b0;
        int32_t *Pr = a.pred + b0;
        uint8_t *U = a.mark + b0;
        const int64_t m = a.prot_len[p];
        int64_t *tmax = a.tmax + tile_base(b0, p);
        // the first anchor of strand 1: 31 probes at a time
        int64_t s0 = 0, s1 = n;                            // strand 0 below s0, strand 1 from s1 on
        while (s0 < s1) {
            const int64_t step = (s1 - s0 + 31) / 32, at = s0 + step * lane;
            const unsigned zero = __ballot_sync(0xffffffffu, at < s1 && anc_strand(A[at]) == 0);
            const int c = __popc(zero);                    // probes on strand 0, the first ones
            if (c < 32 && s0 + step * c < s1) s1 = s0 + step * c;
            if (c) s0 = s0 + step * (c - 1) + 1;
        }
        const int64_t split = s0, nt0 = (split + 31) / 32, nt = nt0 + (n - split + 31) / 32;
        {
            const int64_t from = strand ? split : 0, cnt = strand ? n - split : split;
            int64_t *tm = tmax + (strand ? nt0 : 0);
            uint8_t *Us = U + from;
            // (predecessors are numbered from the strand's first anchor)
            auto run = [&](auto zero) {
                using T = decltype(zero);
                chain_dp<T, BinGeo, kStrandWarps>(
                    A + from, cnt, BinGeo(m), a.log_tab, F + from, Pr + from, sm[strand], 1 + strand, warp, lane,
                    [&](int64_t j0, int64_t j, bool have, const Seeker<T, BinGeo> &me) {
                        if (have) Us[j] = me.gains ? 0 : kNoStart;
                        const T top = warp_max(have && me.gains ? me.best : static_cast<T>(0));
                        if (lane == 0) tm[j0 >> 5] = static_cast<int64_t>(top);
                    });
            };
            if (cnt > 0) {
                if (m <= kMax32) run(static_cast<int32_t>(0));
                else run(static_cast<int64_t>(0));
            }
        }
        __syncthreads();
        if (strand || warp) continue;
        int nc = 0;
        while (nc < a.top) {
            // each lane the first best of its own tiles, then the warp's
            int64_t bf = INT64_MIN, bt = INT64_MAX;
#pragma unroll 4
            for (int64_t t = lane; t < nt; t += 32) {
                const int64_t f = tmax[t];
                if (f > bf) {
                    bf = f;
                    bt = t;
                }
            }
            warp_first_max(bf, bt);
            if (bf <= static_cast<int64_t>(kK) * kScale) break;
            const int64_t base = bt < nt0 ? 0 : split;     // of the strand
            const int64_t at = bt < nt0 ? bt * 32 + lane : split + (bt - nt0) * 32 + lane;
            int64_t f = 0;
            if (at < (bt < nt0 ? split : n) && U[at] == 0 && !(U[base + Pr[at]] & kTaken)) f = F[at];
            const int64_t best = warp_max(f);
            if (best < bf) {
                // some of the tile's were taken, or their predecessors were
                if (lane == 0) tmax[bt] = best;
                __syncwarp();
                continue;
            }
            const int64_t bi = at - lane + __ffs(__ballot_sync(0xffffffffu, f == bf)) - 1;
            int64_t cnt = 0, cur = bi, first = bi;
            do {
                if (lane == 0) U[cur] |= kTaken;
                first = cur;
                ++cnt;
                cur = Pr[cur] < 0 ? -1 : base + Pr[cur];
            } while (cur >= 0 && !(U[cur] & kTaken) && F[cur] < bf);
            __syncwarp();
            if (lane == 0) {
                mp_chain &c = a.chains[static_cast<uint64_t>(p) * a.top + nc];
                c.strand = anc_strand(A[bi]);
                c.n_anchors = static_cast<int32_t>(cnt);
                c.score = bf - (cur >= 0 ? F[cur] : 0);
                c.x_first = anc_x(A[first]);
                c.x_last = anc_x(A[bi]);
                c.y_first = anc_y(A[first]);
                c.y_last = anc_y(A[bi]);
            }
            ++nc;
        }
        if (lane == 0) a.n_chains[p] = static_cast<uint32_t>(nc);
    }
}

// ---------------------------------------------------------- second round

constexpr int kK2 = 5;                      // k-mer length of the second round
constexpr int kRefineMaxProt = 8192;        // protein k-mer table in shared memory (64 KB)
constexpr int kRefineThreads = 256;
constexpr int64_t kRefineBig = 512;          // pairs with more anchors are chained by a whole block

struct RefineArgs {
    const char *seq;                        // every pair's protein and region (ASCII)
    const uint64_t *prot_off, *nt_off;
    const uint32_t *prot_len, *nt_len;
    const int8_t *strand;
    uint32_t n;                             // pairs
    const uint64_t *anc_off;                // pair p's anchors at anc[anc_off[p] ..)
    uint64_t *anc;                          // x << 20 | y
    int64_t *f;
    int32_t *pred;
    mp_chain2 *out;
    const int32_t *log_tab;
};

// FILL = false: count the pair's anchors into total[p]; true: write them from
// anc_off[p] on, in (x, y) order.
//
// One block per pair.  The protein's k-mers are sorted as key << 13 | y
// (bitonic, shared memory), so the k-mers equal to a base's are found by one
// binary search, in ascending y.  The region comes in tiles of kTile bases:
// their letters are read once, then each base's codon is translated once, and
// a base's k-mer is put together from five of them.  Nearly all bases end at a
// filter of 2^15 bits that holds a hash of every protein k-mer (a binary
// search per base, on codons translated for each of the five, took 2.7 ms per
// pass for 6,000 regions; this 0.6 to 0.7).
constexpr int kTile = 4096;
constexpr int kFilterBits = 15;

// the k-mer's bit in the filter
__device__ __forceinline__ uint32_t filter_hash(uint32_t key) { return (key * 2654435761u) >> (32 - kFilterBits); }

template <bool FILL>
__global__ void __launch_bounds__(kRefineThreads) refine_anchor_kernel(RefineArgs a, uint64_t *total)
{
    extern __shared__ uint64_t pk[];                // the protein's k-mers (a power of two of them)
    __shared__ uint32_t filter[(1 << kFilterBits) / 32];
    __shared__ uint8_t code[kTile + 3 * kK2];       // bases (4: not one of A, C, G, T), then codons
    __shared__ uint8_t s_phi[64];
    __shared__ uint32_t warp_cnt[kRefineThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = threadIdx.x; k < 64; k += blockDim.x) s_phi[k] = c_codon_phi.v[k];
    for (uint32_t p = blockIdx.x; p < a.n; p += gridDim.x) {
        const char *P = a.seq + a.prot_off[p];
        const char *T = a.seq + a.nt_off[p];
        const int m = static_cast<int>(a.prot_len[p]);
        const int64_t L = a.nt_len[p];
        const int strand = a.strand[p];
        const int ny = m - kK2 + 1;                 // protein k-mers
        const int64_t nx = ny > 0 ? L - 3 * kK2 + 1 : 0;      // region k-mers (one per base)
        int n2 = 1;
        while (n2 < ny) n2 <<= 1;
        for (int k = threadIdx.x; k < (1 << kFilterBits) / 32; k += blockDim.x) filter[k] = 0;
        __syncthreads();
        for (int y = threadIdx.x; y < n2; y += blockDim.x) {
            uint64_t key = ~0ull;
            if (y < ny) {
                key = 0;
#pragma unroll
                for (int u = 0; u < kK2; ++u) key = key * 16 + c_aa_phi.v[static_cast<unsigned char>(P[y + u])];
                const uint32_t h = filter_hash(static_cast<uint32_t>(key));
                atomicOr(&filter[h >> 5], 1u << (h & 31));
                key = key << 13 | static_cast<uint64_t>(y);
            }
            pk[y] = key;
        }
        __syncthreads();
        for (int k = 2; k <= n2; k <<= 1)
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int i = threadIdx.x; i < n2; i += blockDim.x) {
                    const int l = i ^ j;
                    if (l > i) {
                        const uint64_t u = pk[i], v = pk[l];
                        if ((u > v) == ((i & k) == 0)) {
                            pk[i] = v;
                            pk[l] = u;
                        }
                    }
                }
                __syncthreads();
            }
        uint64_t at = FILL ? a.anc_off[p] : 0;      // the tile's first slot
        uint64_t mine = 0;                          // this thread's anchors so far
        for (int64_t x0 = 0; x0 < nx; x0 += kTile) {
            const int nt = static_cast<int>(nx - x0 < kTile ? nx - x0 : kTile);      // the tile's k-mers
            // the bases they touch, of the aligned strand
            for (int i = threadIdx.x; i < nt + 3 * kK2 - 1; i += blockDim.x) {
                const int64_t x = x0 + i;
                const int c = base_code(static_cast<unsigned char>(strand > 0 ? T[x] : T[L - 1 - x]));
                code[i] = static_cast<uint8_t>(c < 0 ? 4 : strand > 0 ? c : 3 - c);
            }
            __syncthreads();
            // codon phi in place: each thread's part, after it has read the two
            // bases behind it that belong to the next thread
            constexpr int kPart = (kTile + 3 * kK2 + kRefineThreads - 1) / kRefineThreads;
            const int i0 = threadIdx.x * kPart, ic = nt + 3 * (kK2 - 1);              // codons
            const int n0 = i0 + kPart < nt + 3 * kK2 - 1 ? code[i0 + kPart] : 4;
            const int n1 = i0 + kPart + 1 < nt + 3 * kK2 - 1 ? code[i0 + kPart + 1] : 4;
            __syncthreads();
            if (i0 < ic) {
                int b0 = code[i0], b1 = kPart > 1 ? code[i0 + 1] : n0;
                for (int i = i0; i < i0 + kPart && i < ic; ++i) {
                    const int b2 = i + 2 < i0 + kPart ? code[i + 2] : i + 2 == i0 + kPart ? n0 : n1;
                    code[i] = (b0 | b1 | b2) & 4 ? kXCode : s_phi[b0 * 16 + b1 * 4 + b2];
                    b0 = b1;
                    b1 = b2;
                }
            }
            __syncthreads();
            // thread t takes the k-mers [t * per, t * per + per) of the tile
            // (an odd number of bytes apart, for the banks)
            const int per = static_cast<int>((nt + blockDim.x - 1) / blockDim.x) | 1;
            const int xa = threadIdx.x * per < nt ? threadIdx.x * per : nt, xb = xa + per < nt ? xa + per : nt;
            auto each = [&](auto &&found) {
                for (int x = xa; x < xb; ++x) {
                    uint32_t key = 0;
#pragma unroll
                    for (int u = 0; u < kK2; ++u) key = key * 16 + code[x + 3 * u];
                    const uint32_t h = filter_hash(key);
                    if (!(filter[h >> 5] >> (h & 31) & 1)) continue;
                    // first entry >= key << 13
                    const uint64_t want = static_cast<uint64_t>(key) << 13;
                    int lo = 0, hi = ny;
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (pk[mid] < want) lo = mid + 1;
                        else hi = mid;
                    }
                    for (int e = lo; e < ny && (pk[e] >> 13) == key; ++e) found(x, pk[e] & 0x1fffu);
                }
            };
            uint32_t c = 0;
            each([&](int, uint64_t) { ++c; });
            mine += c;
            if (FILL) {
                // the anchors of the threads before this one
                uint32_t incl = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                if (lane == 31) warp_cnt[warp] = incl;
                __syncthreads();
                uint64_t to = at + incl - c;
                for (int w = 0; w < kRefineThreads / 32; ++w) {
                    if (w < warp) to += warp_cnt[w];
                    at += warp_cnt[w];
                }
                if (c) each([&](int x, uint64_t y) { a.anc[to++] = static_cast<uint64_t>(x0 + x) << 20 | y; });
            }
            __syncthreads();                        // the tile's codons and counts are read no more
        }
        if (!FILL) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
            __shared__ uint64_t part[kRefineThreads / 32];
            if (lane == 0) part[warp] = mine;
            __syncthreads();
            if (threadIdx.x == 0) {
                uint64_t sum = 0;
                for (int w = 0; w < kRefineThreads / 32; ++w) sum += part[w];
                total[p] = sum;
            }
        }
        __syncthreads();
    }
}

// The pair's best chain from f and the predecessors (one thread).
__device__ __forceinline__ mp_chain2 best_chain(const uint64_t *A, const int64_t *F, const int32_t *Pr, int64_t bi)
{
    mp_chain2 c{};
    if (bi >= 0 && Pr[bi] >= 0) {
        int64_t cnt = 0, cur = bi, first = bi;
        while (cur >= 0) {
            first = cur;
            ++cnt;
            cur = Pr[cur];
        }
        c.n_anchors = static_cast<int32_t>(cnt);
        c.score = F[bi];
        c.x_first = static_cast<int64_t>(A[first] >> 20);
        c.x_last = static_cast<int64_t>(A[bi] >> 20);
        c.y_first = static_cast<int64_t>(A[first] & 0xfffffu);
        c.y_last = static_cast<int64_t>(A[bi] & 0xfffffu);
    }
    return c;
}

// f of every anchor of pair p with g' = 3 dy - dx by NW warps, then the best
// chain (the first anchor with the largest f and its predecessors).
template <int NW>
__device__ __forceinline__ void refine_pair(const RefineArgs &a, uint32_t p, ChainSmem<NW> &sm, int warp, int lane)
{
    const uint64_t b0 = a.anc_off[p];
    const int64_t n = static_cast<int64_t>(a.anc_off[p + 1] - b0);
    const uint64_t *A = a.anc + b0;
    int64_t *F = a.f + b0;
    int32_t *Pr = a.pred + b0;
    int64_t bf = INT64_MIN, bi = INT64_MAX;             // this lane's first best anchor
    // (proteins have at most kRefineMaxProt residues: 32-bit scores)
    if (n > 0)
        chain_dp<int32_t, BaseGeo, NW>(A, n, BaseGeo(a.prot_len[p]), a.log_tab, F, Pr, sm, 0, warp, lane,
                                       [&](int64_t, int64_t j, bool have, const Seeker<int32_t, BaseGeo> &me) {
                                           if (have && me.best > bf) {
                                               bf = me.best;
                                               bi = j;
                                           }
                                       });
    if (warp == 0) {
        warp_first_max(bf, bi);
        if (lane == 0) a.out[p] = best_chain(A, F, Pr, n > 0 ? bi : -1);
    }
}

// One warp per pair.
constexpr int kRefineWarps = 4;
__global__ void __launch_bounds__(kRefineWarps * 32) refine_chain_kernel(RefineArgs a)
{
    __shared__ ChainSmem<1> sm[kRefineWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (uint32_t p = blockIdx.x * kRefineWarps + warp; p < a.n; p += gridDim.x * kRefineWarps)
        if (static_cast<int64_t>(a.anc_off[p + 1] - a.anc_off[p]) <= kRefineBig)
            refine_pair<1>(a, p, sm[warp], 0, lane);
}

// One block per pair with more than kRefineBig anchors: every earlier anchor
// of a region is within reach, so the tries grow with the square of their
// number, and the warps share each tile's out.
__global__ void __launch_bounds__(kRefineThreads) refine_chain_block_kernel(RefineArgs a)
{
    constexpr int NW = kRefineThreads / 32;
    __shared__ ChainSmem<NW> sm;
    for (uint32_t p = blockIdx.x; p < a.n; p += gridDim.x)
        if (static_cast<int64_t>(a.anc_off[p + 1] - a.anc_off[p]) > kRefineBig) {       // uniform across the block
            refine_pair<NW>(a, p, sm, threadIdx.x >> 5, threadIdx.x & 31);
            __syncthreads();
        }
}

}  // namespace
}  // namespace mpdp

// ===================================================================== host
struct mp_index {
    int device = 0;
    uint64_t n_entries = 0;
    int xbits = 0;                  // bits of the largest bin
    uint32_t *off = nullptr;        // kNKeys + 1
    uint32_t *entries = nullptr;
};

namespace {
using namespace mpdp;

// a device allocation freed when it leaves scope
template <typename T>
struct Tmp {
    T *p = nullptr;
    cudaError_t alloc(uint64_t n) { return cudaMalloc(&p, (n ? n : 1) * sizeof(T)); }
    ~Tmp() { if (p) cudaFree(p); }
    Tmp() = default;
    Tmp(const Tmp &) = delete;
    Tmp &operator=(const Tmp &) = delete;
};

#define SCK(x)                                                                         \
    do {                                                                               \
        cudaError_t e_ = (x);                                                          \
        if (e_ != cudaSuccess) return e_ == cudaErrorMemoryAllocation ? MP_ENOMEM : MP_ECUDA; \
    } while (0)

int grid_for(uint64_t threads, int block)
{
    const uint64_t g = (threads + block - 1) / block;
    return static_cast<int>(g < 65535ull * 16 ? (g ? g : 1) : 65535ull * 16);
}

// whether anchors are numbered in 31 bits throughout (predecessors are 32-bit
// and signed, and a warp numbers the hits of 32 k-mers in 32 bits)
bool few_enough(const std::vector<uint64_t> &anchors)
{
    return std::all_of(anchors.begin(), anchors.end(), [](uint64_t c) { return c <= INT_MAX; });
}

// exclusive prefix sums of n counts: out[0..n] (out[n] the total)
int scan_counts(const uint32_t *in, uint64_t n, uint32_t *out, cudaStream_t st)
{
    const uint32_t nb = static_cast<uint32_t>((n + kScanBlock * 4 - 1) / (kScanBlock * 4));
    Tmp<uint32_t> sums, total;
    SCK(sums.alloc(nb));
    SCK(total.alloc(1));
    scan_blocks<<<nb ? nb : 1, kScanBlock, 0, st>>>(in, n, out, sums.p);
    scan_sums<<<1, 32, 0, st>>>(sums.p, nb, total.p);
    scan_add<<<grid_for(n, 256), 256, 0, st>>>(out, n, sums.p, total.p);
    SCK(cudaGetLastError());
    SCK(cudaStreamSynchronize(st));
    return MP_OK;
}
}  // namespace

extern "C" int mp_index_build(mp_dp_ctx *ctx, const char *genome, uint64_t len, mp_index **out)
{
    if (!ctx || !out || (len && !genome)) return MP_EINVAL;
    *out = nullptr;
    if (len / 3 >= (1ull << 31)) return MP_EINVAL;          // frame-relative positions and bins are 31-bit
    const int dev = ctx_device(ctx);
    if (cudaSetDevice(dev) != cudaSuccess) return MP_ECUDA;
    cudaStream_t st = ctx_stream(ctx);
    Tmp<char> g;
    SCK(g.alloc(len));
    if (len) SCK(cudaMemcpyAsync(g.p, genome, len, cudaMemcpyHostToDevice, st));
    // the six frames: codons, segments
    Frames fr{};
    uint64_t total = 0, nseg = 0;
    for (int f = 0; f < 6; ++f) {
        const uint64_t frame = f % 3;
        fr.len[f] = len > frame ? (len - frame) / 3 : 0;
        fr.seg0[f] = nseg;
        nseg += (fr.len[f] + kSeg - 1) / kSeg;
        total += fr.len[f];
    }
    fr.seg0[6] = nseg;
    Tmp<uint8_t> codes;
    SCK(codes.alloc(total + 6 * 16));
    uint64_t at = 0;
    for (int f = 0; f < 6; ++f) {
        fr.code[f] = codes.p + at;
        at += (fr.len[f] + 15) / 16 * 16;
    }
    Tmp<int64_t> first, last, before, after;
    SCK(first.alloc(nseg));
    SCK(last.alloc(nseg));
    SCK(before.alloc(nseg));
    SCK(after.alloc(nseg));
    Tmp<uint32_t> count, cursor;
    SCK(count.alloc(kNKeys));
    SCK(cursor.alloc(kNKeys + 1));
    SCK(cudaMemsetAsync(count.p, 0, kNKeys * sizeof(uint32_t), st));
    if (total) {
        translate_kernel<<<dim3(grid_for(fr.len[0], kTransTile), 2), kTransThreads, 0, st>>>(g.p, len, fr);
        segment_kernel<<<grid_for(nseg * 32, 256), 256, 0, st>>>(fr, first.p, last.p, nseg);
        segment_scan<<<6, kScanThreads, 0, st>>>(fr, first.p, last.p, before.p, after.p);
        kmer_kernel<<<grid_for(nseg * 32, kKmerWarps * 32), kKmerWarps * 32, 0, st>>>(
            fr, before.p, after.p, nseg, 0, count.p, nullptr, nullptr);
        SCK(cudaGetLastError());
    }
    mp_index *idx = new (std::nothrow) mp_index();
    if (!idx) return MP_ENOMEM;
    idx->device = dev;
    for (uint64_t bin = len / kBin; bin; bin >>= 1) ++idx->xbits;
    auto fail = [&](int rc) {
        mp_index_free(idx);
        return rc;
    };
    if (cudaMalloc(&idx->off, (kNKeys + 1ull) * sizeof(uint32_t)) != cudaSuccess) return fail(MP_ENOMEM);
    int rc = scan_counts(count.p, kNKeys, idx->off, st);
    if (rc != MP_OK) return fail(rc);
    uint32_t n_entries = 0;
    if (cudaMemcpy(&n_entries, idx->off + kNKeys, sizeof(uint32_t), cudaMemcpyDeviceToHost) != cudaSuccess)
        return fail(MP_ECUDA);
    idx->n_entries = n_entries;
    if (cudaMalloc(&idx->entries, (n_entries ? n_entries : 1) * sizeof(uint32_t)) != cudaSuccess)
        return fail(MP_ENOMEM);
    if (total) {
        if (cudaMemcpyAsync(cursor.p, idx->off, kNKeys * sizeof(uint32_t), cudaMemcpyDeviceToDevice, st) !=
            cudaSuccess)
            return fail(MP_ECUDA);
        kmer_kernel<<<grid_for(nseg * 32, kKmerWarps * 32), kKmerWarps * 32, 0, st>>>(
            fr, before.p, after.p, nseg, 1, nullptr, cursor.p, idx->entries);
        bucket_sort_kernel<<<kNKeys / 32 / kBucketWarps, kBucketWarps * 32, 0, st>>>(idx->off, idx->entries);
    }
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) return fail(MP_ECUDA);
    *out = idx;
    return MP_OK;
}

extern "C" int mp_index_download(mp_dp_ctx *ctx, const mp_index *idx, uint64_t *offsets, uint32_t *entries,
                                 uint64_t *n_entries)
{
    if (!ctx || !idx || !n_entries || (!offsets) != (!entries)) return MP_EINVAL;
    if (cudaSetDevice(idx->device) != cudaSuccess) return MP_ECUDA;
    *n_entries = idx->n_entries;
    if (!offsets) return MP_OK;
    std::vector<uint32_t> off(kNKeys + 1ull);
    if (cudaMemcpy(off.data(), idx->off, off.size() * sizeof(uint32_t), cudaMemcpyDeviceToHost) != cudaSuccess ||
        (idx->n_entries && cudaMemcpy(entries, idx->entries, idx->n_entries * sizeof(uint32_t),
                                      cudaMemcpyDeviceToHost) != cudaSuccess))
        return MP_ECUDA;
    for (size_t h = 0; h < off.size(); ++h) offsets[h] = off[h];
    return MP_OK;
}

extern "C" void mp_index_free(mp_index *idx)
{
    if (!idx) return;
    cudaSetDevice(idx->device);
    if (idx->off) cudaFree(idx->off);
    if (idx->entries) cudaFree(idx->entries);
    delete idx;
}

extern "C" int mp_index_chain(mp_dp_ctx *ctx, const mp_index *idx, const char *prot, const uint64_t *prot_off,
                              const uint32_t *prot_len, uint32_t n_prot, int32_t top, mp_chain *chains,
                              uint32_t *n_chains)
{
    if (!ctx || !idx || top < 1 || (n_prot && (!prot || !prot_off || !prot_len || !chains || !n_chains)))
        return MP_EINVAL;
    if (n_prot == 0) return MP_OK;
    if (cudaSetDevice(ctx_device(ctx)) != cudaSuccess || idx->device != ctx_device(ctx)) return MP_ECUDA;
    cudaStream_t st = ctx_stream(ctx);
    uint64_t span = 0;
    for (uint32_t k = 0; k < n_prot; ++k) {
        if (prot_len[k] >= (1u << 20)) return MP_EINVAL;         // residue positions are 20-bit in the anchor keys
        span = std::max<uint64_t>(span, prot_off[k] + prot_len[k]);
    }
    Tmp<char> d_prot;
    Tmp<uint64_t> d_off, d_cnt, d_anc_off;
    Tmp<uint32_t> d_len, d_nch;
    Tmp<mp_chain> d_ch;
    SCK(d_prot.alloc(span));
    SCK(d_off.alloc(n_prot));
    SCK(d_len.alloc(n_prot));
    SCK(d_cnt.alloc(n_prot));
    SCK(d_anc_off.alloc(n_prot + 1ull));
    SCK(d_nch.alloc(n_prot));
    SCK(d_ch.alloc(static_cast<uint64_t>(n_prot) * top));
    SCK(cudaMemcpyAsync(d_prot.p, prot, span, cudaMemcpyHostToDevice, st));
    SCK(cudaMemcpyAsync(d_off.p, prot_off, n_prot * sizeof(uint64_t), cudaMemcpyHostToDevice, st));
    SCK(cudaMemcpyAsync(d_len.p, prot_len, n_prot * sizeof(uint32_t), cudaMemcpyHostToDevice, st));
    Tmp<int32_t> d_log;
    SCK(d_log.alloc(kG));
    log_table_kernel<<<grid_for(kG, 256), 256, 0, st>>>(d_log.p);
    ChainArgs a{};
    a.log_tab = d_log.p;
    a.prot = d_prot.p;
    a.prot_off = d_off.p;
    a.prot_len = d_len.p;
    a.n_prot = n_prot;
    a.off = idx->off;
    a.entries = idx->entries;
    a.top = top;
    a.chains = d_ch.p;
    a.n_chains = d_nch.p;
    anchor_count_kernel<<<grid_for(n_prot * 32ull, 256), 256, 0, st>>>(a, d_cnt.p);
    SCK(cudaGetLastError());
    std::vector<uint64_t> cnt(n_prot);
    SCK(cudaMemcpyAsync(cnt.data(), d_cnt.p, n_prot * sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
    SCK(cudaStreamSynchronize(st));
    if (!few_enough(cnt)) return MP_ETOOLARGE;
    // proteins in groups whose anchors (8 + 8 + 8 + 4 + 1 bytes each) stay within
    // a bound
    constexpr uint64_t kMaxAnchors = 192ull << 20;
    for (uint32_t p0 = 0; p0 < n_prot;) {
        uint32_t p1 = p0;
        uint64_t tot = 0;
        while (p1 < n_prot && (p1 == p0 || tot + cnt[p1] <= kMaxAnchors)) tot += cnt[p1++];
        const uint32_t np = p1 - p0;
        std::vector<uint64_t> aoff(np + 1ull, 0);
        std::vector<uint32_t> order(np);
        for (uint32_t k = 0; k < np; ++k) order[k] = k;
        std::stable_sort(order.begin(), order.end(),
                         [&](uint32_t x, uint32_t y) { return cnt[p0 + x] > cnt[p0 + y]; });
        for (uint32_t k = 0; k < np; ++k) aoff[k + 1] = aoff[k] + cnt[p0 + k];
        Tmp<uint64_t> anc, sc;
        Tmp<int64_t> f;
        Tmp<int32_t> pred;
        Tmp<uint8_t> mark;
        Tmp<int64_t> tmax;
        Tmp<uint32_t> d_order;
        SCK(d_order.alloc(np));
        SCK(cudaMemcpyAsync(d_order.p, order.data(), np * sizeof(uint32_t), cudaMemcpyHostToDevice, st));
        SCK(tmax.alloc(tot / 32 + 2ull * np + 2));
        SCK(anc.alloc(tot));
        SCK(f.alloc(tot));
        SCK(pred.alloc(tot));
        SCK(mark.alloc(tot));
        SCK(sc.alloc(tot));
        SCK(cudaMemcpyAsync(d_anc_off.p, aoff.data(), (np + 1ull) * sizeof(uint64_t), cudaMemcpyHostToDevice, st));
        ChainArgs b = a;
        b.prot_off = d_off.p + p0;
        b.prot_len = d_len.p + p0;
        b.n_prot = np;
        b.anc_off = d_anc_off.p;
        b.anc = anc.p;
        b.f = f.p;
        b.pred = pred.p;
        b.mark = mark.p;
        b.tmax = tmax.p;
        b.order = d_order.p;
        b.chains = d_ch.p + static_cast<uint64_t>(p0) * top;
        b.n_chains = d_nch.p + p0;
        anchor_fill_kernel<<<grid_for(np * 32ull, 256), 256, 0, st>>>(b);
        anchor_sort_kernel<<<np < 65535u * 4 ? np : 65535u * 4, kSortThreads, 0, st>>>(b, sc.p, idx->xbits);
        if (sort_passes(idx->xbits) % 2) b.anc = sc.p;
        chain_kernel<<<np < 65535u * 16 ? np : 65535u * 16, kStrandWarps * 64, 0, st>>>(b);
        SCK(cudaGetLastError());
        SCK(cudaStreamSynchronize(st));
        p0 = p1;
    }
    SCK(cudaMemcpyAsync(chains, d_ch.p, static_cast<uint64_t>(n_prot) * top * sizeof(mp_chain),
                        cudaMemcpyDeviceToHost, st));
    SCK(cudaMemcpyAsync(n_chains, d_nch.p, n_prot * sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
    SCK(cudaStreamSynchronize(st));
    return MP_OK;
}

extern "C" int mp_chain_refine(mp_dp_ctx *ctx, const mp_pair *pairs, size_t n, mp_chain2 *out)
{
    if (!ctx || (n && (!pairs || !out))) return MP_EINVAL;
    if (n == 0) return MP_OK;
    if (n >= (1ull << 31)) return MP_EINVAL;
    // every pair's protein and region, one after the other
    std::vector<uint64_t> poff(n), toff(n);
    std::vector<uint32_t> plen(n), tlen(n);
    std::vector<int8_t> strand(n);
    uint64_t tot = 0;
    for (size_t k = 0; k < n; ++k) {
        const mp_pair &q = pairs[k];
        // (the longest regions that the call takes, as its header says: the anchors
        // of one pair are chained by one block, each against those within G)
        if ((q.prot_len && !q.prot) || (q.nt_len && !q.nt) || q.prot_len > static_cast<uint32_t>(kRefineMaxProt) ||
            (q.strand != 1 && q.strand != -1) ||
            (static_cast<uint64_t>(q.nt_len) / 256 + 1) * q.prot_len >= (1ull << 32))
            return MP_EINVAL;
        poff[k] = tot;
        tot += q.prot_len;
        toff[k] = tot;
        tot += q.nt_len;
        plen[k] = q.prot_len;
        tlen[k] = q.nt_len;
        strand[k] = q.strand;
    }
    std::vector<CopyPiece> pieces(2 * n);
    for (size_t k = 0; k < n; ++k) {
        pieces[2 * k] = CopyPiece{pairs[k].prot, poff[k], plen[k]};
        pieces[2 * k + 1] = CopyPiece{pairs[k].nt, toff[k], tlen[k]};
    }
    if (cudaSetDevice(ctx_device(ctx)) != cudaSuccess) return MP_ECUDA;
    cudaStream_t st = ctx_stream(ctx);
    Tmp<char> d_seq;
    Tmp<uint64_t> d_poff, d_toff, d_cnt, d_aoff;
    Tmp<uint32_t> d_plen, d_tlen;
    Tmp<int8_t> d_strand;
    Tmp<int32_t> d_log;
    Tmp<mp_chain2> d_out;
    SCK(d_seq.alloc(tot));
    SCK(d_poff.alloc(n));
    SCK(d_toff.alloc(n));
    SCK(d_plen.alloc(n));
    SCK(d_tlen.alloc(n));
    SCK(d_strand.alloc(n));
    SCK(d_cnt.alloc(n));
    SCK(d_aoff.alloc(n + 1));
    SCK(d_log.alloc(kG));
    SCK(d_out.alloc(n));
    // (gathered into a fresh host vector and sent from there, pageable, the
    // sequences of 6,000 regions took 6 ms)
    const int sent = ctx_send_pieces(ctx, pieces.data(), pieces.size(), tot, d_seq.p);
    if (sent != MP_OK) return sent;
    SCK(cudaMemcpyAsync(d_poff.p, poff.data(), n * sizeof(uint64_t), cudaMemcpyHostToDevice, st));
    SCK(cudaMemcpyAsync(d_toff.p, toff.data(), n * sizeof(uint64_t), cudaMemcpyHostToDevice, st));
    SCK(cudaMemcpyAsync(d_plen.p, plen.data(), n * sizeof(uint32_t), cudaMemcpyHostToDevice, st));
    SCK(cudaMemcpyAsync(d_tlen.p, tlen.data(), n * sizeof(uint32_t), cudaMemcpyHostToDevice, st));
    SCK(cudaMemcpyAsync(d_strand.p, strand.data(), n, cudaMemcpyHostToDevice, st));
    log_table_kernel<<<grid_for(kG, 256), 256, 0, st>>>(d_log.p);
    RefineArgs a{};
    a.seq = d_seq.p;
    a.prot_off = d_poff.p;
    a.nt_off = d_toff.p;
    a.prot_len = d_plen.p;
    a.nt_len = d_tlen.p;
    a.strand = d_strand.p;
    a.log_tab = d_log.p;
    const uint32_t nb = static_cast<uint32_t>(n < 65535ull * 8 ? n : 65535ull * 8);
    // the k-mer table of the longest protein, a power of two of them
    size_t table = 1;
    for (size_t k = 0; k < n; ++k)
        while (table + kK2 - 1 < plen[k]) table <<= 1;
    const size_t smem = table * sizeof(uint64_t);
    SCK(cudaFuncSetAttribute(refine_anchor_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kRefineMaxProt * sizeof(uint64_t))));
    SCK(cudaFuncSetAttribute(refine_anchor_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kRefineMaxProt * sizeof(uint64_t))));
    a.n = static_cast<uint32_t>(n);
    refine_anchor_kernel<false><<<nb, kRefineThreads, smem, st>>>(a, d_cnt.p);
    SCK(cudaGetLastError());
    std::vector<uint64_t> per(n);
    SCK(cudaMemcpyAsync(per.data(), d_cnt.p, n * sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
    SCK(cudaStreamSynchronize(st));
    if (!few_enough(per)) return MP_ETOOLARGE;
    // pairs in groups whose anchors (8 + 8 + 4 bytes each) stay within a bound
    constexpr uint64_t kMaxAnchors = 192ull << 20;
    for (size_t p0 = 0; p0 < n;) {
        size_t p1 = p0;
        uint64_t na = 0;
        while (p1 < n && (p1 == p0 || na + per[p1] <= kMaxAnchors)) na += per[p1++];
        const uint32_t np = static_cast<uint32_t>(p1 - p0);
        std::vector<uint64_t> aoff(np + 1ull, 0);
        for (uint32_t k = 0; k < np; ++k) aoff[k + 1] = aoff[k] + per[p0 + k];
        Tmp<uint64_t> anc;
        Tmp<int64_t> f;
        Tmp<int32_t> pred;
        SCK(anc.alloc(na));
        SCK(f.alloc(na));
        SCK(pred.alloc(na));
        SCK(cudaMemcpyAsync(d_aoff.p, aoff.data(), (np + 1ull) * sizeof(uint64_t), cudaMemcpyHostToDevice, st));
        RefineArgs b = a;
        b.prot_off = d_poff.p + p0;
        b.nt_off = d_toff.p + p0;
        b.prot_len = d_plen.p + p0;
        b.nt_len = d_tlen.p + p0;
        b.strand = d_strand.p + p0;
        b.n = np;
        b.anc_off = d_aoff.p;
        b.anc = anc.p;
        b.f = f.p;
        b.pred = pred.p;
        b.out = d_out.p + p0;
        const uint32_t gb = np < 65535u * 8 ? np : 65535u * 8;
        refine_anchor_kernel<true><<<gb, kRefineThreads, smem, st>>>(b, nullptr);
        refine_chain_kernel<<<grid_for(np * 32ull, kRefineWarps * 32), kRefineWarps * 32, 0, st>>>(b);
        refine_chain_block_kernel<<<gb, kRefineThreads, 0, st>>>(b);
        SCK(cudaGetLastError());
        SCK(cudaStreamSynchronize(st));
        p0 = p1;
    }
    SCK(cudaMemcpyAsync(out, d_out.p, n * sizeof(mp_chain2), cudaMemcpyDeviceToHost, st));
    SCK(cudaStreamSynchronize(st));
    return MP_OK;
}
