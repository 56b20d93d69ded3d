// How the FP64 kernel stages R in shared memory (plain C++, no CUDA): rows per chunk,
// chunks, bytes.
#pragma once

#include <cstddef>
#include <initializer_list>

namespace gspca {

constexpr int kBlock64 = 512;
constexpr int kWarps64 = kBlock64 / 32;
constexpr int kMaxRc64 = 4;     // rows per staged chunk
constexpr int kDotWarps64 = 8;  // warps that form the row sums of a chunk, two per scheduler
constexpr int kTmp64 = kWarps64 * 32;
// Short rows (kernel variant of its own): chunks of kShortRc64 rows, four to each of those warps;
// the columns, at most 128 pairs, leave at least two of the other 256 threads for each pair
constexpr int kShortLdr64 = 256;
constexpr int kShortRc64 = 4 * kDotWarps64;

// Bytes of dynamic shared memory for rows of ldr doubles, nbuf chunks of rc rows, ldk, a slice
// (the layout is carve64's).
constexpr size_t smem64_bytes(int ldr, int nbuf, int rc, int ldk, int max_slice) {
    const size_t chunk = (size_t)nbuf * rc * ldr, rv = rc > kMaxRc64 ? rc : kMaxRc64;
    return sizeof(double) * (2 * (size_t)ldr + chunk + kMaxRc64 * kDotWarps64 + 4 * rv + 2 * (size_t)ldk + max_slice +
                             (chunk >= kTmp64 ? 0 : kTmp64));
}

struct Chunks64 {
    int rc;    // rows per chunk; 0 where not even one row fits
    int nbuf;  // 3: one each copied, in the row sums and in the column sums; 1: one after another
    size_t bytes;
};

// Short rows: a stage costs its copy's latency, the barriers and one butterfly whatever its rows
// are, so it takes 32 of them (100000 x 60, NIPALS, K = 4, 15 iterations: 18.4 ms with four, 3.71
// with 32), unless the CTA has no more than two stages of the general form hold: the column shares
// are added behind the sweep (1800 x 256, 12 rows a CTA: 1.23 and 1.15; 1200 x 200, 8 rows: 1.09
// and 1.13; 300 x 60, 2 rows: 0.97 and 1.00).  Longer ones: three chunks of
// four rows where they fit in `avail` bytes (ldr up to about 2000), else one chunk of as many rows
// as fit, for the same reason (the row sums of a chunk of 5000 columns take 5.1 us with one row or
// with three) rows before overlap: 1000 x 2500, same fit, 1.86 ms with one chunk of four rows and
// 2.63 with three of two; 1000 x 5000, 3.50 with one of three rows and 6.32 with three of one.
// `rows`: the most rows of a CTA.
inline Chunks64 plan_chunks64(int rows, int ldr, int ldk, int max_slice, long avail) {
    Chunks64 p{0, 1, 0};
    for (const int r : {ldr <= kShortLdr64 && rows > 2 * kMaxRc64 ? kShortRc64 : 0, kMaxRc64})
        if (p.rc == 0 && r > 0 && (long)smem64_bytes(ldr, 3, r, ldk, max_slice) <= avail) {
            p.rc = r;
            p.nbuf = 3;
        }
    for (int r = kMaxRc64; p.rc == 0 && r > 0; --r)
        if ((long)smem64_bytes(ldr, 1, r, ldk, max_slice) <= avail) p.rc = r;
    p.bytes = smem64_bytes(ldr, p.nbuf, p.rc > 0 ? p.rc : 1, ldk, max_slice);
    return p;
}

}  // namespace gspca
