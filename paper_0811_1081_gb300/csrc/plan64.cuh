// How the FP64 kernel stages R in shared memory (plain C++, no CUDA): rows per chunk,
// chunks, bytes.
#pragma once

#include <cstddef>

namespace gspca {

constexpr int kBlock64 = 512;
constexpr int kWarps64 = kBlock64 / 32;
constexpr int kMaxRc64 = 4;     // rows per staged chunk
constexpr int kDotWarps64 = 8;  // warps that form the row sums of a chunk, two per scheduler
constexpr int kTmp64 = kWarps64 * 32;

// Bytes of dynamic shared memory for rows of ldr doubles, nbuf chunks of rc rows, ldk, a slice
// (the layout is carve64's).
constexpr size_t smem64_bytes(int ldr, int nbuf, int rc, int ldk, int max_slice) {
    const size_t chunk = (size_t)nbuf * rc * ldr;
    return sizeof(double) * (2 * (size_t)ldr + chunk + kMaxRc64 * (kDotWarps64 + 4) + 2 * (size_t)ldk + max_slice +
                             (chunk >= kTmp64 ? 0 : kTmp64));
}

struct Chunks64 {
    int rc;    // rows per chunk; 0 where not even one row fits
    int nbuf;  // 3: one each copied, in the row sums and in the column sums; 1: one after another
    size_t bytes;
};

// Three chunks of four rows where they fit in `avail` bytes (ldr up to about 2000), else one
// chunk of as many rows as fit.  A stage costs the latency of its row sums whatever its rows are
// (5.1 us for 5000 columns with one row or with three), so rows come before overlap: 1000 x
// 2500, NIPALS, K = 4, 15 iterations, 1.86 ms with one chunk of four rows and 2.63 with three of
// two; 1000 x 5000, 3.50 with one of three rows and 6.32 with three of one.
inline Chunks64 plan_chunks64(int ldr, int ldk, int max_slice, long avail) {
    Chunks64 p{0, 1, 0};
    if ((long)smem64_bytes(ldr, 3, kMaxRc64, ldk, max_slice) <= avail) {
        p.rc = kMaxRc64;
        p.nbuf = 3;
    }
    for (int r = kMaxRc64; p.rc == 0 && r > 0; --r)
        if ((long)smem64_bytes(ldr, 1, r, ldk, max_slice) <= avail) p.rc = r;
    p.bytes = smem64_bytes(ldr, p.nbuf, p.rc > 0 ? p.rc : 1, ldk, max_slice);
    return p;
}

}  // namespace gspca
