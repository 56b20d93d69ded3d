// FP64 storage path: NIPALS-PCA (Sec. 2.2) and GS-PCA (Sec. 2.3) with R, the
// factors and every product in IEEE double, the precision of the paper's
// programs (Sec. 3).  One persistent cooperative launch runs every iteration
// of every component, as the FP32 kernel does, in a simpler form:
//   - R is row-major (rows of ldr doubles, N rounded up to even); CTA g owns the rows
//     [r0, r1) and the column slice [n0, n1);
//   - one sweep per iteration: the CTA's rows reach shared memory in chunks of
//     rc rows (one bulk copy each), v' = R u' is formed per row and, from the same chunk,
//     s' = R^T v' is accumulated per column (a thread per two columns);
//   - the Gram-Schmidt score correction commutes through R^T: R^T (v' - V b')
//     = s' - W b', with W = R^T V kept by a rank-1 update per deflation, so the
//     loading needs no second read of R;
//   - two grid-wide reductions per GS iteration (after the pass: s', b', ||v'||^2 and the
//     loading's squared norm; after the score step: a' = U^T u_pre') and one barrier
//     that publishes the next loading, every cross-CTA sum in a fixed order, so two
//     runs give the same bits;
//   - the deflation of component k-1 (Eq. 3) is applied inside the sweep that
//     takes the start column R(k) of component k.
// GB300 executes FP64 at 1/64 of its FP32 rate (2 FMAs per clock and SM), so the 2 M N
// FMAs of a sweep bound this path: 4000 x 1500, 19 us at that rate; the sweep takes 29 and
// the iteration 48 (122 in the form before: rows summed a warp each, sums over CTAs as one
// thread's chain of 152 loads, roots and quotients in every thread).  So everything else is
// arranged to cost few FP64 instructions and little latency: four rows share one
// butterfly, a sum over CTAs is one round of loads of half a warp, one warp takes the
// scalars while the others form u_pre'.
#pragma once

#include <cfloat>

#include "device_common.cuh"
#include "plan64.cuh"

namespace gspca {

struct Fit64Args {
    int M, N, K;
    int ldr;                  // doubles between rows of R: N rounded up to even
    int algo;                 // 0 = NIPALS, 1 = GS
    int max_iter;
    double tol;
    double eps_thresh;        // degenerate threshold factor: lambda <= eps_thresh * ||X||_F
    const double* xpart;      // partial sums of squares of the packed X
    int nxpart;
    double* R;                // M x ldr row-major (the padding column is zero)
    double* V;                // M x ldk row-major (GS: unit score directions; NIPALS: scores t)
    double* U;                // N x ldk row-major (loadings)
    double* W;                // N x ldk row-major (R^T V, GS)
    int ldk;
    double* vraw;             // M: v' of the last pass
    double* ut;               // 2 x N: pass input, double-buffered
    double* upre;             // N: s' - W b' of the last iteration (pass scale)
    double* partS;            // G x LS: s' (or s0, column norms) partials, then the k-vector
    int LS;
    double* partA;            // G x LA: a' partials
    int LA;                   // ldk rounded up to a sector
    double* scal;             // G x 4: [0] ||v'||^2 / ||x||^2, [1] ||v' - V b'||^2, [2+b] ||ut[b]||^2
    double* lam;              // K
    int* iters;               // K
    int* info;                // status, found, total iterations (lo, hi)
    unsigned* flags;          // barrier arrival counter, zeroed before the launch
    int* abort;
    const int* iters_lock;    // device, K entries, nullable
    unsigned long long timeout_ns;
    int rc;                   // rows per staged chunk (kShortRc64: the kernel for short rows)
    int nbuf;                 // chunks in shared memory: 3 (one each copied, in the row sums and in the
                              // column sums) or 1 (one after another)
};

// Shared memory (dynamic): u and the s accumulators (ldr each), nbuf chunks (rc x ldr), then
// small vectors: row-sum parts (kMaxRc64 x kDotWarps64), row values and deflation weights
// (2 x rv each, rv = rc or kMaxRc64 if that is more), kb, ka (ldk), the slice (max N / G + 1).  rows_t64's scratch (kTmp64 doubles) is
// the chunk memory, idle then, or follows where that is smaller.
struct Smem64 {
    double* u;
    double* s;
    double* ch;
    double* part;
    double* rowv;
    double* cf;
    double* kb;
    double* ka;
    double* sl;
    double* tmp;
};

__device__ __forceinline__ Smem64 carve64(unsigned char* dyn, const Fit64Args& f, int max_slice) {
    Smem64 m;
    double* p = reinterpret_cast<double*>(dyn);
    m.u = p;
    p += f.ldr;
    m.s = p;
    p += f.ldr;
    m.ch = p;
    p += (size_t)f.nbuf * f.rc * f.ldr;
    m.part = p;
    p += kMaxRc64 * kDotWarps64;
    m.rowv = p;
    p += 2 * max(f.rc, kMaxRc64);
    m.cf = p;
    p += 2 * max(f.rc, kMaxRc64);
    m.kb = p;
    p += f.ldk;
    m.ka = p;
    p += f.ldk;
    m.sl = p;
    m.tmp = f.nbuf * f.rc * f.ldr >= kTmp64 ? m.ch : p + max_slice;
    return m;
}

// Lanes that share a row of kk values: the power of two that holds kk, at most 32.
__device__ __forceinline__ int lane_group(int kk) {
    int gw = 1;
    while (gw < kk && gw < 32) gw *= 2;
    return gw;
}

// The CTA's sum of the values v of every warp's lanes 0, gw, 2 gw, ..., in a fixed order; the
// result in every thread.  One warp adds: an FP64 instruction of all 16 warps takes the SM's FP64
// pipe 256 clocks.
__device__ __forceinline__ double lanes_sum64(double v, int gw, double* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncwarp();
    for (int o = 16; o >= gw; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        double t = lane < kWarps64 ? red[lane] : 0.0;
#pragma unroll
        for (int o = kWarps64 / 2; o >= 1; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
        __syncwarp();
        if (lane == 0) red[0] = t;
    }
    __syncthreads();
    return red[0];
}

// The same over lanes 0, 8, 16 and 24 of warp 0 (the other values are not read).
__device__ __forceinline__ double block_sum64_warp0(double v, double* red) {
    __syncthreads();
    if (threadIdx.x < 32) {
        v += __shfl_xor_sync(kFull, v, 16);
        v += __shfl_xor_sync(kFull, v, 8);
        if (threadIdx.x == 0) red[0] = v;
    }
    __syncthreads();
    return red[0];
}

// CTA-wide sum of one double per thread, in a fixed order; the result in every thread.
__device__ __forceinline__ double block_sum64(double v, double* red) { return lanes_sum64(v, 1, red); }

// out(t) = the sum over the G CTAs of value t (at src(t), `stride(t)` doubles between CTAs),
// t < n: 16 lanes per value; a lane adds CTAs sub, sub + 16, ... in order (10 loads under way
// at once cover 152 CTAs), then a fixed butterfly.  Ends with a CTA barrier.
template <class Src, class Stride, class Out>
__device__ __forceinline__ void team_sums64(int G, int n, Src src, Stride stride, Out out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane & 15;
    for (int tb = warp * 2; tb < n; tb += 2 * kWarps64) {
        const int t = tb + (lane >> 4);
        double x = 0.0;
        if (t < n) {
            const double* a = src(t);
            const size_t st = stride(t);
#pragma unroll 10
            for (int g = sub; g < G; g += 16) x += __ldcg(a + g * st);
        }
        __syncwarp();
        x += __shfl_xor_sync(kFull, x, 8);
        x += __shfl_xor_sync(kFull, x, 4);
        x += __shfl_xor_sync(kFull, x, 2);
        x += __shfl_xor_sync(kFull, x, 1);
        if (sub == 0 && t < n) out(t, x);
    }
    __syncthreads();
}

// out(t) = the sum over the G CTAs of vec[t], t < n (`stride` doubles between CTAs, a multiple of
// four).  All CTAs read the vector at the same time, so its few lines are what the L2 is
// asked for: four neighbouring values (one sector) go to four lanes, the CTAs to the rest of
// the warp and to the W warps that share four values; the warps' parts are added in order
// through tmp (4 x kWarps64).  k = 10 and 152 CTAs: 2.2 us, 4.2 with team_sums64.  Ends with a CTA
// barrier.
template <class Out>
__device__ __forceinline__ void team_vec64(int G, int n, const double* vec, size_t stride, double* tmp, Out out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nq = (n + 3) / 4, W = nq < kWarps64 ? kWarps64 / nq : 1;
    for (int unit = warp; unit < nq * W; unit += kWarps64) {
        const int q = unit / W, p = unit % W, t = 4 * q + (lane & 3);
        double x = 0.0;
        if (t < n) {
            const double* a = vec + t;
#pragma unroll 5
            for (int g = 8 * p + (lane >> 2); g < G; g += 8 * W) x += __ldcg(a + g * stride);
        }
        __syncwarp();
        x += __shfl_xor_sync(kFull, x, 16);
        x += __shfl_xor_sync(kFull, x, 8);
        x += __shfl_xor_sync(kFull, x, 4);
        if (W > 1) {
            if (lane < 4) tmp[unit * 4 + lane] = x;
        } else if (lane < 4 && t < n) {
            out(t, x);
        }
        __syncwarp();
    }
    __syncthreads();
    if (W > 1) {
        if ((int)threadIdx.x < n) {
            const int t = threadIdx.x;
            const double* a = tmp + (t >> 2) * W * 4 + (t & 3);
            double x = a[0];
            for (int p = 1; p < W; ++p) x += a[4 * p];
            out(t, x);
        }
        __syncthreads();
    }
}

// Chunks of R on their way to shared memory: chunk q (counted on from sweep to sweep) is one
// bulk copy into buffer q % nbuf and completes phase q / nbuf of its mbarrier.
struct Ring64 {
    uint64_t* bar;
    unsigned base;    // number of the next sweep's first chunk
    unsigned issued;  // number of the next chunk to be copied
    bool dead;        // a copy did not arrive within the bound

    __device__ __forceinline__ int slot(const Fit64Args& f, unsigned q) const { return f.nbuf > 1 ? (int)(q % 3) : 0; }
    __device__ __forceinline__ unsigned phase(const Fit64Args& f, unsigned q) const {
        return (f.nbuf > 1 ? q / 3 : q) & 1u;
    }
    // Starts the copy of chunk i of rows [r0, r1) unless it is under way.  Its buffer is free:
    // last used before a CTA barrier, and whoever wrote to it fenced before that.
    __device__ __forceinline__ void issue(const Fit64Args& f, const Smem64& m, int r0, int r1, int i) {
        if (dead || issued != base + i || r0 + i * f.rc >= r1) return;
        if (threadIdx.x == kBlock64 - 32) {
            const int rb = r0 + i * f.rc, s = slot(f, issued);
            tma_load_1d(m.ch + (size_t)s * f.rc * f.ldr, f.R + (size_t)rb * f.ldr,
                        (uint32_t)(min(f.rc, r1 - rb) * f.ldr * sizeof(double)), &bar[s]);
        }
        ++issued;
    }
    // Behind a sweep of n chunks.
    __device__ __forceinline__ void advance(int n) {
        base += n;
        if (!dead) {  // slot and phase repeat every six chunks
            const unsigned d = base / 6 * 6;
            base -= d;
            issued -= d;
        }
    }
    // Waits for chunk i.
    __device__ __forceinline__ void wait(const Fit64Args& f, int i) {
        if (!dead && !mbar_wait(&bar[slot(f, base + i)], phase(f, base + i), f.timeout_ns)) {
            atomicCAS(f.abort, 0, kStTimeout);
            dead = true;
        }
    }
};

__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async;" ::: "memory"); }

// One sweep over the CTA's rows [r0, r1).
//   start == false: row value x_r = R_r . u (u in smem), written to vraw;
//   start == true:  with `deflate`, R_r <- R_r - a_r u^T first (a_r = lamf V[r, kprev],
//                   u = the previous loading in smem; the deflated rows are stored),
//                   then x_r = R[r, kcol].
// Both accumulate s[c] += R[r, c] x_r (smem, a thread per two columns) and return the
// CTA's sum of x_r^2 (every thread).  Sums run in row order within the CTA.
// Three chunks are in shared memory: in each stage warps 0-7 form the row values of chunk t
// while the others add chunk t - 1 to the columns and chunk t + 1 is copied, so the FP64
// pipe, which both share, is kept busy across the row sums' butterflies and the barriers
// (29 us for 4000 x 1500, 34 with one after the other).  A chunk's four rows are summed
// together by each of the eight warps over an eighth of the columns, and one butterfly
// reduces a lane's four sums (6 FP64 additions instead of 20).
__device__ __forceinline__ double sweep64(const Fit64Args& f, const Smem64& m, Ring64& rg, double* red, int r0, int r1,
                                          bool start, bool deflate, double lamf, int kprev, int kcol) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, T = blockDim.x;
    const int ldr = f.ldr, n2 = ldr >> 1, rc = f.rc;
    const size_t cstride = (size_t)rc * ldr;
    const int nchunks = (r1 - r0 + rc - 1) / rc;
    auto chunk = [&](int i) { return m.ch + rg.slot(f, rg.base + i) * cstride; };
    auto issue = [&](int i) {
        rg.issue(f, m, r0, r1, i);
        const int rb = r0 + i * rc;
        const int q = tid - 32 * kDotWarps64;
        if (deflate && q >= 0 && q < min(rc, r1 - rb))
            m.cf[(i & 1) * kMaxRc64 + q] = -lamf * f.V[(size_t)(rb + q) * f.ldk + kprev];
    };
    // u is in place; what the CTA wrote to the chunk memory or (deflation) to R before this
    // point precedes the copies
    fence_async_proxy();
    __syncthreads();
    double sq = 0.0;
    // row values of chunk i into rowv[i & 1] (warps 0-7; their own named barrier)
    auto rows = [&](int i) {
        const int rb = r0 + i * rc, nr = min(rc, r1 - rb);
        double* ch = chunk(i);
        double* rowv = m.rowv + (i & 1) * kMaxRc64;
        if (start) {
            if (deflate) {
                double cf[kMaxRc64];
#pragma unroll
                for (int r = 0; r < kMaxRc64; ++r) cf[r] = r < nr ? m.cf[(i & 1) * kMaxRc64 + r] : 0.0;
                for (int c = tid; c < n2; c += 32 * kDotWarps64) {
                    const double2 u = reinterpret_cast<const double2*>(m.u)[c];
#pragma unroll
                    for (int r = 0; r < kMaxRc64; ++r)
                        if (r < nr) {
                            double2* p = reinterpret_cast<double2*>(ch + (size_t)r * ldr) + c;
                            double2 v = *p;
                            v.x = fma(cf[r], u.x, v.x);
                            v.y = fma(cf[r], u.y, v.y);
                            *p = v;
                            reinterpret_cast<double2*>(f.R + (size_t)(rb + r) * ldr)[c] = v;
                        }
                }
                fence_async_proxy();
                asm volatile("barrier.sync 1, %0;" ::"n"(32 * kDotWarps64) : "memory");
            }
            if (warp == 0 && (lane & 7) == 0 && (lane >> 3) < nr) {
                const double x = ch[(size_t)(lane >> 3) * ldr + kcol];
                rowv[lane >> 3] = x;
                sq = fma(x, x, sq);
            }
            return;
        }
        const double2* p = reinterpret_cast<const double2*>(ch);
        const int c0 = (int)((long long)warp * n2 / kDotWarps64), c1 = (int)((long long)(warp + 1) * n2 / kDotWarps64);
        double a[4] = {0.0, 0.0, 0.0, 0.0};
        if (nr == 4) {
#pragma unroll 2
            for (int c = c0 + lane; c < c1; c += 32) {
                const double2 u = reinterpret_cast<const double2*>(m.u)[c];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const double2 d = p[q * n2 + c];
                    a[q] = fma(d.x, u.x, a[q]);
                    a[q] = fma(d.y, u.y, a[q]);
                }
            }
        } else {
            for (int c = c0 + lane; c < c1; c += 32) {
                const double2 u = reinterpret_cast<const double2*>(m.u)[c];
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    if (q < nr) {
                        const double2 d = p[q * n2 + c];
                        a[q] = fma(d.x, u.x, a[q]);
                        a[q] = fma(d.y, u.y, a[q]);
                    }
            }
        }
        const double t = warp_sum4(a);
        if ((lane & 7) == 0 && (lane >> 3) < nr) m.part[(lane >> 3) * kDotWarps64 + warp] = t;
        __syncwarp();
        asm volatile("barrier.sync 1, %0;" ::"n"(32 * kDotWarps64) : "memory");
        if (warp == 0) {  // lane = row * kDotWarps64 + part
            static_assert(kMaxRc64 * kDotWarps64 == 32, "a lane per part");
            double v = lane < nr * kDotWarps64 ? m.part[lane] : 0.0;
            v += __shfl_xor_sync(kFull, v, 4);
            v += __shfl_xor_sync(kFull, v, 2);
            v += __shfl_xor_sync(kFull, v, 1);
            if ((lane & 7) == 0 && (lane >> 3) < nr) {
                rowv[lane >> 3] = v;
                f.vraw[rb + (lane >> 3)] = v;
                sq = fma(v, v, sq);
            }
            __syncwarp();
        }
    };
    // columns: s += R^T x over chunk i, by the threads from t0 on
    auto cols = [&](int i, int t0) {
        const int nr = min(rc, r1 - (r0 + i * rc));
        const double2* p0 = reinterpret_cast<const double2*>(chunk(i));
        const double* rowv = m.rowv + (i & 1) * kMaxRc64;
        double x[kMaxRc64];
#pragma unroll
        for (int r = 0; r < kMaxRc64; ++r) x[r] = r < nr ? rowv[r] : 0.0;
        for (int c = tid - t0; c < n2; c += T - t0) {
            double2 a = i > 0 ? reinterpret_cast<double2*>(m.s)[c] : make_double2(0.0, 0.0);
#pragma unroll
            for (int r = 0; r < kMaxRc64; ++r)
                if (r < nr) {
                    const double2 d = p0[r * n2 + c];
                    a.x = fma(d.x, x[r], a.x);
                    a.y = fma(d.y, x[r], a.y);
                }
            reinterpret_cast<double2*>(m.s)[c] = a;
        }
    };
    if (nchunks == 0)
        for (int c = tid; c < ldr; c += T) m.s[c] = 0.0;
    if (f.nbuf > 1) {
        if (nchunks > 0) issue(0);
        for (int t = 0; t <= nchunks && nchunks > 0; ++t) {
            if (t < nchunks) rg.wait(f, t);
            __syncthreads();  // chunk t has landed, chunk t - 1's row values are formed, chunk t - 2 is free
            if (t + 1 < nchunks) issue(t + 1);
            if (warp < kDotWarps64) {
                if (t < nchunks) rows(t);
            } else if (t > 0) {
                cols(t - 1, 32 * kDotWarps64);
            }
        }
    } else {
        for (int i = 0; i < nchunks; ++i) {
            __syncthreads();
            issue(i);
            rg.wait(f, i);
            __syncthreads();
            if (warp < kDotWarps64) rows(i);
            __syncthreads();
            cols(i, 0);
        }
    }
    rg.advance(nchunks);
    return block_sum64_warp0(sq, red);
}

// The sweep for short rows (ldr <= kShortLdr64): chunks of kShortRc64 rows, so that a stage's fixed
// cost (copy latency, barrier, butterfly) is shared by 32 rows instead of four.  Warp w < 8 takes
// rows 4 w to 4 w + 3 of a chunk over all columns; the other 256 threads own a pair of columns
// and every S-th row of the chunk before, their sums stay in registers for the whole sweep and
// are added in a fixed order behind it.  100000 x 60, a NIPALS iteration: 288 us with four rows a
// stage, 58 so (FP64 pipe: 19).
__device__ __forceinline__ double sweep64_short(const Fit64Args& f, const Smem64& m, Ring64& rg, double* red, int r0,
                                                int r1, bool start, bool deflate, double lamf, int kprev, int kcol) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, T = blockDim.x;
    const int ldr = f.ldr, n2 = ldr >> 1, nd = 32 * kDotWarps64;
    constexpr int rc = kShortRc64;
    const size_t cstride = (size_t)rc * ldr;
    const int nchunks = (r1 - r0 + rc - 1) / rc;
    const int S = min((T - nd) / n2, 16);  // row shares of the column sums: S x ldr <= kTmp64
    const int c = (tid % nd) % n2, share = (tid % nd) / n2;
    double2 acc = make_double2(0.0, 0.0);
    double sq = 0.0;
    auto issue = [&](int i) {
        rg.issue(f, m, r0, r1, i);
        const int rb = r0 + i * rc, q = tid - nd;
        if (deflate && q >= 0 && q < min(rc, r1 - rb))
            m.cf[(i & 1) * rc + q] = -lamf * f.V[(size_t)(rb + q) * f.ldk + kprev];
    };
    // row values of chunk i into rowv[i & 1] (warps 0-7)
    auto rows = [&](int i) {
        const int rb = r0 + i * rc, nr = min(rc, r1 - rb);
        double* ch = m.ch + rg.slot(f, rg.base + i) * cstride;
        double* rowv = m.rowv + (i & 1) * rc;
        if (start) {
            if (deflate) {
                const double2 u = reinterpret_cast<const double2*>(m.u)[c];
                const int step = nd / n2;
                for (int r = share; share < step && r < nr; r += step) {
                    const double cf = m.cf[(i & 1) * rc + r];
                    double2* p = reinterpret_cast<double2*>(ch + (size_t)r * ldr) + c;
                    double2 v = *p;
                    v.x = fma(cf, u.x, v.x);
                    v.y = fma(cf, u.y, v.y);
                    *p = v;
                    reinterpret_cast<double2*>(f.R + (size_t)(rb + r) * ldr)[c] = v;
                }
                fence_async_proxy();
                asm volatile("barrier.sync 1, %0;" ::"n"(32 * kDotWarps64) : "memory");
            }
            if (tid < nr) {
                const double x = ch[(size_t)tid * ldr + kcol];
                rowv[tid] = x;
                sq = fma(x, x, sq);
            }
            return;
        }
        if (4 * warp >= nr) return;
        const double2* p = reinterpret_cast<const double2*>(ch) + 4 * warp * n2;  // rows past nr: read, not used
        double a[4] = {0.0, 0.0, 0.0, 0.0};
        for (int j = lane; j < n2; j += 32) {
            const double2 u = reinterpret_cast<const double2*>(m.u)[j];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const double2 d = p[q * n2 + j];
                a[q] = fma(d.x, u.x, a[q]);
                a[q] = fma(d.y, u.y, a[q]);
            }
        }
        __syncwarp();
        const double v = warp_sum4(a);
        const int r = 4 * warp + (lane >> 3);
        if ((lane & 7) == 0 && r < nr) {
            rowv[r] = v;
            f.vraw[rb + r] = v;
            sq = fma(v, v, sq);
        }
    };
    // columns: this thread's share of s += R^T x over chunk i (warps 8-15)
    auto cols = [&](int i) {
        const int nr = min(rc, r1 - (r0 + i * rc));
        const double2* p = reinterpret_cast<const double2*>(m.ch + rg.slot(f, rg.base + i) * cstride) + c;
        const double* rowv = m.rowv + (i & 1) * rc;
        if (share < S)
#pragma unroll 2
            for (int r = share; r < nr; r += S) {
                const double2 d = p[r * n2];
                const double x = rowv[r];
                acc.x = fma(d.x, x, acc.x);
                acc.y = fma(d.y, x, acc.y);
            }
    };
    fence_async_proxy();
    __syncthreads();
    issue(0);
    for (int t = 0; t <= nchunks; ++t) {
        if (t < nchunks) rg.wait(f, t);
        __syncthreads();  // chunk t has landed, chunk t - 1's row values are formed, chunk t - 2 is free
        if (t + 1 < nchunks) issue(t + 1);
        if (warp < kDotWarps64) {
            if (t < nchunks) rows(t);
        } else if (t > 0) {
            cols(t - 1);
        }
    }
    rg.advance(nchunks);
    __syncthreads();  // the chunks are read: their memory takes the shares
    if (tid >= nd && share < S) {
        double* d = m.tmp + share * ldr + 2 * c;  // 8-byte aligned only, where it is not chunk memory
        d[0] = acc.x;
        d[1] = acc.y;
    }
    __syncthreads();
    if (tid < ldr) {
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        for (int q = 0; q < S; q += 4)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (q + e < S) v[e] += m.tmp[(q + e) * ldr + tid];
        m.s[tid] = (v[0] + v[1]) + (v[2] + v[3]);
    }
    return lanes_sum64(sq, start ? 1 : 8, red);
}

// dst[j] = sum_{r in [a0, a1)} A[r * lda + j] y(r), j < kk.  `gw` lanes take
// neighbouring columns, the warps and the rest of a warp share the rows; the parts are added
// in a fixed order through tmp (kWarps64 x 32).
template <class Y>
__device__ __forceinline__ void rows_t64(const double* A, int lda, int a0, int a1, int kk, Y y, double* dst,
                                         double* tmp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gw = lane_group(kk), per = 32 / gw, j0 = lane & (gw - 1);
    for (int jb = 0; jb < kk; jb += gw) {
        const int j = jb + j0;
        double t = 0.0;
        if (j < kk)
#pragma unroll 4
            for (int r = a0 + warp * per + lane / gw; r < a1; r += kWarps64 * per) t = fma(A[(size_t)r * lda + j], y(r), t);
        __syncwarp();
        for (int o = gw; o < 32; o <<= 1) t += __shfl_xor_sync(kFull, t, o);
        __syncthreads();  // tmp free
        if (lane < gw) tmp[warp * 32 + lane] = t;
        __syncthreads();
        if ((int)threadIdx.x < gw && jb + (int)threadIdx.x < kk) {
            double q[4];  // four chains: an FP64 addition waits long for the one before
#pragma unroll
            for (int i = 0; i < 4; ++i) q[i] = tmp[i * 32 + threadIdx.x];
#pragma unroll
            for (int w = 4; w < kWarps64; ++w) q[w & 3] += tmp[w * 32 + threadIdx.x];
            dst[jb + threadIdx.x] = (q[0] + q[1]) + (q[2] + q[3]);
        }
    }
}

// For every r in [a0, a1): fn(r, sum_j A[r * lda + j] x[j]) with x (kk) in smem; `gw` lanes
// (as above) per row, lanes over j, fixed butterfly; fn runs in a row's first lane.
template <class Fn>
__device__ __forceinline__ void rows_dot64(const double* A, int lda, int a0, int a1, int kk, const double* x, Fn fn) {
    const int lane = threadIdx.x & 31, warp = kWarps64 - 1 - (threadIdx.x >> 5);  // warp 0 is the last to get rows
    const int gw = lane_group(kk), per = 32 / gw, j0 = lane & (gw - 1);
#pragma unroll 2
    for (int rb = a0 + warp * per; rb < a1; rb += kWarps64 * per) {
        const int r = rb + lane / gw;
        double t = 0.0;
        if (r < a1)
            for (int j = j0; j < kk; j += gw) t = fma(A[(size_t)r * lda + j], x[j], t);
        __syncwarp();
        for (int o = gw >> 1; o >= 1; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
        if (j0 == 0 && r < a1) fn(r, t);
        __syncwarp();
    }
}

// Single problem, whole grid (cooperative launch), FP64 throughout.  Short: rows of at most
// kShortLdr64 doubles.
template <bool Short>
__global__ void __launch_bounds__(kBlock64, 1) fit64_kernel(const Fit64Args f) {
    extern __shared__ __align__(16) unsigned char dyn64[];
    __shared__ double red[kWarps64];
    __shared__ double sums[2];
    __shared__ double team[4 * kWarps64];  // parts of a sum over the CTAs
    __shared__ double scal[4];  // lambda, 1 / ||u'||, 1 / ||v'||, the next loading's scale
    __shared__ int s_stop, s_dead;
    __shared__ uint64_t mbar[3];
    __shared__ int s_flag;
    __shared__ double s_best[kWarps64];
    __shared__ int s_bidx[kWarps64];
    const int G = gridDim.x, g = blockIdx.x, tid = threadIdx.x, T = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5;
    const int M = f.M, N = f.N, K = f.K;
    const int r0 = (int)(((long long)g * M) / G), r1 = (int)(((long long)(g + 1) * M) / G);
    const int n0 = (int)(((long long)g * N) / G), n1 = (int)(((long long)(g + 1) * N) / G);
    const Smem64 m = carve64(dyn64, f, (N + G - 1) / G + 1);
    const int ldr = f.ldr, nc = n1 - n0;
    const GridBarrier bar{f.flags, f.abort, f.timeout_ns};
    unsigned epoch = 0;
    const bool gs = f.algo == 1;
    auto sweep = [&](Ring64& rg, bool start, bool deflate, double lamf, int kprev, int kcol) {
        if constexpr (Short) return sweep64_short(f, m, rg, red, r0, r1, start, deflate, lamf, kprev, kcol);
        else return sweep64(f, m, rg, red, r0, r1, start, deflate, lamf, kprev, kcol);
    };
    if (tid == 0) {
        for (int i = 0; i < 3; ++i) mbar_init(&mbar[i], 1);
        fence_mbar_init();
        s_dead = 0;
    }
    Ring64 rg{mbar, 0u, 0u, false};
    double xx = 0.0;  // ||X||_F^2 from the pack kernel's partials, in a fixed order
    for (int i = tid; i < f.nxpart; i += T) xx += f.xpart[i];
    xx = block_sum64(xx, red);
    const double thresh = f.eps_thresh * sqrt(xx);
    if (tid == 0 && ldr > N) m.u[N] = 0.0;  // the padding column's loading
    double* pS = f.partS + (size_t)g * f.LS;
    double* pA = f.partA + (size_t)g * f.LA;
    double* sc = f.scal + (size_t)g * 4;
    int status = kStOK, found = K;
    long long total = 0;
    bool alive = true;
    double lam_prev = 0.0, vinv_prev = 0.0, inv_nu = 0.0;
    double gram_dev = 0.0, cut = 0.25;  // warp 0: ||V^T V - I||_F^2, and what b'^T b' / ||v'||^2 may reach
    int buf = 0;

// Leaves the kernel when a copy of the sweep before did not arrive.
#define ALIVE64()                            \
    do {                                     \
        if (rg.dead) s_dead = 1;             \
        __syncthreads();                     \
        if (s_dead) {                        \
            alive = false;                   \
            goto leave64;                    \
        }                                    \
    } while (0)
#define SYNC64()                             \
    do {                                     \
        if (!bar.sync(epoch, &s_flag)) {     \
            alive = false;                   \
            goto leave64;                    \
        }                                    \
    } while (0)

    for (int k = 0; k < K && found == K; ++k) {
        // ------------- start: deflate component k-1 in the sweep that takes R(k)
        const bool defl = k > 0;
        const double lamf = gs ? lam_prev : 1.0;
        // u_{k-1} = the last pass input / its norm: complete behind the barrier before that pass
        // (U(k-1) itself was written slice by slice when the component stopped, with no barrier since)
        if (defl)
            for (int c = tid; c < N; c += T) m.u[c] = __ldcg(f.ut + (size_t)buf * N + c) * inv_nu;
        double xs = sweep(rg, true, defl, lamf, k - 1, k);
        ALIVE64();
        for (int c = tid; c < N; c += T) pS[c] = m.s[c];
        if (gs && k > 0)  // Gram row v_{k-1} . v_j over this CTA's rows
            rows_t64(f.V, f.ldk, r0, r1, k, [&](int r) { return f.V[(size_t)r * f.ldk + (k - 1)]; }, pS + N, m.tmp);
        if (tid == 0) sc[0] = xs;
        SYNC64();
        // ||x||^2, this CTA's slice of s0 and the Gram row
        const int nk = gs ? k : 0;
        auto gather_s = [&](int slot) {  // value 0 (and 1): scalars; then the slice; then the k-vector
            const int ns = slot >= 0 ? 2 : 1;
            team_sums64(
                G, ns + nc + nk,
                [&](int t) {
                    if (t < ns) return f.scal + (t == 0 ? 0 : slot);
                    return t < ns + nc ? f.partS + n0 + t - ns : f.partS + N + t - ns - nc;
                },
                [&](int t) { return t < ns ? (size_t)4 : (size_t)f.LS; },
                [&](int t, double v) { (t < ns ? sums[t] : t < ns + nc ? m.sl[t - ns] : m.kb[t - ns - nc]) = v; });
        };
        auto gather_a = [&]() {
            team_vec64(G, k, f.partA, (size_t)f.LA, team, [&](int t, double v) { m.ka[t] = v; });
        };
        gather_s(-1);
        double xxs = sums[0];
        if (xxs == 0.0) {
            // Zero start column: the residual column of largest norm (lowest index on ties);
            // every column zero => rank exhausted.
            for (int c = tid; c < N; c += T) {
                double t = 0.0;
                for (int r = r0; r < r1; ++r) t = fma(f.R[(size_t)r * ldr + c], f.R[(size_t)r * ldr + c], t);
                pS[c] = t;
            }
            SYNC64();
            double best = 0.0;
            int bi = N;
            for (int c = tid; c < N; c += T) {
                double v = 0.0;
#pragma unroll 8
                for (int q = 0; q < G; ++q) v += __ldcg(f.partS + (size_t)q * f.LS + c);
                if (v > best) {
                    best = v;
                    bi = c;
                }
            }
            for (int o = 16; o >= 1; o >>= 1) {
                const double ob = __shfl_xor_sync(kFull, best, o);
                const int oi = __shfl_xor_sync(kFull, bi, o);
                if (ob > best || (ob == best && oi < bi)) {
                    best = ob;
                    bi = oi;
                }
            }
            if (lane == 0) {
                s_best[warp] = best;
                s_bidx[warp] = bi;
            }
            __syncthreads();
            best = 0.0;
            bi = N;
            for (int w = 0; w < kWarps64; ++w)
                if (s_best[w] > best || (s_best[w] == best && s_bidx[w] < bi)) {
                    best = s_best[w];
                    bi = s_bidx[w];
                }
            __syncthreads();
            if (!(best > 0.0)) {
                found = k;
                status = kStDegenerate;
                break;
            }
            SYNC64();  // every CTA has read the norms
            xs = sweep(rg, true, false, 0.0, 0, bi);
            ALIVE64();
            for (int c = tid; c < N; c += T) pS[c] = m.s[c];
            if (tid == 0) sc[0] = xs;
            SYNC64();
            gather_s(-1);
            xxs = sums[0];
        }
        if (gs && k > 0) {
            // the Gram row is the new column of V^T V: how far V is from orthonormal bounds the error
            // of ||v'||^2 - b'^T b' by ||V^T V - I||_F b'^T b' (NaN: cut is NaN, the rows are summed)
            if (warp == 0) {
                double e = 0.0;
                for (int i = lane; i < k; i += 32) {
                    const double d = i < k - 1 ? m.kb[i] : m.kb[i] - 1.0;
                    e = fma(i < k - 1 ? 2.0 * d : d, d, e);
                }
                gram_dev += warp_sum(e);
                const double dev = sqrt(gram_dev);
                cut = dev <= 16.0 * DBL_EPSILON ? 0.25 : 4.0 * DBL_EPSILON / dev;
            }
            // W <- R_k^T V for the deflation of component k-1: W(:, j) -= lambda u (v_{k-1} . v_j),
            // new column R_{k-1}^T v_{k-1} - lambda u |v_{k-1}|^2 with R_{k-1}^T v_{k-1} = u_pre / ||v' - V b'||
            const int km = k - 1;
            for (int e = tid; e < (n1 - n0) * k; e += T) {
                const int n = n0 + e / k, jj = e % k;
                const double un = f.U[(size_t)n * f.ldk + km];
                double* w = f.W + (size_t)n * f.ldk + jj;
                if (jj < km)
                    *w = fma(-lam_prev * un, m.kb[jj], *w);
                else
                    *w = fma(-lam_prev * un, m.kb[km], f.upre[n] * vinv_prev);
            }
            __syncthreads();
            // a = U_(k)^T s0 over the slice
            rows_t64(f.U, f.ldk, n0, n1, k, [&](int n) { return m.sl[n - n0]; }, pA, m.tmp);
            SYNC64();
            gather_a();
        }
        {
            if (tid == 0) scal[0] = 1.0 / xxs;  // keeps the first loading's norm O(1)
            fence_async_proxy();
            __syncthreads();
            rg.issue(f, m, r0, r1, 0);  // R stays as it is until the next start: the sweep's first chunk
            const double xx_inv = scal[0];
            const int nb = buf ^ 1;
            double nq = 0.0;
            if (gs && k > 0) {
                rows_dot64(f.U, f.ldk, n0, n1, k, m.ka, [&](int n, double s) {
                    const double un = (m.sl[n - n0] - s) * xx_inv;
                    f.ut[(size_t)nb * N + n] = un;
                    nq = fma(un, un, nq);
                });
            } else {
                for (int n = n0 + tid; n < n1; n += T) {
                    const double un = m.sl[n - n0] * xx_inv;
                    f.ut[(size_t)nb * N + n] = un;
                    nq = fma(un, un, nq);
                }
            }
            nq = lanes_sum64(nq, gs && k > 0 ? lane_group(k) : 1, red);
            if (tid == 0) sc[2 + nb] = nq;
            buf = nb;
        }
        SYNC64();

        // ------------- power iterations
        double mu = 0.0;
        int j = 0;
        for (;;) {
            for (int c = tid; c < N; c += T) m.u[c] = __ldcg(f.ut + (size_t)buf * N + c);
            const double vs = sweep(rg, false, false, 0.0, 0, 0);
            ALIVE64();
            for (int c = tid; c < N; c += T) pS[c] = m.s[c];
            if (gs && k > 0)  // b' = V_(k)^T v' over this CTA's rows
                rows_t64(f.V, f.ldk, r0, r1, k, [&](int r) { return f.vraw[r]; }, pS + N, m.tmp);
            if (tid == 0) sc[0] = vs;
            SYNC64();
            ++j;
            ++total;
            gather_s(2 + buf);
            const double nvp = sums[0], nu2 = sums[1];
            if (!(nu2 > 0.0)) {
                found = k;
                status = kStDegenerate;
                break;
            }
            const int nbuf = buf ^ 1;
            // lambda from l2 = ||v' - V b'||^2 (GS) or ||v'||^2 (pass scale) and the relative strict
            // test (Sec. 2.2 / 2.3, as the appendix programs).  Warp 0 takes the quotients and
            // roots, a lane each: in every thread they cost 5 us.
            auto decide = [&](double l2) {
                const double q = (lane == 0 ? l2 : 1.0) / (lane == 2 ? l2 : nu2);
                const double r = sqrt(q);  // lane 0: lambda, 1: 1 / ||u'||, 2: 1 / ||v'||
                const double inu = __shfl_sync(kFull, r, 1), il2 = __shfl_sync(kFull, q, 2);
                if (lane < 3) scal[lane] = r;
                if (lane == 0) {
                    scal[3] = nu2 * inu * il2;  // ||u'|| / ||v'||^2: keeps ||ut|| ~ 1
                    int st;
                    if (!(r > thresh)) {
                        st = 2;
                    } else if (f.iters_lock != nullptr) {
                        st = j >= f.iters_lock[k];
                    } else {
                        st = fabs(mu - r) < f.tol * r;
                        if (!st && j >= f.max_iter) st = 3;
                    }
                    s_stop = st;
                }
                __syncwarp();
            };
            // ||v' - V b'||^2 = ||v'||^2 - 2 b'^T b' + b'^T (V^T V) b', so with V orthonormal it is
            // ||v'||^2 - b'^T b', which keeps its digits while b' is small: after the deflation b' is
            // rounding where the earlier components have converged, and otherwise as large as what
            // they are off (b'^T b' / ||v'||^2 of 0.4 with one iteration a component).  The difference is
            // taken up to `cut`: 0.25, or less where V has lost orthonormality, so that the loss
            // (V^T V - I enters with b'^T b') moves lambda by no more than three roundings.  Beyond,
            // the norm is formed from the rows, with the second reduction.
            if (warp == 0) {
                double bb = 0.0;
                if (gs)
                    for (int i = lane; i < k; i += 32) bb = fma(m.kb[i], m.kb[i], bb);
                bb = warp_sum(bb);
                if (!gs || k == 0 || bb <= cut * nvp) decide(nvp - bb);
                else if (lane == 0) s_stop = -1;
                __syncwarp();
            }
            // u_pre = s' - W b' (slice, in place of s')
            if (gs && k > 0)
                rows_dot64(f.W, f.ldk, n0, n1, k, m.kb, [&](int n, double s) { m.sl[n - n0] -= s; });
            __syncthreads();
            const bool rows_norm = s_stop < 0;
            if (gs && k > 0 && (rows_norm || s_stop == 0))  // a' = U^T u_pre (partials)
                rows_t64(f.U, f.ldk, n0, n1, k, [&](int n) { return m.sl[n - n0]; }, pA, m.tmp);
            if (rows_norm) {
                double lp = 0.0;
                rows_dot64(f.V, f.ldk, r0, r1, k, m.kb, [&](int r, double s) {
                    const double vc = f.vraw[r] - s;
                    lp = fma(vc, vc, lp);
                });
                lp = lanes_sum64(lp, lane_group(k), red);
                if (tid == 0) sc[1] = lp;
                SYNC64();
                team_sums64(G, 1, [&](int) { return f.scal + 1; }, [&](int) { return (size_t)4; },
                            [&](int, double v) { sums[0] = v; });
                if (warp == 0) decide(sums[0]);
                __syncthreads();
            }
            const double lam = scal[0];
            inv_nu = scal[1];
            const int stop = s_stop;
            if (stop == 2) {
                found = k;
                status = kStDegenerate;
                break;
            }
            if (stop) {
                if (stop == 3 && status == kStOK) status = kStNotConverged;
                const double vinv = scal[2];
                if (gs && k > 0)
                    rows_dot64(f.V, f.ldk, r0, r1, k, m.kb,
                               [&](int r, double s) { f.V[(size_t)r * f.ldk + k] = (f.vraw[r] - s) * vinv; });
                else
                    for (int r = r0 + tid; r < r1; r += T) f.V[(size_t)r * f.ldk + k] = f.vraw[r] * (gs ? vinv : inv_nu);
                for (int n = n0 + tid; n < n1; n += T) {
                    f.U[(size_t)n * f.ldk + k] = __ldcg(f.ut + (size_t)buf * N + n) * inv_nu;
                    if (gs) f.upre[n] = m.sl[n - n0];
                }
                lam_prev = lam;
                vinv_prev = vinv;
                if (g == 0 && tid == 0) {
                    f.lam[k] = lam;
                    f.iters[k] = j;
                }
                SYNC64();  // every CTA has read the partial sums that the next sweep overwrites
                break;
            }
            if (gs && k > 0) {
                if (!rows_norm) SYNC64();
                gather_a();
            }
            fence_async_proxy();
            __syncthreads();
            rg.issue(f, m, r0, r1, 0);  // the next sweep's first chunk arrives behind the barrier
            mu = lam;
            const double nscale = scal[3];
            double nq2 = 0.0;
            if (!gs || k == 0) {
                for (int n = n0 + tid; n < n1; n += T) {
                    const double un = m.sl[n - n0] * nscale;
                    f.ut[(size_t)nbuf * N + n] = un;
                    nq2 = fma(un, un, nq2);
                }
            } else {
                rows_dot64(f.U, f.ldk, n0, n1, k, m.ka, [&](int n, double s) {
                    const double un = (m.sl[n - n0] - s) * nscale;
                    f.ut[(size_t)nbuf * N + n] = un;
                    nq2 = fma(un, un, nq2);
                });
            }
            nq2 = lanes_sum64(nq2, gs && k > 0 ? lane_group(k) : 1, red);
            if (tid == 0) sc[2 + nbuf] = nq2;
            buf = nbuf;
            SYNC64();
        }
    }
#undef SYNC64
#undef ALIVE64
leave64:
    if (tid == kBlock64 - 32 && rg.issued != 0)  // copies still on their way (after a wait that ran out)
        for (unsigned i = 1; i <= (unsigned)f.nbuf && i <= rg.issued; ++i)
            mbar_wait(&mbar[rg.slot(f, rg.issued - i)], rg.phase(f, rg.issued - i), kSettleNs);
    if (alive && g == 0 && tid == 0) {
        f.info[0] = status;
        f.info[1] = found;
        f.info[2] = (int)(total & 0x7fffffff);
        f.info[3] = (int)(total >> 31);
    }
}

}  // namespace gspca
