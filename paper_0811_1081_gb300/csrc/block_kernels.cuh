// Small dense kernels of the block power iteration (gspca_fit_block): Gram
// matrices with FP64 accumulation, Cholesky factor inverse (CholQR), a
// symmetric eigensolver for b x b matrices, the convergence test, and the
// output scaling.  The large products (R U, R^T V, projections, the rank-b
// deflation) are plain FP32 GEMMs of cuBLAS.  Every sum runs in a fixed order.
#pragma once

#include <cooperative_groups.h>

#include <cfloat>

#include "device_common.cuh"

namespace gspca {

constexpr int kBlkMax = 32;          // widest block
constexpr int kGramRows = 64;        // rows of A and of B per staged chunk of the Gram kernel
constexpr int kGramCtas = 128;       // CTAs of the Gram kernel
constexpr int kGramCluster = 8;      // CTAs whose sums are added in the kernel itself
constexpr int kGramParts = kGramCtas / kGramCluster;
constexpr int kGramThreads = 512;
constexpr int kBlkLd = kBlkMax + 2;  // row stride of staged FP64 rows (16-byte pairs)

// part[p] (n x m, FP64, column-major) = sum over the rows of the 8 CTAs of cluster p of
// A^T B, with A (rows x n, lda) and B (rows x m, ldb) FP32 column-major; n, m <= kBlkMax.
// Rows are staged as FP64 (converted once each); a thread owns a 2 x 2 tile of the product
// (of the upper half when A is B) for every ng-th row, so the FP64 pipe, 2 FMAs per clock and
// SM, is the bound; the thread groups are added in order in shared memory, then the 8 CTAs
// through their cluster's shared memory, so a consumer adds 16 parts itself and no kernel is
// launched for that.  10000 x 16: 37 us + 31 us for the sum of 128 parts with a thread per
// entry that converted its operands for every product; 14 us now, 9 for 2000 x 16.
__global__ void __cluster_dims__(kGramCluster, 1, 1) __launch_bounds__(kGramThreads)
gram_part_kernel(const float* A, int lda, const float* B, int ldb, int rows, int n, int m, double* part) {
    __shared__ __align__(16) double stage[2 * kGramRows * kBlkLd];
    __shared__ double mine[kBlkMax * kBlkMax];
    const int t = threadIdx.x, G = gridDim.x, g = blockIdx.x;
    const int r0 = (int)(((long long)g * rows) / G), r1 = (int)(((long long)(g + 1) * rows) / G);
    const bool sym = A == B && n == m;
    const int tn = (n + 1) / 2, tm = (m + 1) / 2;
    const int ntile = sym ? tn * (tn + 1) / 2 : tn * tm, ng = min(kGramThreads / ntile, kGramRows);
    const int tile = t % ntile, grp = t / ntile;
    int ti, tj;
    if (sym) {
        ti = tile;
        for (tj = 0; ti > tj; ++tj) ti -= tj + 1;
    } else {
        ti = tile % tn;
        tj = tile / tn;
    }
    double* sa = stage;
    double* sb = sym ? stage : stage + kGramRows * kBlkLd;
    const int lg = sym ? 7 : 6, chunk = 1 << lg;  // A alone may use all of it
    static_assert(kGramRows == 64, "lg");
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int rb = r0; rb < r1; rb += chunk) {
        const int nr = min(chunk, r1 - rb);
#pragma unroll 4
        for (int e = t; e < chunk * 2 * tn; e += kGramThreads) {
            const int r = e & (chunk - 1), c = e >> lg;
            sa[r * kBlkLd + c] = (r < nr && c < n) ? (double)A[(size_t)c * lda + rb + r] : 0.0;
        }
        if (!sym)
            for (int e = t; e < kGramRows * 2 * tm; e += kGramThreads) {
                const int r = e % kGramRows, c = e / kGramRows;
                sb[r * kBlkLd + c] = (r < nr && c < m) ? (double)B[(size_t)c * ldb + rb + r] : 0.0;
            }
        __syncthreads();
        if (grp < ng) {
#pragma unroll 2
            for (int r = grp; r < nr; r += ng) {
                const double2 x = *reinterpret_cast<const double2*>(sa + r * kBlkLd + 2 * ti);
                const double2 y = *reinterpret_cast<const double2*>(sb + r * kBlkLd + 2 * tj);
                acc[0] = fma(x.x, y.x, acc[0]);
                acc[1] = fma(x.y, y.x, acc[1]);
                acc[2] = fma(x.x, y.y, acc[2]);
                acc[3] = fma(x.y, y.y, acc[3]);
            }
        }
        __syncthreads();
    }
    // thread groups in order: stage holds kGramThreads x 4 doubles
    static_assert(2 * kGramRows * kBlkLd >= 4 * kGramThreads, "room for the groups");
    if (grp < ng)
#pragma unroll
        for (int q = 0; q < 4; ++q) stage[((size_t)grp * 4 + q) * ntile + tile] = acc[q];
    __syncthreads();
    for (int e = t; e < 4 * ntile; e += kGramThreads) {
        double v[4] = {0.0, 0.0, 0.0, 0.0};  // four chains: an FP64 addition waits long for the one before
        for (int i = 0; i < ng; i += 4)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i + q < ng) v[q] += stage[(size_t)(i + q) * 4 * ntile + e];
        mine[e] = (v[0] + v[1]) + (v[2] + v[3]);
    }
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    cl.sync();
    const int rank = (int)cl.block_rank(), per = (4 * ntile + kGramCluster - 1) / kGramCluster;
    double* out = part + (size_t)(g / kGramCluster) * n * m;
    for (int e = rank * per + t; e < min((rank + 1) * per, 4 * ntile); e += kGramThreads) {
        double x[kGramCluster];
#pragma unroll
        for (int c = 0; c < kGramCluster; ++c) x[c] = cl.map_shared_rank(mine, c)[e];
        const double v = ((x[0] + x[1]) + (x[2] + x[3])) + ((x[4] + x[5]) + (x[6] + x[7]));
        const int q = e / ntile;
        int i = e % ntile, j;
        if (sym) {
            for (j = 0; i > j; ++j) i -= j + 1;
        } else {
            j = i / tn;
            i = i % tn;
        }
        i = 2 * i + (q & 1);
        j = 2 * j + (q >> 1);
        if (i < n && j < m) {
            out[(size_t)j * n + i] = v;
            if (sym) out[(size_t)i * n + j] = v;
        }
    }
    cl.sync();  // the others read this CTA's sums
}

// out(i, j, sum of the kGramParts parts (n x m each)), in a fixed order; the whole CTA.
template <class Out>
__device__ __forceinline__ void sum_parts(const double* part, int n, int m, Out out) {
    for (int e = threadIdx.x; e < n * m; e += blockDim.x) {
        double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int p = 0; p < kGramParts; ++p) v[p & 3] += __ldg(part + (size_t)p * n * m + e);
        out(e % n, e / n, (v[0] + v[1]) + (v[2] + v[3]));
    }
}

// Cholesky G = S^T S (S upper triangular, positive diagonal) of the n x n FP64 Gram matrix
// (given as parts), and Sinv = S^{-1} written as FP32 (n x n column-major, zero below the
// diagonal).  One CTA of four warps.  *flag |= 1 when a pivot is not above 1e-12 of the
// largest diagonal entry of G (numerically dependent columns); Sinv is then the identity.
// Elimination on [G | I] gives S^{-T} beside S in the same n steps: at step k columns j > k hold
// the trailing matrix and columns j <= k the inverse, so one array serves both.  A lane owns a
// column, a warp every fourth row; what bounds it is the chain of n inverse roots, one
// barrier each (37 us for n = 16 with three barriers a step and a second chain of n^2 / 2
// terms for the inverse; 16 us now, with the sum of the parts).
__global__ void __launch_bounds__(128) chol_inv_kernel(const double* part, int n, float* Sinv, int* flag) {
    __shared__ double a[kBlkMax][kBlkMax + 1];
    __shared__ double row[2][kBlkMax];
    __shared__ int bad;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    sum_parts(part, n, n, [&](int i, int j, double v) { a[i][j] = v; });
    if (t == 0) bad = 0;
    __syncthreads();
    double dmax = lane < n ? a[lane][lane] : 0.0;
    for (int o = 16; o >= 1; o >>= 1) dmax = fmax(dmax, __shfl_xor_sync(kFull, dmax, o));
    dmax = fmax(dmax, 0.0);
    // G is scaled by an even power of two (exact) that brings its diagonal into FP32's range, so
    // an inverse root is its FP32 value and one third-order step in FP64
    const int sh = dmax > 0.0 && dmax <= DBL_MAX ? ilogb(dmax) / 2 : 0;
    const double down = scalbn(1.0, -2 * sh), back = scalbn(1.0, -sh);
    dmax *= down;
    double r[kBlkMax / 4];
#pragma unroll
    for (int q = 0; q < kBlkMax / 4; ++q) {
        const int i = warp + 4 * q;
        r[q] = i < n && lane < n ? a[i][lane] * down : 0.0;
    }
#pragma unroll
    for (int kq = 0; kq < kBlkMax / 4; ++kq)
        for (int kw = 0; kw < 4; ++kw) {
            const int k = 4 * kq + kw;
            if (k >= n) break;
            double* rk = row[k & 1];
            if (warp == kw) {
                const double p = __shfl_sync(kFull, r[kq], k);
                if (!(p > 1e-12 * dmax) && lane == 0) bad = 1;
                const double y = (double)rsqrtf((float)p), e = fma(-p * y, y, 1.0);
                const double rs = fma(y, fma(0.375, e, 0.5) * e, y);
                r[kq] = lane == k ? rs : r[kq] * rs;
                rk[lane] = r[kq];
            }
            __syncthreads();
            const double x = rk[lane];
#pragma unroll
            for (int q = kq; q < kBlkMax / 4; ++q) {
                const int i = warp + 4 * q;
                if (i > k && i < n) r[q] = fma(-rk[i], x, lane == k ? 0.0 : r[q]);
            }
        }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kBlkMax / 4; ++q) {
        const int i = warp + 4 * q;
        if (i < n && lane < n)
            Sinv[(size_t)i * n + lane] = bad ? (i == lane ? 1.f : 0.f) : (lane <= i ? (float)(r[q] * back) : 0.f);
    }
    if (t == 0 && bad) atomicOr(flag, 1);
}

constexpr int kJacobiThreads = 512;

// Work of the eigensolver: two copies of the matrix (a step reads one and writes the other),
// the vectors, a step's pairs and rotations.
struct JacobiMem {
    double A[2][kBlkMax][kBlkMax + 1];
    double W[kBlkMax][kBlkMax + 1];
    double2 cs[kBlkMax / 2];
    int2 pq[kBlkMax / 2];
    double red[2][kJacobiThreads / 32];
    double ev[kBlkMax];
    int rank[kBlkMax];
};

// Symmetric eigen-decomposition of the n x n FP64 matrix m.A[0] (zero outside n x n) by
// the cyclic Jacobi method with the parallel (round-robin) pair ordering of
// Golub & Van Loan Sec. 8.5: every step rotates n/2 disjoint pairs at once.
// Sweeps until the off-diagonal norm is at most 1e-15 ||G||_F (at most 40).
// m.ev: eigenvalues, m.rank: their places in decreasing order (lowest index on ties); with
// `vectors` the unit vectors are the columns of m.W.  One CTA.
// A step is a chain of two barriers, the rotation and its use, so the rotation is kept short:
// the tangent comes from FP32 (its error leaves 1e-7 of an entry, removed with what the next
// sweep removes anyway), the cosine from it in FP64, so rotations are orthogonal to FP64 (n = 8,
// 11, 16, 24 matrices of each of three spectra against 40 digits: the errors of eigenvalues and
// vectors are those of FP64 tangents to 0.9 to 1.2 in the mean, with as many sweeps).  A
// thread takes a column of a 2 x 2 block through both sides at once, from one copy of the
// matrix into the other.  n = 16: 142 us; 445 with four barriers a step, FP64 quotients and
// roots, and the norms and the order found by one thread.
__device__ __forceinline__ void jacobi_eig(JacobiMem& m, int n, bool vectors) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int n2 = (n + 1) / 2 * 2, np = n2 / 2;  // an odd n plays with a dummy index n
    int cur = 0;
    if (vectors)
        for (int e = t; e < kBlkMax * kBlkMax; e += kJacobiThreads)
            m.W[e % kBlkMax][e / kBlkMax] = e % kBlkMax == e / kBlkMax ? 1.0 : 0.0;
    // an exact power of two brings the largest diagonal entry near 1, within FP32's range
    __syncthreads();
    double top = lane < n ? fabs(m.A[0][lane][lane]) : 0.0;
    for (int o = 16; o >= 1; o >>= 1) top = fmax(top, __shfl_xor_sync(kFull, top, o));
    const int sh = top > 0.0 && top <= DBL_MAX ? ilogb(top) : 0;
    __syncthreads();
    for (int e = t; e < kBlkMax * kBlkMax; e += kJacobiThreads) {
        double& x = m.A[0][e / kBlkMax][e % kBlkMax];
        x = scalbn(x, -sh);
    }
    __syncthreads();
    for (int sweep = 0; sweep < 40; ++sweep) {
        double o = 0.0, d = 0.0;
        for (int e = t; e < n * n; e += kJacobiThreads) {
            const int i = e % n, j = e / n;
            const double x = m.A[cur][i][j];
            if (i == j) d = fma(x, x, d);
            else o = fma(x, x, o);
        }
        o = warp_sum(o);
        d = warp_sum(d);
        if (lane == 0) {
            m.red[0][warp] = o;
            m.red[1][warp] = d;
        }
        __syncthreads();
        o = warp_sum(lane < kJacobiThreads / 32 ? m.red[0][lane] : 0.0);
        d = warp_sum(lane < kJacobiThreads / 32 ? m.red[1][lane] : 0.0);
        if (!(o > 1e-30 * (o + d))) break;  // the same in every warp
        for (int step = 0; step < n2 - 1; ++step) {
            // pairs (c(q), c(n2 - 1 - q)) of the circle c(0) = 0, c(i) = 1 + (i - 1 - step) mod
            // (n2 - 1): over n2 - 1 steps every pair meets once
            if (t < np) {
                int i1 = n2 - 2 - t - step;
                if (i1 < 0) i1 += n2 - 1;
                int p = 0, q = 1 + i1;
                if (t > 0) {
                    p = t - 1 - step;
                    if (p < 0) p += n2 - 1;
                    ++p;
                }
                if (p > q) {
                    const int s = p;
                    p = q;
                    q = s;
                }
                const float h = (float)(2.0 * m.A[cur][p][q]), f = (float)(m.A[cur][q][q] - m.A[cur][p][p]);
                const float big = fmaxf(fabsf(h), fabsf(f));
                double c = 1.0, s = 0.0;
                if (fabsf(h) >= FLT_MIN) {
                    const float hs = h / big, fs = f / big;
                    const float tt = (fs > 0.f ? hs : fs < 0.f ? -hs : fabsf(hs)) / (fabsf(fs) + sqrtf(fs * fs + hs * hs));
                    // 1 / sqrt(1 + tt^2): the FP32 value and one third-order step
                    const double td = (double)tt, x = fma(td, td, 1.0);
                    const double y = (double)rsqrtf(fmaf(tt, tt, 1.f));
                    const double e = fma(-x * y, y, 1.0);
                    c = fma(y, fma(0.375, e, 0.5) * e, y);
                    s = td * c;
                }
                m.pq[t] = make_int2(p, q);
                m.cs[t] = make_double2(c, s);
            }
            __syncthreads();
            // A <- J^T A J: a thread per block (a, b) and column of it
            for (int e = t; e < np * np * 2; e += kJacobiThreads) {
                const int b = e % np, a = (e / np) % np;
                const bool second = e >= np * np;
                const int2 ra = m.pq[a], rb = m.pq[b];
                const double2 ca = m.cs[a], cb = m.cs[b];
                const double k1 = second ? cb.y : cb.x, k2 = second ? cb.x : -cb.y;
                const double y0 = fma(k1, m.A[cur][ra.x][rb.x], k2 * m.A[cur][ra.x][rb.y]);
                const double y1 = fma(k1, m.A[cur][ra.y][rb.x], k2 * m.A[cur][ra.y][rb.y]);
                const int j = second ? rb.y : rb.x;
                m.A[cur ^ 1][ra.x][j] = fma(ca.x, y0, -ca.y * y1);
                m.A[cur ^ 1][ra.y][j] = fma(ca.y, y0, ca.x * y1);
            }
            if (vectors)  // W <- W J: a thread per pair and row
                for (int e = t; e < np * n; e += kJacobiThreads) {
                    const int b = e % np, i = e / np;
                    const int2 rb = m.pq[b];
                    const double2 cb = m.cs[b];
                    if (rb.y < n) {
                        const double x = m.W[i][rb.x], y = m.W[i][rb.y];
                        m.W[i][rb.x] = fma(cb.x, x, -cb.y * y);
                        m.W[i][rb.y] = fma(cb.y, x, cb.x * y);
                    }
                }
            cur ^= 1;
            __syncthreads();
        }
    }
    if (t < n) m.ev[t] = scalbn(m.A[cur][t][t], sh);
    __syncthreads();
    if (t < n) {
        int r = 0;
        for (int j = 0; j < n; ++j) r += m.ev[j] > m.ev[t] || (m.ev[j] == m.ev[t] && j < t);
        m.rank[t] = r;
    }
    __syncthreads();
}

// Ritz values s_i = sqrt(max(ev_i, 0)) of the Gram matrix Z^T Z (given as parts), in
// decreasing order; the block stops when every |s_i - sp_i| < tol s_i; then sp <- s.  The
// host reads *host = *flag | 2 (stop) and *change = the largest |s_i - sp_i| / s_i in FP32, by which
// it guesses the next test; *flag is cleared for the iteration after the next.  One CTA.
__global__ void __launch_bounds__(kJacobiThreads) ritz_test_kernel(const double* part, double* sp, int n, double tol,
                                                                   int* flag, volatile int* host,
                                                                   volatile float* change) {
    __shared__ JacobiMem m;
    const int t = threadIdx.x;
    for (int e = t; e < kBlkMax * (kBlkMax + 1); e += kJacobiThreads) (&m.A[0][0][0])[e] = 0.0;
    __syncthreads();
    sum_parts(part, n, n, [&](int i, int j, double v) { m.A[0][i][j] = v; });
    __syncthreads();
    jacobi_eig(m, n, false);
    bool same = true;
    float rel = 0.f;
    if (t < n) {
        const double ev = m.ev[t], s = sqrt(ev > 0.0 ? ev : 0.0), d = fabs(sp[m.rank[t]] - s);
        same = d < tol * s;
        rel = (float)d / (float)s;
        sp[m.rank[t]] = s;
    }
    static_assert(kBlkMax == 32, "a warp holds the values");
    for (int o = 16; o >= 1; o >>= 1) rel = fmaxf(rel, __shfl_xor_sync(kFull, rel, o));
    const int stop = __syncthreads_and(same);
    if (t == 0) {
        *change = rel;
        *host = *flag | (stop ? 2 : 0);
        *flag = 0;
    }
}

// Rayleigh-Ritz rotations from B = Z^T U (n x n, FP64, given as parts) and the eigenpairs
// (ev, w) of B^T B: sigma_i = sqrt(ev_i), also into lambda; Zh (FP32) = the eigenvectors; Yh
// (FP32) = B Zh / sigma.  The host reads *host = 1 when a sigma is zero.  One CTA.
__global__ void __launch_bounds__(kJacobiThreads) ritz_rot_kernel(const double* part, int n, double* sigma,
                                                                  double* lambda, float* Yh, float* Zh, volatile int* host) {
    __shared__ JacobiMem m;
    __shared__ double B[kBlkMax][kBlkMax + 1];
    const int t = threadIdx.x;
    for (int e = t; e < kBlkMax * (kBlkMax + 1); e += kJacobiThreads) (&m.A[0][0][0])[e] = 0.0;
    sum_parts(part, n, n, [&](int i, int j, double v) { B[i][j] = v; });
    __syncthreads();
    for (int e = t; e < n * n; e += kJacobiThreads) {
        const int i = e % n, j = e / n;
        double s = 0.0;
        for (int l = 0; l < n; ++l) s = fma(B[l][i], B[l][j], s);
        m.A[0][i][j] = s;
    }
    __syncthreads();
    jacobi_eig(m, n, true);
    bool zero = false;
    if (t < n) {
        const double ev = m.ev[t], s = sqrt(ev > 0.0 ? ev : 0.0);
        sigma[m.rank[t]] = s;
        lambda[m.rank[t]] = s;
        zero = !(s > 0.0);
    }
    for (int e = t; e < n * n; e += kJacobiThreads) {
        const int i = e % n, c = e / n, j = m.rank[c];
        const double sj = sqrt(m.ev[c] > 0.0 ? m.ev[c] : 0.0);
        double s = 0.0;
        for (int l = 0; l < n; ++l) s = fma(B[i][l], m.W[l][c], s);
        Yh[(size_t)j * n + i] = sj > 0.0 ? (float)(s / sj) : 0.f;
        Zh[(size_t)j * n + i] = (float)m.W[i][c];
    }
    const int any = __syncthreads_or(zero);
    if (t == 0) *host = any ? 1 : 0;
}

// out[0 .. n) = v (iterations of a block's components).
__global__ void fill_int_kernel(int* out, int n, int v) {
    if ((int)threadIdx.x < n) out[threadIdx.x] = v;
}

// D (rows x n, ld) = S (rows x n, lds) with column j scaled by sigma[j].
__global__ void scale_cols_kernel(const float* S, int lds, float* D, int ld, int rows, int n, const double* sigma) {
    const size_t total = (size_t)rows * n, stride = (size_t)gridDim.x * blockDim.x;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += stride) {
        const int r = (int)(e % rows), j = (int)(e / rows);
        D[(size_t)j * ld + r] = (float)((double)S[(size_t)j * lds + r] * sigma[j]);
    }
}

// R (M x N, ld M, column-major FP32) <- X with optional centring (1: column
// means, 2: row means, both FP64), ||R||_F^2 not needed here.
__global__ void pack_colmajor_kernel(const float* X, int layout, long ldx, int M, int N, int center,
                                     const double* cmean, const double* rmean, float* R) {
    const size_t total = (size_t)M * N, stride = (size_t)gridDim.x * blockDim.x;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += stride) {
        int r, c;
        if (layout == 0) {
            r = (int)(e % M);
            c = (int)(e / M);
        } else {
            r = (int)(e / N);
            c = (int)(e % N);
        }
        float v = layout == 0 ? X[(size_t)c * ldx + r] : X[(size_t)r * ldx + c];
        if (center == 1) v = (float)((double)v - cmean[c]);
        else if (center == 2) v = (float)((double)v - rmean[r]);
        R[(size_t)c * M + r] = v;
    }
}

}  // namespace gspca
