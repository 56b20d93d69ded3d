// gspca_fit_block: block power iteration (components b at a time), the block
// form of the GS-PCA loop of Sec. 2.3 (not in the paper).  Per block of width
// bw, on the caller's stream:
//   U = R^T R(:, k0 .. k0+bw-1); U -= U_(k0) U_(k0)^T U; U = qr(U)
//   repeat: Y = R U; Y -= V_(k0) V_(k0)^T Y; V = qr(Y)
//           Z = R^T V; Z -= U_(k0) U_(k0)^T Z; s = sqrt(eig(Z^T Z)) (Ritz values)
//           stop when every |s_i - s_i'| < tol s_i (or max_iter / the lock); else U = qr(Z)
//   Rayleigh-Ritz on B = Z^T U; R -= V diag(sigma) U^T.
// The large products are FP32 GEMMs of cuBLAS; qr is Cholesky QR applied twice
// with the Gram matrix accumulated in FP64 (block_kernels.cuh).  The residual
// lives column-major in the handle's R buffer; V and U are kept in the caller's
// T and P (unit columns until the block ends).  One host synchronisation per
// iteration reads the stop and degenerate flags, behind the next half step.
#include <cublas_v2.h>
#include <cuda_runtime.h>

#include <cstring>
#include <utility>
#include <vector>

#include "../../include/gspca.h"
#include "block_kernels.cuh"
#include "handle.h"
#include "launch_common.cuh"

using namespace gspca;

namespace {

#define BL_CUBLAS(call)                                                       \
    do {                                                                      \
        if ((call) != CUBLAS_STATUS_SUCCESS) {                                \
            cuda_ok(cudaErrorUnknown);                                        \
            return GSPCA_ERR_CUDA;                                            \
        }                                                                     \
    } while (0)

struct BlockWs {
    float *Y, *V, *Vnext, *Z, *U, *Unext, *tmp, *Sinv, *Yh, *Zh;
    double *part, *partZ, *sp, *sigma;
    int* flag;
    size_t bytes;
};

BlockWs carve_block(void* base, long M, int N, int K) {
    BlockWs w{};
    char* b = static_cast<char*>(base);
    size_t off = 0;
    auto take = [&](size_t bytes) -> void* {
        off = (off + 255) / 256 * 256;
        void* p = b ? b + off : nullptr;
        off += bytes > 0 ? bytes : 1;
        return p;
    };
    const size_t B = kBlkMax;
    w.Y = (float*)take(sizeof(float) * (size_t)M * B);
    w.V = (float*)take(sizeof(float) * (size_t)M * B);
    w.Vnext = (float*)take(sizeof(float) * (size_t)M * B);
    w.Z = (float*)take(sizeof(float) * (size_t)N * B);
    w.U = (float*)take(sizeof(float) * (size_t)N * B);
    w.Unext = (float*)take(sizeof(float) * (size_t)N * B);
    w.tmp = (float*)take(sizeof(float) * (size_t)((size_t)K > B ? (size_t)K : B) * B);
    w.Sinv = (float*)take(sizeof(float) * B * B);
    w.Yh = (float*)take(sizeof(float) * B * B);
    w.Zh = (float*)take(sizeof(float) * B * B);
    w.part = (double*)take(sizeof(double) * kGramParts * B * B);
    w.partZ = (double*)take(sizeof(double) * kGramParts * B * B);
    w.sp = (double*)take(sizeof(double) * B);
    w.sigma = (double*)take(sizeof(double) * B);
    w.flag = (int*)take(sizeof(int) * 4);
    w.bytes = (off + 255) / 256 * 256;
    return w;
}

// Gram matrix A^T B (n x m, FP64) of FP32 column-major A (rows x n), B (rows x m), as
// kGramParts parts.
void gram(cudaStream_t s, const float* A, int lda, const float* B, int ldb, int rows, int n, int m, double* part) {
    gram_part_kernel<<<kGramCtas, kGramThreads, 0, s>>>(A, lda, B, ldb, rows, n, m, part);
}

// Cholesky QR applied twice: Q (rows x n) = A S1^{-1} S2^{-1}, A left unchanged
// (Q and A distinct buffers).  `have`: the parts of A^T A where they are formed already.
gspca_status cholqr2(cublasHandle_t cb, cudaStream_t s, const float* A, float* Q, int rows, int n, const BlockWs& w,
                     const double* have, int* flag, int* launches) {
    const float one = 1.f, zero = 0.f;
    if (!have) {
        gram(s, A, rows, A, rows, rows, n, n, w.part);
        ++*launches;
    }
    chol_inv_kernel<<<1, 128, 0, s>>>(have ? have : w.part, n, w.Sinv, flag);
    BL_CUBLAS(cublasSgemm(cb, CUBLAS_OP_N, CUBLAS_OP_N, rows, n, n, &one, A, rows, w.Sinv, n, &zero, Q, rows));
    gram(s, Q, rows, Q, rows, rows, n, n, w.part);
    chol_inv_kernel<<<1, 128, 0, s>>>(w.part, n, w.Sinv, flag);
    // Q <- Q S2^{-1} in place: an upper-triangular factor on the right (column j uses columns <= j)
    BL_CUBLAS(cublasStrmm(cb, CUBLAS_SIDE_RIGHT, CUBLAS_FILL_MODE_UPPER, CUBLAS_OP_N, CUBLAS_DIAG_NON_UNIT, rows, n,
                          &one, w.Sinv, n, Q, rows, Q, rows));
    *launches += 5;
    return GSPCA_OK;
}

// X (rows x n) -= Q (rows x k) (Q^T X); nothing when k == 0.
gspca_status project_out(cublasHandle_t cb, const float* Q, int rows, int k, float* X, int n, float* tmp) {
    if (k == 0) return GSPCA_OK;
    const float one = 1.f, zero = 0.f, mone = -1.f;
    BL_CUBLAS(cublasSgemm(cb, CUBLAS_OP_T, CUBLAS_OP_N, k, n, rows, &one, Q, rows, X, rows, &zero, tmp, k));
    BL_CUBLAS(cublasSgemm(cb, CUBLAS_OP_N, CUBLAS_OP_N, rows, n, k, &mone, Q, rows, tmp, k, &one, X, rows));
    return GSPCA_OK;
}

}  // namespace

gspca_status gspca::block_release(gspca_handle* h) {
    gspca_status st = GSPCA_OK;
    if (h->blk_base && cudaFree(h->blk_base) != cudaSuccess) st = GSPCA_ERR_CUDA;
    if (h->cublas) cublasDestroy((cublasHandle_t)h->cublas);
    if (h->h_blk) cudaFreeHost(h->h_blk);
    if (h->blk_stream) cudaStreamDestroy(h->blk_stream);
    if (h->blk_gram) cudaEventDestroy(h->blk_gram);
    if (h->blk_test) cudaEventDestroy(h->blk_test);
    h->blk_stream = nullptr;
    h->blk_gram = h->blk_test = nullptr;
    h->blk_base = nullptr;
    h->cublas = nullptr;
    h->h_blk = nullptr;
    return st;
}

extern "C" gspca_status gspca_fit_block(gspca_t h, void* stream, const float* X, gspca_layout layout, long ldx, int M,
                                        int N, int K, int block, double tol, int max_iter, float* T, float* P,
                                        double* lambda, int* iters, float* R_out, const gspca_opts* opts) {
    if (!h || !X || !T || !P || !lambda) return GSPCA_ERR_INVALID_ARG;
    if (h->dtype != GSPCA_F32) return GSPCA_ERR_INVALID_ARG;
    if (M < 1 || N < 1 || K < 1 || K > M || K > N) return GSPCA_ERR_INVALID_ARG;
    if (M > h->max_M || N > h->max_N || K > h->max_K) return GSPCA_ERR_INVALID_ARG;
    if (block < 1 || block > kBlkMax || !(tol > 0.0) || max_iter < 1) return GSPCA_ERR_INVALID_ARG;
    if ((layout == GSPCA_COL_MAJOR && ldx < M) || (layout == GSPCA_ROW_MAJOR && ldx < N) ||
        (layout != GSPCA_COL_MAJOR && layout != GSPCA_ROW_MAJOR))
        return GSPCA_ERR_INVALID_ARG;
    const gspca_status ost = check_opts(opts, K);
    if (ost != GSPCA_OK) return ost;
    if (opts && (opts->warm || opts->gs_passes == 2 || opts->coef_trace)) return GSPCA_ERR_NOT_SUPPORTED;
    GS_CUDA(cudaSetDevice(h->device));
    cudaStream_t s = (cudaStream_t)stream;
    if (!h->blk_base) {
        const BlockWs probe = carve_block(nullptr, h->max_M, (int)h->max_N, h->max_K);
        void* base = nullptr;
        cudaError_t e = cudaMalloc(&base, probe.bytes);
        if (e != cudaSuccess) {
            cuda_ok(e);
            return e == cudaErrorMemoryAllocation ? GSPCA_ERR_OOM : GSPCA_ERR_CUDA;
        }
        h->blk_base = base;
        cublasHandle_t cb = nullptr;
        if (cublasCreate(&cb) != CUBLAS_STATUS_SUCCESS) {
            block_release(h);
            return GSPCA_ERR_CUDA;
        }
        h->cublas = cb;
        int lo = 0, hi = 0;
        if (!cuda_ok(cudaDeviceGetStreamPriorityRange(&lo, &hi)) ||
            !cuda_ok(cudaStreamCreateWithPriority(&h->blk_stream, cudaStreamNonBlocking, hi)) ||
            !cuda_ok(cudaEventCreateWithFlags(&h->blk_gram, cudaEventDisableTiming)) ||
            !cuda_ok(cudaEventCreateWithFlags(&h->blk_test, cudaEventDisableTiming))) {
            block_release(h);
            return GSPCA_ERR_CUDA;
        }
        if (!cuda_ok(cudaMallocHost((void**)&h->h_blk, sizeof(int) * 4))) {
            block_release(h);
            return GSPCA_ERR_CUDA;
        }
    }
    BlockWs w = carve_block(h->blk_base, h->max_M, (int)h->max_N, h->max_K);
    cublasHandle_t cb = (cublasHandle_t)h->cublas;
    BL_CUBLAS(cublasSetStream(cb, s));
    BL_CUBLAS(cublasSetMathMode(cb, CUBLAS_DEFAULT_MATH));  // FP32 products, no TF32
    float* R = h->ws.R;  // the handle's residual buffer, here column-major M x N
    const float one = 1.f, zero = 0.f, mone = -1.f;
    int launches = 0;
    const int center = opts ? opts->center : 0;
    if (center == 1) {
        launches += enqueue_colmean(h->ws, s, X, layout, ldx, M, N);
    } else if (center == 2) {
        rowmean_kernel<<<(M + 7) / 8, 256, 0, s>>>(X, (int)layout, ldx, M, N, h->ws.rmean);
        ++launches;
    }
    pack_colmajor_kernel<<<1024, 256, 0, s>>>(X, (int)layout, ldx, M, N, center, h->ws.cmean, h->ws.rmean, R);
    ++launches;
    GS_CUDA(cudaGetLastError());
    GS_CUDA(cudaEventRecord(h->ev0, s));

    std::vector<long long> blk_iters;
    int status = GSPCA_OK, found = 0;
    long long total = 0;
    bool not_converged = false;
    for (int k0 = 0; k0 < K; k0 += block) {
        const int bw = (K - k0) < block ? (K - k0) : block;
        GS_CUDA(cudaMemsetAsync(w.flag, 0, sizeof(int) * 4, s));
        GS_CUDA(cudaMemsetAsync(w.sp, 0, sizeof(double) * kBlkMax, s));
        // U = R^T R(:, k0 .. k0+bw-1), against U_(k0), orthonormal
        BL_CUBLAS(cublasSgemm(cb, CUBLAS_OP_T, CUBLAS_OP_N, N, bw, M, &one, R, M, R + (size_t)k0 * M, M, &zero, w.Z, N));
        if (project_out(cb, P, N, k0, w.Z, bw, w.tmp) != GSPCA_OK) return GSPCA_ERR_CUDA;
        if (cholqr2(cb, s, w.Z, w.U, N, bw, w, nullptr, w.flag, &launches) != GSPCA_OK) return GSPCA_ERR_CUDA;
        // V = qr(R U), against V_(k0); `flag` takes what the factorisations find
        auto half_step = [&](const float* U, float* V, int* flag) -> gspca_status {
            BL_CUBLAS(cublasSgemm(cb, CUBLAS_OP_N, CUBLAS_OP_N, M, bw, N, &one, R, M, U, N, &zero, w.Y, M));
            if (project_out(cb, T, M, k0, w.Y, bw, w.tmp) != GSPCA_OK) return GSPCA_ERR_CUDA;
            launches += 1 + (k0 > 0 ? 2 : 0);
            return cholqr2(cb, s, w.Y, V, M, bw, w, nullptr, flag, &launches);
        };
        if (half_step(w.U, w.V, w.flag) != GSPCA_OK) return GSPCA_ERR_CUDA;
        int j = 0, fl = 0;
        double change = 1.0, before = 1.0;  // of the Ritz values, in the last test and the one before
        bool last = false;
        for (;;) {
            // Z = R^T V, against U_(k0); Ritz values from Z^T Z
            BL_CUBLAS(cublasSgemm(cb, CUBLAS_OP_T, CUBLAS_OP_N, N, bw, M, &one, R, M, w.V, M, &zero, w.Z, N));
            if (project_out(cb, P, N, k0, w.Z, bw, w.tmp) != GSPCA_OK) return GSPCA_ERR_CUDA;
            gram(s, w.Z, N, w.Z, N, N, bw, bw, w.partZ);
            // The test, one CTA and a long chain, runs on a stream of its own, and the next U = qr(Z) and
            // V = qr(R U) go ahead meanwhile, into second buffers and with the other flag word:
            // 10000 x 2000, two blocks of 16, 6 iterations each, 6.1 ms with the test before them, 4.8 so.
            // They are dropped when the test says stop, and left out where this iteration is the last
            // in any case.
            GS_CUDA(cudaEventRecord(h->blk_gram, s));
            GS_CUDA(cudaStreamWaitEvent(h->blk_stream, h->blk_gram, 0));
            ritz_test_kernel<<<1, kJacobiThreads, 0, h->blk_stream>>>(w.partZ, w.sp, bw, tol, w.flag + (j & 1), h->h_blk,
                                                                    reinterpret_cast<float*>(h->h_blk + 2));
            GS_CUDA(cudaGetLastError());
            GS_CUDA(cudaEventRecord(h->blk_test, h->blk_stream));
            launches += 3 + (k0 > 0 ? 2 : 0);
            ++j;
            ++total;
            last = opts && opts->iters_lock ? j >= opts->iters_lock[k0] : j >= max_iter;
            if (last) break;
            // Where the test is likely to stop the block they wait for it: the first test compares with
            // zero, a change of 1, so it stops a block exactly when tol > 1; later changes shrink
            // about as the one before did (to a tenth where nothing is known).  Only narrow blocks go
            // by that guess: their test is short (a wrong guess costs one) and the half step is not;
            // a wide block's test hides all or most of it, and a wrong guess would cost 0.14 (16) to
            // 0.45 ms (32).  15000 x 7500, two blocks of 1: 3.58 ms with tol 10, 3.24 so, 9.98 and 9.62
            // with 1e-3; 10000 x 2000, blocks of 4, 1e-2: 2.72 and 2.61.
            const bool locked = opts && opts->iters_lock;
            const double guess = j == 1 ? 1.0 : change * change / before;
            const bool ahead = locked || guess >= tol || (j > 1 && bw > 4);
            const auto tested = [&]() -> cudaError_t {
                const cudaError_t e = cudaEventSynchronize(h->blk_test);
                fl = ((volatile int*)h->h_blk)[0];
                before = j == 1 ? 10.0 : change;
                change = ((volatile float*)h->h_blk)[2];
                return e;
            };
            const auto ends = [&] { return (fl & 1) || (!locked && (fl & 2)); };  // dependent columns, or stop
            int* nflag = w.flag + (j & 1);
            if (!ahead) {
                GS_CUDA(tested());
                if (ends()) break;
            }
            if (cholqr2(cb, s, w.Z, w.Unext, N, bw, w, w.partZ, nflag, &launches) != GSPCA_OK) return GSPCA_ERR_CUDA;
            if (half_step(w.Unext, w.Vnext, nflag) != GSPCA_OK) return GSPCA_ERR_CUDA;
            if (ahead) {
                GS_CUDA(tested());
                if (ends()) break;
            }
            std::swap(w.U, w.Unext);
            std::swap(w.V, w.Vnext);
        }
        if (!last && (fl & 1)) {
            status = GSPCA_ERR_DEGENERATE;
            break;
        }
        // Rayleigh-Ritz: B = Z^T U (FP64), B^T B = Zh diag(sigma^2) Zh^T, Yh = B Zh / sigma
        gram(s, w.Z, N, w.U, N, N, bw, bw, w.part);
        ritz_rot_kernel<<<1, kJacobiThreads, 0, s>>>(w.part, bw, w.sigma, lambda + k0, w.Yh, w.Zh, h->h_blk + 1);
        launches += 2;
        if (last) {
            GS_CUDA(cudaEventSynchronize(h->blk_test));
            fl = ((volatile int*)h->h_blk)[0];
            if (fl & 1) {
                status = GSPCA_ERR_DEGENERATE;
                break;
            }
            if (!(opts && opts->iters_lock) && !(fl & 2)) not_converged = true;
        }
        // V <- V Yh (into T's columns), U <- U Zh (into P's columns)
        BL_CUBLAS(cublasSgemm(cb, CUBLAS_OP_N, CUBLAS_OP_N, M, bw, bw, &one, w.V, M, w.Yh, bw, &zero,
                              T + (size_t)k0 * M, M));
        BL_CUBLAS(cublasSgemm(cb, CUBLAS_OP_N, CUBLAS_OP_N, N, bw, bw, &one, w.U, N, w.Zh, bw, &zero,
                              P + (size_t)k0 * N, N));
        // R -= (V diag(sigma)) U^T
        scale_cols_kernel<<<256, 256, 0, s>>>(T + (size_t)k0 * M, M, w.Y, M, M, bw, w.sigma);
        BL_CUBLAS(cublasSgemm(cb, CUBLAS_OP_N, CUBLAS_OP_T, M, N, bw, &mone, w.Y, M, P + (size_t)k0 * N, N, &one, R, M));
        GS_CUDA(cudaStreamSynchronize(s));
        if (((volatile int*)h->h_blk)[1] & 1) {
            status = GSPCA_ERR_DEGENERATE;
            break;
        }
        if (iters) {
            fill_int_kernel<<<1, kBlkMax, 0, s>>>(iters + k0, bw, j);
            ++launches;
        }
        found = k0 + bw;
        blk_iters.push_back(j);
        launches += 2;
    }
    GS_CUDA(cudaEventRecord(h->ev1, s));
    // T = V Lambda (unless the SVD form is asked for); zero past `found`
    if (!(opts && opts->svd_form == 1) && found > 0) {
        scale_cols_kernel<<<256, 256, 0, s>>>(T, M, T, M, M, found, lambda);
        ++launches;
    }
    if (found < K) {
        GS_CUDA(cudaMemsetAsync(T + (size_t)found * M, 0, sizeof(float) * (size_t)M * (K - found), s));
        GS_CUDA(cudaMemsetAsync(P + (size_t)found * N, 0, sizeof(float) * (size_t)N * (K - found), s));
        GS_CUDA(cudaMemsetAsync(lambda + found, 0, sizeof(double) * (K - found), s));
        if (iters) GS_CUDA(cudaMemsetAsync(iters + found, 0, sizeof(int) * (K - found), s));
    }
    if (R_out) GS_CUDA(cudaMemcpyAsync(R_out, R, sizeof(float) * (size_t)M * N, cudaMemcpyDeviceToDevice, s));
    GS_CUDA(cudaStreamSynchronize(s));
    float ms = 0.f;
    GS_CUDA(cudaEventElapsedTime(&ms, h->ev0, h->ev1));
    h->last.kernel_ms = ms;
    h->last.found = found;
    h->last.total_iters = total;
    h->last.kernel_launches = launches;
    h->last.grid_ctas = kGramCtas;
    h->last.team_ctas = 0;
    h->last.block_threads = kGramThreads;
    h->last.batch_pass = 0;
    // algorithmic bytes: per iteration R read twice (R U, R^T V) and the factors of the earlier
    // blocks twice on each side (projections); per block R read and written once (deflation)
    {
        double bytes = 0.0;
        int k0 = 0;
        for (const long long it : blk_iters) {
            bytes += (double)it * (8.0 * M * N + 16.0 * (double)(M + N) * k0) + 8.0 * M * N;
            k0 += block;
        }
        h->last.alg_bytes = bytes;
    }
    if (status == GSPCA_ERR_DEGENERATE) return GSPCA_ERR_DEGENERATE;
    if (not_converged) return GSPCA_WARN_NOT_CONVERGED;
    return GSPCA_OK;
}
