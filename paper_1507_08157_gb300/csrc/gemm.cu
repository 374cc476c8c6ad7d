// Dense row-major GEMM on CUDA cores (float32 / float64), batched with strides.
//
// C[b] = alpha * op(A[b]) * op(B[b]) + beta * C[b], op = identity or transpose.
// 64, 32 or 16 wide output tile per 256-thread block, 16-deep K slices staged in shared memory; thread
// (tx, ty) owns rows ty + 16u and columns tx + 16v, so shared-memory reads are broadcasts (A) or
// conflict-free (B) and the C stores are coalesced along tx.
#include "tddft_internal.h"

#include <cstdlib>

namespace tddft {

void tc_gemm(cudaStream_t st, bool ta, bool tb, int M, int N, int K, float alpha, const float *A, int lda,
             long long sA, const float *B, int ldb, long long sB, float beta, float *C, int ldc, long long sC,
             int batch, bool split);
bool tc_gemm_available();

bool tc_enabled() {
    static const bool on = []() {
        const char *e = std::getenv("TDDFT_NO_TC");
        return !(e && e[0] == '1') && tc_gemm_available();
    }();
    return on;
}

namespace {

constexpr int BK = 16;

// Output tile B x B, 256 threads as 16 x 16, each with (B / 16)^2 outputs. The next K slice is loaded
// into registers while this one is multiplied. Every output adds its products in order of K, whatever
// the tile.
template <typename T, bool TA, bool TB, int B>
__global__ void __launch_bounds__(256) gemm_kernel(int M, int N, int K, T alpha,
                                                   const T *__restrict__ A, int lda, long long sA,
                                                   const T *__restrict__ Bm, int ldb, long long sB,
                                                   T beta, T *__restrict__ C, int ldc,
                                                   long long sC) {
    constexpr int R = B / 16;
    __shared__ T As[BK][B + 1];
    __shared__ T Bs[BK][B + 1];
    const int b = blockIdx.z;
    A += (long long)b * sA;
    Bm += (long long)b * sB;
    C += (long long)b * sC;
    const int m0 = blockIdx.y * B, n0 = blockIdx.x * B;
    const int t = threadIdx.x;
    const int tx = t & 15, ty = t >> 4;
    T acc[R][R];
#pragma unroll
    for (int u = 0; u < R; ++u)
#pragma unroll
        for (int v = 0; v < R; ++v) acc[u][v] = T(0);

    // element i of a thread's share of a slice: consecutive threads along the operand's rows
    auto a_at = [&](int i, int &m, int &kk) {
        if (!TA) { kk = t & 15; m = (t >> 4) + 16 * i; }
        else { const int e = t + 256 * i; m = e % B; kk = e / B; }
    };
    auto b_at = [&](int i, int &n, int &kk) {
        if (TB) { kk = t & 15; n = (t >> 4) + 16 * i; }
        else { const int e = t + 256 * i; n = e % B; kk = e / B; }
    };
    T ra[R], rb[R];
    auto load = [&](int k0) {
#pragma unroll
        for (int i = 0; i < R; ++i) {
            int m, n, kk;
            a_at(i, m, kk);
            int g = m0 + m, gk = k0 + kk;
            ra[i] = (g < M && gk < K) ? (TA ? A[(long long)gk * lda + g] : A[(long long)g * lda + gk]) : T(0);
            b_at(i, n, kk);
            g = n0 + n, gk = k0 + kk;
            rb[i] = (g < N && gk < K) ? (TB ? Bm[(long long)g * ldb + gk] : Bm[(long long)gk * ldb + g]) : T(0);
        }
    };
    load(0);
    for (int k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
        for (int i = 0; i < R; ++i) {
            int m, n, kk;
            a_at(i, m, kk);
            As[kk][m] = ra[i];
            b_at(i, n, kk);
            Bs[kk][n] = rb[i];
        }
        __syncthreads();
        if (k0 + BK < K) load(k0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            T a[R], bb[R];
#pragma unroll
            for (int u = 0; u < R; ++u) a[u] = As[kk][ty + 16 * u];
#pragma unroll
            for (int v = 0; v < R; ++v) bb[v] = Bs[kk][tx + 16 * v];
#pragma unroll
            for (int u = 0; u < R; ++u)
#pragma unroll
                for (int v = 0; v < R; ++v) acc[u][v] = fma(a[u], bb[v], acc[u][v]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int gm = m0 + ty + 16 * u;
        if (gm >= M) continue;
#pragma unroll
        for (int v = 0; v < R; ++v) {
            const int gn = n0 + tx + 16 * v;
            if (gn >= N) continue;
            T *c = &C[(long long)gm * ldc + gn];
            *c = (beta == T(0)) ? alpha * acc[u][v] : fma(alpha, acc[u][v], beta * *c);
        }
    }
}

template <typename T, bool TA, bool TB, int B>
void launch_tile(cudaStream_t st, int M, int N, int K, T alpha, const T *A, int lda, long long sA,
                 const T *Bm, int ldb, long long sB, T beta, T *C, int ldc, long long sC, int batch) {
    dim3 grid((N + B - 1) / B, (M + B - 1) / B, batch);
    gemm_kernel<T, TA, TB, B><<<grid, 256, 0, st>>>(M, N, K, alpha, A, lda, sA, Bm, ldb, sB, beta, C, ldc, sC);
    check_launch("gemm_kernel");
}

// The tile by the outputs that the busiest SM computes, padding included: a product of few or ragged
// 64-wide tiles leaves most of the 152 SMs idle, and float64 is bound by its rate per SM (32 x 32 x 32,
// batch 2: 39 us in 64-wide tiles, 6 us in 16-wide ones). Of equal ones the largest, which
// reads the operands least; sizes past the y or z grid limits of the smaller tiles keep 64.
template <typename T, bool TA, bool TB>
void launch(cudaStream_t st, int M, int N, int K, T alpha, const T *A, int lda, long long sA,
            const T *Bm, int ldb, long long sB, T beta, T *C, int ldc, long long sC, int batch) {
    auto cost = [&](int B) {
        const long long tiles = (long long)((N + B - 1) / B) * ((M + B - 1) / B) * batch;
        return (tiles + 151) / 152 * B * B;
    };
    const bool small_ok = (M + 15) / 16 <= 65535;
    if (small_ok && cost(16) < cost(32) && cost(16) < cost(64))
        launch_tile<T, TA, TB, 16>(st, M, N, K, alpha, A, lda, sA, Bm, ldb, sB, beta, C, ldc, sC, batch);
    else if (small_ok && cost(32) < cost(64))
        launch_tile<T, TA, TB, 32>(st, M, N, K, alpha, A, lda, sA, Bm, ldb, sB, beta, C, ldc, sC, batch);
    else
        launch_tile<T, TA, TB, 64>(st, M, N, K, alpha, A, lda, sA, Bm, ldb, sB, beta, C, ldc, sC, batch);
}

}  // namespace

template <typename T>
void gemm(cudaStream_t st, bool ta, bool tb, int M, int N, int K, T alpha, const T *A, int lda,
          long long sA, const T *B, int ldb, long long sB, T beta, T *C, int ldc, long long sC,
          int batch, bool approx) {
    if (M <= 0 || N <= 0 || batch <= 0) return;
    const double bytes = sizeof(T) * ((double)M * K * (sA ? batch : 1) + (double)K * N * (sB ? batch : 1) +
                                      (double)M * N * batch * (beta == T(0) ? 1 : 2));
    ProfScope ps(st, ST_GEMM, 2.0 * M * N * K * batch, bytes);
    // float32 products of useful size go to the tensor cores (three-term TF32 split: float32
    // accuracy); float64 and tiny products stay on the CUDA cores
    if (sizeof(T) == 4 && tc_enabled() && (double)M * N * K * batch >= 2.0e6) {
        tc_gemm(st, ta, tb, M, N, K, (float)alpha, (const float *)A, lda, sA, (const float *)B, ldb, sB,
                (float)beta, (float *)C, ldc, sC, batch, !approx);
        return;
    }
    if (!ta && !tb) launch<T, false, false>(st, M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch);
    else if (!ta && tb) launch<T, false, true>(st, M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch);
    else if (ta && !tb) launch<T, true, false>(st, M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch);
    else launch<T, true, true>(st, M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch);
}

template void gemm<float>(cudaStream_t, bool, bool, int, int, int, float, const float *, int,
                          long long, const float *, int, long long, float, float *, int,
                          long long, int, bool);
template void gemm<double>(cudaStream_t, bool, bool, int, int, int, double, const double *, int,
                           long long, const double *, int, long long, double, double *, int,
                           long long, int, bool);

}  // namespace tddft
