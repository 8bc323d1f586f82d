// grass_fim_apply for many right-hand sides: the substitution block column by block column, all right-hand sides at a time.
//
// Two launches per 64 columns and direction, a product with the diagonal block's stored inverse and a C -= A B update
// on 64 x 64 tiles (plain fp32 multiply-adds, 4 x 4 per thread).  What bounds it: 31 us of dependent launches per block
// column, then the multiply-adds (26 TFLOP/s).  The cluster kernel of grass_fim.cu has no such chain, but reads the whole
// factor for every 32 right-hand sides at most and does 11-15 TFLOP/s; grass_fim_apply says where the line lies.
//   k = 4,096: 256 rows 926 us there, 2,141 here; 600 rows 3,274 and 2,619; 16,384 rows 46.1 ms and 23.2.
//   k = 64, 16,384 rows: 43 and 25 us.
#include "grass_common.cuh"

namespace grass {
namespace fim {

constexpr int NB = 64;

// Rows of C (rows x jb, at the block's column offset) solved against the diagonal block through its stored
// inverse (grass_fim.cu leaves it above the block's diagonal):  forward  x Ljj^T = c  ->  x = c (Ljj^-1)^T,   backward  x Ljj = c  ->
// x = c Ljj^-1.  64 rows per CTA, a 4 x 4 register tile of the product per thread.
template <bool BACKWARD>
__global__ void __launch_bounds__(256)
trsm_rows_kernel(const float* __restrict__ Ljj, int64_t ld_l, int jb, float* __restrict__ C, int64_t ld_c, int64_t rows)
{
    __shared__ __align__(16) float w[NB][NB + 4];    // w[p][q]: x[q] = sum_p c[p] * w[p][q]
    __shared__ __align__(16) float ct[NB][NB + 4];   // ct[p][r] = c[r][p]
    const int tid = threadIdx.x;
    const int64_t r0 = (int64_t)blockIdx.x * NB;
    float lraw[NB * NB / 256], craw[NB * NB / 256];
#pragma unroll
    for (int u = 0; u < NB * NB / 256; ++u) {        // all global loads first: they are independent
        const int e = tid + u * 256, i = e / NB, j = e % NB;
        lraw[u] = (i < jb && j < jb) ? Ljj[(int64_t)i * ld_l + j] : 0.0f;
        craw[u] = (j < jb && r0 + i < rows) ? C[(r0 + i) * ld_c + j] : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < NB * NB / 256; ++u) {
        const int e = tid + u * 256, i = e / NB, j = e % NB;   // consecutive threads: consecutive columns
        float v = 0.0f;
        if (i < jb && j < jb) v = (i == j) ? 1.0f / lraw[u] : lraw[u];   // j > i: inverse entry (j, i); j < i: unused
        // inverse entry (row a, col b), a >= b, is stored at block position [b][a]
        if (!BACKWARD) { w[i][j] = (j >= i) ? v : 0.0f; }                        // w[p][q] = inv[q][p], p <= q
        else           { if (j >= i) w[j][i] = v; if (j > i) w[i][j] = 0.0f; }   // w[p][q] = inv[p][q], p >= q
        ct[j][i] = craw[u];
    }
    __syncthreads();
    const int ty = tid / 16, tx = tid % 16;          // rows ty*4.., outputs tx*4..
    float acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = 0.0f;
#pragma unroll 8
    for (int p = 0; p < NB; ++p) {
        const float4 c4 = *reinterpret_cast<const float4*>(&ct[p][ty * 4]);
        const float4 w4 = *reinterpret_cast<const float4*>(&w[p][tx * 4]);
        const float c[4] = {c4.x, c4.y, c4.z, c4.w}, ww[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(c[u], ww[v], acc[u][v]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int64_t r = r0 + ty * 4 + u;
        if (r >= rows) continue;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int q = tx * 4 + v;
            if (q < jb) C[r * ld_c + q] = acc[u][v];
        }
    }
}

// C[i][j] -= sum_{q<K} A[i][q] * B(j, q), 64 x 64 tile per CTA, 4 x 4 per thread, K <= 64.
//   B_TRANS = false: B(j, q) = Bm[j * ldb + q]  (C -= A B^T);  true: B(j, q) = Bm[q * ldb + j]  (C -= A B).
template <bool B_TRANS>
__global__ void __launch_bounds__(256)
gemm_sub_kernel(float* __restrict__ C, int64_t ldc, int64_t rows, int64_t cols, const float* __restrict__ A, int64_t lda,
                const float* __restrict__ Bm, int64_t ldb, int K)
{
    __shared__ __align__(16) float as[NB][NB + 4];   // as[q][i]
    __shared__ __align__(16) float bs[NB][NB + 4];   // bs[q][j]
    const int tid = threadIdx.x;
    const int64_t i0 = (int64_t)blockIdx.y * NB, j0 = (int64_t)blockIdx.x * NB;
    {
        float av[NB * NB / 256], bv[NB * NB / 256];
#pragma unroll
        for (int u = 0; u < NB * NB / 256; ++u) {     // all global loads first: they are independent
            const int e = tid + u * 256, hi = e / NB, lo = e % NB;   // consecutive threads: consecutive addresses
            av[u] = (i0 + hi < rows && lo < K) ? A[(i0 + hi) * lda + lo] : 0.0f;
            if (!B_TRANS) bv[u] = (j0 + hi < cols && lo < K) ? Bm[(j0 + hi) * ldb + lo] : 0.0f;
            else bv[u] = (j0 + lo < cols && hi < K) ? Bm[(int64_t)hi * ldb + j0 + lo] : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < NB * NB / 256; ++u) {
            const int e = tid + u * 256, hi = e / NB, lo = e % NB;
            as[lo][hi] = av[u];
            if (!B_TRANS) bs[lo][hi] = bv[u]; else bs[hi][lo] = bv[u];
        }
    }
    __syncthreads();
    const int ty = tid / 16, tx = tid % 16;
    float acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = 0.0f;
    for (int q = 0; q < K; ++q) {
        const float4 a4 = *reinterpret_cast<const float4*>(&as[q][ty * 4]);
        const float4 b4 = *reinterpret_cast<const float4*>(&bs[q][tx * 4]);
        const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(a[u], b[v], acc[u][v]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int64_t i = i0 + ty * 4 + u;
        if (i >= rows) continue;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int64_t j = j0 + tx * 4 + v;
            if (j < cols) C[i * ldc + j] -= acc[u][v];
        }
    }
}

static inline unsigned blocks(int64_t n) { return (unsigned)((n + NB - 1) / NB); }

}  // namespace fim

grass_status launch_apply_blocks(const float* Lf, int64_t k, int64_t ld_f, float* Bm, int64_t M, int64_t ld_b, cudaStream_t st)
{
    using namespace fim;
    // L y = b, block column by block column: solve the diagonal block, then remove its contribution from
    // the columns to the right
    for (int64_t j0 = 0; j0 < k; j0 += NB) {
        const int jb = (int)((k - j0) < NB ? (k - j0) : NB);
        trsm_rows_kernel<false><<<blocks(M), 256, 0, st>>>(Lf + j0 * ld_f + j0, ld_f, jb, Bm + j0, ld_b, M);
        const int64_t rest = k - j0 - jb;
        if (rest > 0)
            gemm_sub_kernel<false><<<dim3(blocks(rest), blocks(M)), 256, 0, st>>>(Bm + j0 + jb, ld_b, M, rest, Bm + j0, ld_b,
                                                                                  Lf + (j0 + jb) * ld_f + j0, ld_f, jb);
    }
    // L^T x = y, from the last block column to the first
    for (int64_t j0 = ((k - 1) / NB) * NB; j0 >= 0; j0 -= NB) {
        const int jb = (int)((k - j0) < NB ? (k - j0) : NB);
        trsm_rows_kernel<true><<<blocks(M), 256, 0, st>>>(Lf + j0 * ld_f + j0, ld_f, jb, Bm + j0, ld_b, M);
        if (j0 > 0)
            gemm_sub_kernel<true><<<dim3(blocks(j0), blocks(M)), 256, 0, st>>>(Bm, ld_b, M, j0, Bm + j0, ld_b, Lf + j0 * ld_f, ld_f, jb);
    }
    return launch_status();
}

}  // namespace grass
