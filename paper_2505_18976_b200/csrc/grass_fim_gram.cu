// grass_fim: F = (1/n) X^T X of compressed gradients (Section 2.1, cache stage step 2) on the tensor cores.
//
// Both operands are the same n x k fp32 matrix, the contraction runs over its rows.  A thread block owns one
// 128 x 128 tile of F on or above the diagonal and a range of samples.  Per step of 32 samples its threads read the
// two 128-column strips with 16-byte loads (consecutive lanes, consecutive columns), split every value into three
// bf16 pieces and store them as they lie: eight consecutive COLUMNS are one 16-byte chunk of an MN-major operand tile
// (128-byte swizzle), so nothing is transposed on the way to the tensor core.  A tile on the diagonal stages one
// strip and uses it as both operands.  Six products per 16 samples (tcgen05.mma, M = N = 128), hi*hi into one
// accumulator, the correction terms into a second (the tensor core truncates after every accumulation).
//
// The thread blocks that share a tile form a cluster: each writes its partial tile, slice by slice, into the owners'
// shared memory (the operand stages, free by then), every owner adds the slices of its rows and stores them and their
// mirror image.  Only when one cluster of eight cannot fill the machine do several clusters share a tile; they add
// into the zeroed matrix.
//
// What bounds it: the six products (12 MMAs of 64 cycles per step and SM) once two thread blocks per SM hide the
// loads and the split of each other.  It still runs at about half that rate: shared memory serves the MMAs' operand
// reads (128 bytes a cycle at M = N = 128) and the split's stores.  Measured against the gathering kernel used before
// (4-byte loads, column by column): n = 4,656, k = 1,024 117 -> 54 us, 46 with its results stored four at a time, n = 16,384, k = 4,096 2,090 -> 1,675 us.
#include "factgrass_common.cuh"

#include <cooperative_groups.h>

#include <algorithm>

namespace cg = cooperative_groups;

namespace grass {
namespace gram {

constexpr int TILE = 128;                     // rows and columns of F per thread block
constexpr int STEP = 32;                      // samples per pipeline step
constexpr int THREADS = 256;
constexpr int NBUF = 2;
constexpr int PIECE = TILE * STEP * 2;        // one bf16 piece of one strip: 8 KB
constexpr int STRIP = 3 * PIECE;
constexpr int STAGE = 2 * STRIP;              // 48 KB
constexpr uint32_t LBO = (STEP / 8) * 1024;   // bytes between blocks of 64 columns
constexpr uint32_t SBO = 1024;                // bytes between groups of 8 samples
constexpr uint32_t ACC_COLS = 2 * TILE;
static_assert(THREADS % TILE == 0, "the rows of a thread stay the same");
constexpr int CHUNKS = TILE / 8;              // 16-byte chunks (8 columns) per sample
constexpr int PER_THREAD = STEP * CHUNKS / THREADS;    // chunks per thread, strip and step (2)
static_assert(PER_THREAD * THREADS == STEP * CHUNKS, "even split");
static_assert(NBUF * STAGE >= TILE * TILE * 4, "the partial slices fit where the operand stages were");

// byte offset of the 16-byte chunk `ch` (columns 8 ch .. 8 ch + 7) of sample `t` in an operand tile: blocks of 64
// columns, groups of 8 samples, 128-byte rows, chunk position xor-ed with the sample's position in its group
__device__ __forceinline__ uint32_t chunk_offset(int t, int ch)
{
    return (uint32_t)(ch >> 3) * LBO + (uint32_t)(t >> 3) * SBO + (uint32_t)(t & 7) * 128u +
           (uint32_t)(((ch & 7) ^ (t & 7)) << 4);
}
// MN-major descriptor, 128-byte swizzle: leading offset between blocks of 64 columns, stride offset between groups
// of 8 samples; 16 samples further on are 2 * SBO bytes further on
__device__ __forceinline__ uint64_t make_desc(uint32_t addr)
{
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)(LBO >> 4) << 16) | ((uint64_t)(SBO >> 4) << 32) | (1ull << 46) |
           (2ull << 61);
}
// where element (row, c) of a slice sits: 16-byte chunks xor-ed with the row, so that the writers (lanes on consecutive rows) and the
// readers of rows (lanes on consecutive chunks) are free of bank conflicts.  The readers of four rows of a column (lanes four rows
// apart) are too at 16 and 32 rows to a slice, meet in pairs at 64 and four at a time at 128; without bits 3 and 4 of the row two,
// four, eight and sixteen at a time.
__device__ __forceinline__ int slice_offset(int row, int c)
{
    return row * TILE + ((((c >> 2) ^ (row & 7) ^ ((row >> 2) & 2) ^ ((row >> 4) & 1)) << 2) | (c & 3));
}

__global__ void __launch_bounds__(THREADS, 2)
gram_kernel(const float* __restrict__ X, int32_t n, int32_t k, int64_t ld, int32_t tiles, int32_t nchunks, int32_t chunk_len, float scale,
            float* __restrict__ F, int64_t ld_f, int vec_ok, int vec_f, int add_out, int nprod)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long bars[NBUF + 1];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;

    cg::cluster_group cluster = cg::this_cluster();
    const int cs = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    // blockIdx.x = (tile on or above the diagonal, row by row) * nchunks + sample chunk
    const int chunk = (int)(blockIdx.x % (unsigned)nchunks);
    int tm = 0, rest = (int)(blockIdx.x / (unsigned)nchunks);
    while (rest >= tiles - tm) { rest -= tiles - tm; ++tm; }
    const int tn = tm + rest;
    const bool diag = tm == tn;
    const int64_t t_begin64 = (int64_t)chunk * chunk_len;
    const int t_begin = (int)(t_begin64 < n ? t_begin64 : n);
    const int t_end = (int)(t_begin64 + chunk_len < n ? t_begin64 + chunk_len : n);

    const uint32_t bar0 = tc::smem_u32(&bars[0]), bar_done = tc::smem_u32(&bars[NBUF]);
    if (tid == 0) {
        for (int i = 0; i < NBUF; ++i) tc::mbar_init(bar0 + 8 * i, 1);
        tc::mbar_init(bar_done, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&tmem_slot)),
                     "r"(ACC_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_d = tmem_slot;

    // chunk q of a thread: columns 8 (tid % 16) .., sample tid / 16 + 16 q of the step
    const int ch = tid % CHUNKS, ts = tid / CHUNKS;
    float xa[PER_THREAD][8], xg[PER_THREAD][8];
    auto load8 = [&](float (&x)[8], int64_t t, int col) {
        if (t < t_end && col + 8 <= k && vec_ok) {
            const float4 u = __ldg(reinterpret_cast<const float4*>(X + t * ld + col));
            const float4 w = __ldg(reinterpret_cast<const float4*>(X + t * ld + col) + 1);
            x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w;
            x[4] = w.x; x[5] = w.y; x[6] = w.z; x[7] = w.w;
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) x[e] = (t < t_end && col + e < k) ? __ldg(X + t * ld + col + e) : 0.0f;
        }
    };
    auto prefetch = [&](int t0) {
#pragma unroll
        for (int q = 0; q < PER_THREAD; ++q) {
            const int64_t t = (int64_t)t0 + ts + q * (THREADS / CHUNKS);
            load8(xa[q], t, tm * TILE + ch * 8);
            if (!diag) load8(xg[q], t, tn * TILE + ch * 8);
        }
    };
    auto put = [&](unsigned char* strip, int q, const float (&x)[8]) {
        uint4 hi, mid, lo;
        tc::split8(x, hi, mid, lo);
        const uint32_t off = chunk_offset(ts + q * (THREADS / CHUNKS), ch);
        *reinterpret_cast<uint4*>(strip + off) = hi;
        *reinterpret_cast<uint4*>(strip + PIECE + off) = mid;
        *reinterpret_cast<uint4*>(strip + 2 * PIECE + off) = lo;
    };

    const uint64_t desc0 = make_desc(tc::smem_u32(smem));      // addresses below are 16-byte units added to it
    // as make_idesc, both operands MN-major
    const uint32_t idesc = tc::make_idesc(TILE, TILE) | (1u << 15) | (1u << 16);
    bool ok = true;
    if (t_begin < t_end) prefetch(t_begin);
    int it = 0;
    for (int t0 = t_begin; t0 < t_end; t0 += STEP, ++it) {
        const int buf = it % NBUF;
        unsigned char* sa = smem + buf * STAGE;
        // the MMAs that read this stage two steps ago must have finished before it is overwritten
        if (it >= NBUF) ok = tc::mbar_wait(bar0 + 8 * buf, (uint32_t)(it / NBUF - 1) & 1u) && ok;
#pragma unroll
        for (int q = 0; q < PER_THREAD; ++q) {
            put(sa, q, xa[q]);
            if (!diag) put(sa + STRIP, q, xg[q]);
        }
        if (t0 + STEP < t_end) prefetch(t0 + STEP);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (warp == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (tc::elect_one()) {
                const uint64_t a0 = desc0 + (uint32_t)(buf * (STAGE >> 4)), g0 = diag ? a0 : a0 + (STRIP >> 4);
#pragma unroll
                for (int ks = 0; ks < STEP / 16; ++ks)
#pragma unroll
                    for (int q = 0; q < 6; ++q) {
                        if (q >= nprod) break;
                        tc::umma_bf16(q == 0 ? tmem_d : tmem_d + TILE, a0 + ((tc::split_piece_a(q) * PIECE + ks * 2 * (int)SBO) >> 4),
                                      g0 + ((tc::split_piece_b(q) * PIECE + ks * 2 * (int)SBO) >> 4), idesc,
                                      (it > 0 || ks > 0 || q > 1) ? 1u : 0u);
                    }
                tc::umma_commit(bar0 + 8 * buf);
                if (t0 + STEP >= t_end) tc::umma_commit(bar_done);
            }
            __syncwarp();
        }
    }
    const bool work = it > 0;
    if (work) ok = tc::mbar_wait(bar_done, 0) && ok;
    if (!ok) abort_flag = 1;
    __syncthreads();
    ok = abort_flag == 0;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // every thread block of the cluster has finished its products: all operand stages may become receive areas
    cluster.sync();

    // partial rows -> their owners (thread block r owns rows [r R, (r + 1) R) of the tile): slice `rank` there.  NaN
    // marks a tile whose products never completed (a bounded wait expired), so that it cannot pass for a result.
    const int R = TILE / cs;
    float* recv = reinterpret_cast<float*>(smem);
    {
        const int a = (warp & 3) * 32 + lane;
        const uint32_t tq = tmem_d + ((uint32_t)((warp & 3) * 32) << 16);
        float* dst = cluster.map_shared_rank(recv, a / R) + rank * (R * TILE);
#pragma unroll 1
        for (int c0 = (warp >> 2) * 32; c0 < TILE; c0 += 64) {
            uint32_t v[32], w[32];
            if (work && ok) {
                tc::tmem_ld32_pair_wait(tq + (uint32_t)c0, v, tq + (uint32_t)(TILE + c0), w);
            } else {
#pragma unroll
                for (int e = 0; e < 32; ++e) { v[e] = ok ? 0u : 0x7FC00000u; w[e] = 0u; }
            }
#pragma unroll
            for (int e = 0; e < 32; e += 4)
                *reinterpret_cast<float4*>(dst + slice_offset(a % R, c0 + e)) =
                    make_float4(__uint_as_float(v[e]) + __uint_as_float(w[e]),
                                __uint_as_float(v[e + 1]) + __uint_as_float(w[e + 1]),
                                __uint_as_float(v[e + 2]) + __uint_as_float(w[e + 2]),
                                __uint_as_float(v[e + 3]) + __uint_as_float(w[e + 3]));
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(ACC_COLS) : "memory");
    }
    cluster.sync();      // the slices have arrived; from here on nobody touches another thread block's memory

    const int a_base = tm * TILE + rank * R, c_base = tn * TILE;
    auto emit = [&](int64_t r, int64_t c, float x) {
        float* p = F + r * ld_f + c;
        if (add_out) atomicAdd(p, x); else *p = x;
    };
    // four entries of a row of F at once where it allows that (vec_f), which a tile on the diagonal or at the edge does not (n = 4,656,
    // k = 1,024, four clusters to a tile: 54.0 us entry by entry, 47.7 so, 45.7 without the bank conflicts of the mirror image)
    auto emit4 = [&](int64_t r, int64_t c, const float4& x) {
        float* p = F + r * ld_f + c;
        if (!add_out) *reinterpret_cast<float4*>(p) = x;
        else asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x.x), "f"(x.y), "f"(x.z), "f"(x.w) : "memory");
    };
    // The others leave entry by entry, by the thread that added up the four: one after the other by consecutive lanes, from slice 0 and
    // behind a barrier, was slower (k = 1,023 54.1 us, 55.3 so; k = 2,050 244, 247).
    const bool whole = vec_f && !diag && a_base + R <= k && c_base + TILE <= k;
    for (int e = tid; e < R * CHUNKS * 2; e += THREADS) {
        const int row = e / (CHUNKS * 2), c = e % (CHUNKS * 2) * 4, off = slice_offset(row, c);
        float4 x = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        for (int q = 0; q < cs; ++q) {
            const float4 y = *reinterpret_cast<const float4*>(recv + q * (R * TILE) + off);
            x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w;
        }
        x.x *= scale; x.y *= scale; x.z *= scale; x.w *= scale;
        *reinterpret_cast<float4*>(recv + off) = x;        // slice 0 keeps the finished rows for the mirror image
        const int a = a_base + row, cc = c_base + c;
        if (whole) {
            emit4(a, cc, x);
        } else {
            // a tile on the diagonal keeps its upper half and mirrors it, so that F is symmetric to the bit (where one cluster has the
            // tile: what several add into it arrives in any order)
            const float y[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (a < k && cc + u < k && (!diag || a <= cc + u)) emit(a, cc + u, y[u]);
        }
    }
    __syncthreads();
    if (whole) {
        // consecutive threads: consecutive columns of the mirror image (R / 4 divides THREADS: the rows of a thread stay the same)
        const int row = tid % (R / 4) * 4;
        for (int c = tid / (R / 4); c < TILE; c += THREADS / (R / 4))
            emit4(c_base + c, a_base + row, make_float4(recv[slice_offset(row, c)], recv[slice_offset(row + 1, c)],
                                                        recv[slice_offset(row + 2, c)], recv[slice_offset(row + 3, c)]));
        return;
    }
    const int row = tid % R, a = a_base + row;
    for (int c = tid / R; c < TILE; c += THREADS / R) {
        const int cc = c_base + c;
        if (a < k && cc < k && (!diag || a < cc)) emit(cc, a, recv[slice_offset(row, c)]);
    }
}

}  // namespace gram

grass_status launch_fim(const float* X, int64_t n, int64_t k, int64_t ld, float scale, float* F, int64_t ld_f,
                        cudaStream_t st)
{
    using namespace gram;
    int dev = 0, sms = 148;
    if (cuda_failed(cudaGetDevice(&dev))) return GRASS_ERR_CUDA;
    if (cuda_failed(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return GRASS_ERR_CUDA;
    constexpr size_t smem = (size_t)NBUF * STAGE;
    if (cuda_failed(cudaFuncSetAttribute(gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) ||
        cuda_failed(cudaFuncSetAttribute(gram_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100)))
        return GRASS_ERR_CUDA;
    const int64_t tiles = (k + TILE - 1) / TILE, ntiles = tiles * (tiles + 1) / 2;
    // Thread blocks per tile: enough to fill the machine (two per SM) with at least four steps each, and no accumulator
    // over more than 8,192 samples.  Up to eight are one cluster; what is beyond that are further clusters.
    const int64_t slots = 2 * (int64_t)sms;
    int64_t want = std::max<int64_t>(1, slots / ntiles);
    want = std::min<int64_t>(want, std::max<int64_t>(1, n / (4 * STEP)));
    want = std::max<int64_t>(want, (n + 8191) / 8192);
    // With many tiles, pairs: wide clusters leave SMs of a partition idle (36 tiles: 46 us with pairs, 66 with fours and 67 with
    // eights at n = 4,656, k = 1,024; 21 tiles, k = 768: 36, 38 and 42); with few tiles, eights save global reductions (10 tiles:
    // 12.5 us, 14.6 with fours and 19.7 with pairs at n = 512, k = 512).
    int64_t cs = 1;
    // (eight also where there are too few samples for them: each stores an eighth of the tile)
    while (cs < (ntiles >= 16 ? 2 : 8) && (cs * 2 <= want || ntiles < 16)) cs *= 2;
    int64_t groups = std::max<int64_t>(1, want / cs);
    groups = std::max<int64_t>(groups, (n + 8192 * cs - 1) / (8192 * cs));
    int64_t chunk = (n + groups * cs - 1) / (groups * cs);
    chunk = (chunk + STEP - 1) / STEP * STEP;
    if (ntiles * groups * cs > 0x7FFFFFFFLL) return GRASS_ERR_UNSUPPORTED;
    const int add_out = groups > 1;
    if (add_out && cuda_failed(cudaMemset2DAsync(F, (size_t)ld_f * sizeof(float), 0, (size_t)k * sizeof(float), (size_t)k, st)))
        return GRASS_ERR_CUDA;
    int nprod = (int)tuning(GRASS_TUNE_SPLIT_PRODUCTS, tc::kSplitProductsDefault);
    if (nprod != 3 && nprod != 4) nprod = 6;
    const int vec_ok = (uintptr_t)X % 16 == 0 && ld % 4 == 0, vec_f = (uintptr_t)F % 16 == 0 && ld_f % 4 == 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(ntiles * groups * cs), 1, 1);
    cfg.blockDim = dim3(THREADS, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, gram_kernel, X, (int32_t)n, (int32_t)k, ld, (int32_t)tiles,
                                             (int32_t)(groups * cs), (int32_t)chunk,
                                             scale, F, ld_f, vec_ok, vec_f, add_out, nprod);
    return cuda_ok(e);
}

}  // namespace grass
