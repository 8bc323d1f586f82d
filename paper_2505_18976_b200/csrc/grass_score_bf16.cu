// grass_score_bf16: scores of compressed vectors kept in bf16 (a cache at half the size; the paper does not fix the
// storage precision, this is an option beside the fp32 path).
//
// No split of the operands is needed, so there are no producer warps: TMA writes the bf16 tiles (128-byte rows of 64
// k-values, 128-byte swizzle) straight into the K-major operand layout.  A pair of thread blocks on neighbouring SMs
// runs tcgen05.mma.cta_group::2 on 256 train rows x up to 512 test rows (two accumulators of up to 256 columns): each
// block stages its own 128 train rows and half of the test rows of every accumulator.  The loads of both blocks count
// their bytes on the LEADER's barrier (TMA's .cta_group::2 form), so a stage is complete where the MMA issuer waits for
// it; forwarding "landed" from block to block cost a microsecond per stage.
//
// Work is cut by k: the pairs share all (tile, k-tile) units evenly, each walking one contiguous range of them, so there
// is no last wave.  A tile that one pair covers alone is stored; the others are added into the zeroed output.  No
// accumulator runs over more than 8,192 k-values once D exceeds 16,384: the tensor core truncates after every MMA.
//
// What bounds it: the tensor cores for M of a few hundred, the train matrix's bytes for fewer; next to that the L2, which
// delivers (128 + M / 2) rows per block and 64 k-values, hence the 256-row pairs and a tile as wide as the test set.  One
// turn of the issuing threads (wait, expect, load; wait, multiply, commit) takes 600 cycles whatever it moves, 16 KB of
// train rows a turn are then 3.7-4.8 TB/s over the chip and 32 KB 6.7: stages of 128 k-values wherever three of them fit.
// Measured (before: 256-column pairs for M > 256, one block per 128 rows for M <= 256): 4,656 x 300 x 49,152 285 -> 138 us on
// a cool chip (164 in a loop that the power cap holds),
// 16,384 x 256 x 16,384 148 -> 128 us, 16,384 x 256 x 4,096 46 -> 42 us, 3,854 x 4 x 55,512 127 -> 83 us (5.2 TB/s).
//   warp 0-3  drain the accumulator, warp 4 allocates tensor memory and issues the MMAs (leader), warp 5 issues the loads
// Every mbarrier wait is bounded; a block whose wait expires marks its part with NaN and still reaches the cluster barrier.
#include <algorithm>

#include "score_common.cuh"

namespace grass {
namespace tc {
namespace h {

constexpr int ROWS = 128;                      // train rows per block
constexpr int BKH = 64;                        // k-values per TMA box: 128-byte rows
constexpr int ROW = BKH * 2;
constexpr int A_BYTES = ROWS * ROW;            // 16 KB
constexpr int MAX_STAGES = 12;
constexpr int EPI_WARPS = 4;
constexpr int THREADS_H = (EPI_WARPS + 2) * 32;
constexpr int SMEM_BUDGET = 216 * 1024;        // for the stages
constexpr uint32_t COLS = 512;                 // all of tensor memory: two accumulators of up to 256 columns
constexpr int64_t MAX_RUN = 8192;              // k-values per accumulator run when D > 16,384

constexpr int SCRATCH_BYTES = EPI_WARPS * 32 * 16 * 4;         // the epilogue warps' transposition buffers, behind the stages
static_assert(kSoleSmem <= SMEM_BUDGET + SCRATCH_BYTES, "what the kernel asks the right to");

struct Plan {
    WorkPlan work;         // k tiles of KW * 64 k-values, one stage each
    int64_t tiles_n;       // row tiles of 256
    int width;             // test rows per tile (a multiple of 32; of 64 above 256)
    int stages;
};

// K-major tiles with 128-byte rows and the 128-byte swizzle (8-row groups 1,024 bytes apart; 16-byte chunk c of row r at
// chunk c ^ (r & 7)); 32 * i bytes into the tile are k-values 16 i .. 16 i + 15
__device__ __forceinline__ uint64_t desc128(uint32_t addr)
{
    return (uint64_t)((addr >> 4) & 0x3FFF) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// TMA load into this block's shared memory whose bytes are counted on a barrier of the pair's leader
__device__ __forceinline__ void load_pair(uint32_t dst, const CUtensorMap* map, int32_t x, int32_t y, uint32_t leader_bar)
{
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
                 "[%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(leader_bar)
                 : "memory");
}

// KW: boxes of 64 k-values per stage; SUBS: accumulators per tile (2 for a width above 256)
template <int KW, int SUBS>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS_H, 1)
score_bf16_kernel(const __grid_constant__ CUtensorMap map_train, const __grid_constant__ CUtensorMap map_test,
                  const __grid_constant__ Plan plan, int64_t N, int64_t M, float* __restrict__ scores, int64_t ld_s,
                  int out_vec_ok)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long bars[2 * MAX_STAGES + 4];
    __shared__ uint32_t tmem_base_slot;
    __shared__ volatile int abort_flag;

    const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
    const uint32_t rank = cluster_ctarank();
    int64_t u0, u1;
    pair_range(plan.work, blockIdx.x >> 1, u0, u1);
    const int S = plan.stages;
    const int n_sub = plan.width / SUBS, n_half = n_sub / 2;      // columns per accumulator; test rows of it staged here
    const int b_bytes = n_half * ROW;                             // one box of them
    const int stage_bytes = KW * (A_BYTES + SUBS * b_bytes);      // KW train boxes, then KW test boxes per accumulator
    constexpr int nbuf = SUBS == 1 ? 2 : 1;                       // accumulators of consecutive segments alternate

    // full[s] (leader): the tiles of both blocks have landed; empty[s] (both): the MMAs that read stage s are done;
    // acc_full[b] (both): a segment's accumulator is complete; acc_empty[b] (leader): both blocks have drained it
    const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[MAX_STAGES]);
    const uint32_t acc_full0 = smem_u32(&bars[2 * MAX_STAGES]), acc_empty0 = acc_full0 + 16;
    if (tid == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(acc_full0 + 8 * b, 1);
            mbar_init(acc_empty0 + 8 * b, 2 * EPI_WARPS);
        }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    cluster_sync_all();            // both blocks' barriers are initialised before anybody signals them
    early_wait();                  // (launch and set-up lie under the end of the kernel before)
    if (warp == EPI_WARPS) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                     "r"(COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    // (what the other block has allocated the MMAs touch only after its loads, which come after this barrier there)
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    early_go();                    // (this block has its tensor memory)
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_d = tmem_base_slot;
    const uint32_t smem_base = smem_u32(smem);

    if (warp < EPI_WARPS) {
        // ---------------- epilogue: this block's 128 rows of every segment ----------------
        const uint32_t leader_empty = map_to_cta(acc_empty0, 0);
        float* scratch = reinterpret_cast<float*>(smem + S * stage_bytes) + warp * (32 * 16);
        bool ok = true;
        int64_t u = u0;
        Segment seg;
        for (int i = 0; next_segment(plan.work, u, u1, seg); ++i) {
            const int b = i % nbuf;
            if (ok) ok = mbar_wait(acc_full0 + 8 * b, (uint32_t)(i / nbuf) & 1) && !abort_flag;
            if (!ok) abort_flag = 1;
            ok = __all_sync(0xFFFFFFFFu, ok);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int64_t tn = seg.tile % plan.tiles_n, tm = seg.tile / plan.tiles_n;
            const int64_t row = tn * (2 * ROWS) + rank * ROWS + warp * 32, m0 = tm * plan.width;
            const int rows = (int)((N - row) < 32 ? (N - row) : 32);
            const bool whole = seg.k0 == 0 && seg.k1 == plan.work.ktiles;
            const int cols = (int)((M - m0) < plan.width ? (M - m0) : plan.width);
            for (int c0 = 0; c0 < cols; c0 += 32) {
                uint32_t v[32];
                if (ok) {
                    // columns of the second accumulator start at tensor-memory column 256
                    const int sub = c0 >= n_sub ? 1 : 0;
                    tmem_ld32_wait(tmem_d + ((uint32_t)(warp * 32) << 16) + (uint32_t)(b * 256 + sub * 256 + c0 - sub * n_sub), v);
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = 0x7FC00000u;        // NaN marks an aborted tile
                }
                emit_block<16>(scratch, v, scores + row * ld_s + m0 + c0, ld_s, rows, cols - c0, out_vec_ok != 0, !whole);
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(leader_empty + 8 * b);
        }
    } else if (warp == EPI_WARPS + 1) {
        // ---------------- loads (one warp per block) ----------------
        const uint32_t leader_full0 = map_to_cta(full0, 0);
        const uint32_t both = 2u * (uint32_t)stage_bytes;
        int s = 0;                                         // stage to fill next
        uint32_t wrapped = 0;                              // how often the ring has come round
        bool ok = true;
        int64_t u = u0;
        Segment seg;
        while (ok && next_segment(plan.work, u, u1, seg)) {
            const int64_t tn = seg.tile % plan.tiles_n, tm = seg.tile / plan.tiles_n;
            const int32_t row_a = (int32_t)(tn * (2 * ROWS) + rank * ROWS);
            const int32_t row_b = (int32_t)(tm * plan.width + rank * n_half);
            // pairs that cover whole tiles walk them in rotated order, so that at any moment they ask L2 for
            // different parts of the test matrix (pieces of tiles start at different k-values anyway)
            const int len = (int)(seg.k1 - seg.k0);
            const int rot = len == plan.work.ktiles && len <= 128 ? (int)((int64_t)(blockIdx.x >> 1) * len / (gridDim.x >> 1)) : 0;
            int32_t x = (int32_t)((seg.k0 + rot) * (KW * BKH));
            for (int kt = 0; kt < len; ++kt) {
                if (wrapped > 0) ok = mbar_wait(empty0 + 8 * s, (wrapped - 1) & 1) && !abort_flag;
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                if (elect_one()) {
                    const uint32_t dst = smem_base + (uint32_t)s * stage_bytes, bar = leader_full0 + 8 * s;
                    if (rank == 0) mbar_expect_tx(full0 + 8 * s, both);
#pragma unroll
                    for (int w = 0; w < KW; ++w) load_pair(dst + w * A_BYTES, &map_train, x + w * BKH, row_a, bar);
#pragma unroll
                    for (int q = 0; q < SUBS; ++q)
#pragma unroll
                        for (int w = 0; w < KW; ++w)
                            load_pair(dst + KW * A_BYTES + (q * KW + w) * b_bytes, &map_test, x + w * BKH, row_b + q * n_sub, bar);
                }
                __syncwarp();
                x = kt + rot + 1 == len ? (int32_t)(seg.k0 * (KW * BKH)) : x + KW * BKH;
                if (++s == S) { s = 0; ++wrapped; }
            }
        }
        if (!ok) abort_flag = 1;
        // no copy may still be in flight when the pair leaves: the leader's barriers count both blocks' bytes
        if (rank == 0)
            for (int q = 0; q < S; ++q)                    // stage q was last filled in round wrapped (q < s) or the one before
                if ((q < s || wrapped > 0) && !mbar_wait(full0 + 8 * q, (q < s ? wrapped : wrapped - 1) & 1)) abort_flag = 1;
    } else if (warp == EPI_WARPS && rank == 0) {
        // ---------------- MMA issuer (leader only) ----------------
        const uint32_t idesc = make_idesc(2 * ROWS, (uint32_t)n_sub);
        const uint64_t desc0 = desc128(smem_base);             // addresses below are 16-byte units added to it
        bool ok = true;
        int s = 0;
        uint32_t phase = 0;
        int64_t u = u0;
        Segment seg;
        for (int i = 0; ok && next_segment(plan.work, u, u1, seg); ++i) {
            const int b = i % nbuf;
            if (i >= nbuf) ok = mbar_wait_cluster(acc_empty0 + 8 * b, (uint32_t)(i / nbuf - 1) & 1) && !abort_flag;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int len = (int)(seg.k1 - seg.k0);
            for (int kt = 0; ok && kt < len; ++kt) {
                ok = mbar_wait(full0 + 8 * s, phase) && !abort_flag;
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                if (elect_one()) {
                    const uint64_t a0 = desc0 + (uint32_t)(s * stage_bytes >> 4), b0 = a0 + (KW * A_BYTES >> 4);
#pragma unroll
                    for (int w = 0; w < KW; ++w)
#pragma unroll
                        for (int ks = 0; ks < BKH / 16; ++ks)
#pragma unroll
                            for (int q = 0; q < SUBS; ++q)
                                umma_bf16_pair(tmem_d + (uint32_t)((b + q) * 256), a0 + ((w * A_BYTES + ks * 32) >> 4),
                                               b0 + (uint32_t)(((q * KW + w) * b_bytes + ks * 32) >> 4), idesc,
                                               (kt > 0 || w > 0 || ks > 0) ? 1u : 0u);
                    umma_commit_pair(empty0 + 8 * s);
                    if (kt + 1 == len) umma_commit_pair(acc_full0 + 8 * b);
                }
                __syncwarp();
                if (++s == S) { s = 0; phase ^= 1; }
            }
        }
        if (!ok) abort_flag = 1;
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();            // nobody leaves while the other block may still signal it or read its tiles
    if (warp == EPI_WARPS) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(COLS) : "memory");
    }
}

}  // namespace h
}  // namespace tc

bool score_bf16_supported(const void* train, int64_t ld_train, const void* test, int64_t ld_test, int64_t D)
{
    return D > 0 && ((uintptr_t)train % 16 == 0) && ((uintptr_t)test % 16 == 0) && (ld_train % 8 == 0) &&
           (ld_test % 8 == 0) && encode_tiled_fn() != nullptr;
}

grass_status launch_score_bf16(const void* train, int64_t N, int64_t ld_train, const void* test, int64_t M,
                               int64_t ld_test, int64_t D, float* scores, int64_t ld_s, cudaStream_t st)
{
    using namespace tc::h;
    if (N > 0x7FFFFFFFLL || M > 0x7FFFFFFFLL || D > 0x7FFFFFFFLL) return GRASS_ERR_UNSUPPORTED;
    int dev = 0, sms = 148;
    if (cuda_failed(cudaGetDevice(&dev))) return GRASS_ERR_CUDA;
    if (cuda_failed(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return GRASS_ERR_CUDA;
    Plan p;
    int subs = 1, kw = 1, stage_bytes = 0;
    int64_t tiles_m = 1, ktiles = 1, run = 1;
    // column tiles: as few as hold `cap` test rows each, of equal width
    auto shape = [&](int64_t cap) {
        tiles_m = (M + cap - 1) / cap;
        const int64_t want_w = (M + tiles_m - 1) / tiles_m;
        p.width = (int)(want_w <= 256 ? (want_w + 31) / 32 * 32 : (want_w + 63) / 64 * 64);
        subs = p.width > 256 ? 2 : 1;
        const int box_bytes = A_BYTES + p.width / 2 * ROW;
        kw = 3 * 2 * box_bytes <= SMEM_BUDGET && D > BKH ? 2 : 1;
        stage_bytes = kw * box_bytes;
        ktiles = (D + kw * BKH - 1) / (kw * BKH);
        run = D > 16384 ? MAX_RUN / (kw * BKH) : ktiles;
    };
    p.tiles_n = (N + 2 * ROWS - 1) / (2 * ROWS);
    // Tiles of up to 512 test rows read the train rows once for two accumulators, but take twice as long to drain as tiles of
    // up to 256, which decides for all but large problems (4,656 x 300 x 49,152: 138 us in one tile of 320, 197 in two; 4,656 x
    // 512 x 1,024: 39 and 22; 1,000 x 512 x 512: 23 and 14).  Estimated in microseconds: 64 k-values are a turn of the issuing
    // threads or the operands' way from L2, whichever is longer; then the drain and, for pieces of tiles, the zeroing.  Of 310
    // combinations of N = 1 .. 8,000, M = 257 .. 1,024 and D = 64 .. 49,152 two were more than 4 % slower than with 512.
    auto estimate = [&]() {
        const double t = kw * std::max(0.3 / kw, std::max(0.2 / 256 * p.width, 0.3 / 256 * (128 + p.width / 2)));
        tc::WorkPlan trial;
        bool unused;
        int64_t least;
        tc::plan_work(trial, p.tiles_n * tiles_m, ktiles, run, sms / 2, (int64_t)((1.0 + 0.025 * p.width) / t), (int64_t)(4.0 / t), 0, &unused, &least);
        return (double)least * t;
    };
    shape(512);
    if (subs == 2) {
        const double wide = estimate();
        shape(256);
        if (wide <= estimate()) shape(512);
    }
    p.stages = std::min(MAX_STAGES, SMEM_BUDGET / stage_bytes);
    // 64 k-values take about 0.3 us
    bool adds;
    const int64_t used = plan_work(p.work, p.tiles_n * tiles_m, ktiles, run, sms / 2, 10 / kw, 12 / kw, tuning(GRASS_TUNE_SCORE_SPLITS, -1), &adds);
    CUtensorMap map_train, map_test;
    if (!make_map(&map_train, train, N, D, ld_train, true, ROWS) ||
        !make_map(&map_test, test, M, D, ld_test, true, p.width / subs / 2))
        return GRASS_ERR_CUDA;
    if (adds && cuda_failed(cudaMemset2DAsync(scores, (size_t)ld_s * sizeof(float), 0, (size_t)M * sizeof(float), (size_t)N, st)))
        return GRASS_ERR_CUDA;
    const int out_vec = ((uintptr_t)scores % 16 == 0) && (ld_s % 4 == 0);
    auto launch = [&](auto kern) -> grass_status {
        if (cuda_failed(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BUDGET + SCRATCH_BYTES)))
            return GRASS_ERR_CUDA;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(2 * used), 1, 1);
        cfg.blockDim = dim3(THREADS_H, 1, 1);
        cfg.dynamicSmemBytes = std::max(kSoleSmem, (size_t)p.stages * stage_bytes + SCRATCH_BYTES);
        cfg.stream = st;
        cudaLaunchAttribute attr[1] = {early_launch()};
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cuda_ok(cudaLaunchKernelEx(&cfg, kern, map_train, map_test, p, N, M, scores, ld_s, out_vec));
    };
    if (kw == 2) return subs == 2 ? launch(score_bf16_kernel<2, 2>) : launch(score_bf16_kernel<2, 1>);
    return subs == 2 ? launch(score_bf16_kernel<1, 2>) : launch(score_bf16_kernel<1, 1>);
}

}  // namespace grass
