// grass_score on the 5th-generation tensor cores (tcgen05 + TMEM), fp32-accurate, pairs of thread blocks.
//
// scores[i, m] = <train[i, :], test[m, :]> (attribute stage, Section 2.1) is the one dense contraction
// of the path.  fp32 inputs are split exactly into three bf16 pieces, x = hi + mid + lo, and the product is rebuilt
// from the six partial products whose weight is at least 2^-16 of the leading one (hi*hi, hi*mid, mid*hi, mid*mid,
// hi*lo, lo*hi); what is dropped is below 2^-23 of |x||y|, the size of one fp32 rounding.  hi*hi accumulates in one
// fp32 tile in tensor memory and the five correction terms in a second one; the epilogue adds the two.
//
// Two blocks on neighbouring SMs (a cluster of 2) own a 256 x (<=256) output tile and run one
// tcgen05.mma.cta_group::2 (M = 256, N <= 256, K = 16) per product: each block stages its own 128 train
// rows and HALF of the test rows, the tensor cores of both SMs read both halves, and each block ends up
// with its 128 x N accumulators in its own tensor memory.
//   warp 17    one thread brings the raw fp32 tiles (32 k-values of this block's train and test rows) from global memory
//              into a ring of shared-memory slots with TMA (128-byte swizzle); rows and k-values beyond the matrices
//              arrive as zeros;
//   warps 0-15 producers, in two groups that take alternate k tiles: read a raw slot, split, and write the pieces into
//              shared memory in the tensor core's K-major layout with the 64-byte swizzle; one lane per warp then arrives
//              on the LEADER's "full" barrier (a remote arrive for the second block) and frees the raw slot; after
//              a tile's last k tile they drain their block's accumulators;
//   warp 16    allocates / frees tensor memory in both blocks; in the leader one elected thread issues the MMAs
//              and commits, multicast to both blocks, the stage-free and accumulator-ready barriers.
// What bounds it: a stage's round trip (split 0.5 us, proxy fence 0.6-0.9, arrival at the leader, MMAs 0.8, commit)
// divided by the number of stages, next to the MMAs themselves.  Narrow tiles (few test rows) have smaller stages
// and so get more of them.  (Loading from global memory straight into the producers' registers, to free the ring for a
// fourth stage, took 229 us instead of 152 at 16,384 x 256 x 4,096: 64 KB of loads in flight per SM are not enough.)
// Work is cut by k: the pairs share all (tile, k tile) units evenly where that beats whole tiles per pair; a tile that one
// pair covers alone is stored, pieces are added into the zeroed output.  No accumulator runs over more than 8,192
// k-values once D exceeds 16,384.
// Every mbarrier wait is bounded: if one expires the block marks its tile with NaN, still frees its tensor memory, and
// returns; the cluster barriers are reached by every thread of both blocks unconditionally.
// TMA needs 16-byte aligned bases and row strides; other inputs take the plain FMA kernel (grass_score.cu).
#include <algorithm>

#include "score_common.cuh"

namespace grass {
namespace tc {

constexpr int BM = 128;            // train rows per block (the pair's MMA M is 256)
constexpr int BN = 256;            // test rows per pair (MMA N, upper bound); each block stages half
constexpr int BNH = BN / 2;
constexpr int MAX_STAGES = 6;      // bf16 operand stages
constexpr int MAX_RING = 4;        // raw fp32 slots filled by TMA
constexpr int PRODUCERS = 512;     // threads of the producer warps
constexpr int PWARPS = PRODUCERS / 32;
constexpr int THREADS = PRODUCERS + 64;       // + the MMA / tensor-memory warp and the TMA warp
constexpr int A_SPLIT_BYTES = BM * BK * 2;    // one bf16 piece of the train tile: 8 KB
constexpr int RAW_A = BM * BK * 4;            // raw fp32 train tile (128 rows x 32 k-values): 16 KB
constexpr int CHUNKS = BK / 8;     // 16-byte chunks (8 bf16) per row per stage
constexpr int GROUPS = 2;          // producer warps work in two groups that take alternate k tiles
constexpr int GROUP_THREADS = PRODUCERS / GROUPS;
constexpr int GROUP_WARPS = PWARPS / GROUPS;
constexpr int TASKS = (BM + BNH) * CHUNKS / GROUP_THREADS;   // (row, chunk) tasks per producer per k tile = 4
// Parity waits are only unambiguous if a waiter never lags a barrier by two phases:
//  - every k tile that uses a given raw slot belongs to the same group (so a group sees all phases of its slots): the
//    number of slots is a multiple of GROUPS;
//  - a group's previous tile has already waited for an MMA at least as late as the one two rounds back on any stage: at
//    least GROUPS stages.
constexpr uint32_t TMEM_COLS = 512;   // two fp32 accumulators of BN columns each
constexpr int SMEM_BUDGET = 224 * 1024;
constexpr int64_t MAX_RUN = 8192 / BK;        // k tiles per accumulator run when D > 16,384

struct ScorePlan {
    WorkPlan work;
    int64_t tiles_n;       // row tiles of 256
    int width;             // test rows per tile, a multiple of 32
    int stages, ring;
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
grass_score_tc_kernel(const __grid_constant__ CUtensorMap map_train, const __grid_constant__ CUtensorMap map_test,
                      const __grid_constant__ ScorePlan plan, int64_t N, int64_t M, float* __restrict__ scores, int64_t ld_s,
                      int out_vec_ok, int nprod)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long bars[2 * MAX_STAGES + 2 * MAX_RING + 2];
    __shared__ uint32_t tmem_base_slot;
    __shared__ volatile int abort_flag;

    const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
    const uint32_t rank = cluster_ctarank();                       // 0 = leader (issues the MMAs)
    int64_t u0, u1;
    pair_range(plan.work, blockIdx.x >> 1, u0, u1);
    const int n_half = plan.width / 2;                             // test rows staged by each block
    const int S = plan.stages, ring = plan.ring;
    const int b_split = n_half * BK * 2, stage_bytes = 3 * (A_SPLIT_BYTES + b_split), raw_bytes = RAW_A + n_half * BK * 4;

    // rawfull[r]: the raw tile of slot r has landed; rawempty[r]: its group has read it; full[s] (leader): both blocks' pieces of a k tile are in stage s; empty[s] (both): the MMAs that read it are done;
    // accum (both): a segment's accumulators are complete; drained (leader): both blocks have read them
    const uint32_t full0 = smem_u32(&bars[0]), empty0 = full0 + 8 * MAX_STAGES;
    const uint32_t rawfull0 = empty0 + 8 * MAX_STAGES, rawempty0 = rawfull0 + 8 * MAX_RING;
    const uint32_t accum = rawempty0 + 8 * MAX_RING, drained = accum + 8;
    if (tid == 0) {
        for (int r = 0; r < MAX_RING; ++r) {
            mbar_init(rawfull0 + 8 * r, 1);              // the TMA thread's expect_tx arrival + the bytes
            mbar_init(rawempty0 + 8 * r, GROUP_WARPS);   // one arrival per warp of the group that read the slot
        }
        for (int s = 0; s < MAX_STAGES; ++s) {
            mbar_init(full0 + 8 * s, 2 * GROUP_WARPS);   // one arrival per warp of the stage's group in both blocks
            mbar_init(empty0 + 8 * s, 1);
        }
        mbar_init(accum, 1);
        mbar_init(drained, 2 * PWARPS);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    cluster_sync_all();            // both blocks' barriers are initialised before anybody arrives remotely
    early_wait();                  // (launch and set-up lie under the end of the kernel before)
    if (warp == PWARPS) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    // (what the other block has allocated the MMAs touch only after its operands, which come after this barrier there)
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    early_go();                    // (this block has its tensor memory)
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_d = tmem_base_slot;
    const uint32_t smem_base = smem_u32(smem);

    if (warp < PWARPS) {
        // ---------------- producers ----------------
        // The split of one k tile is a latency chain (shared-memory loads, the arithmetic, stores, the proxy
        // fence) about as long as the MMAs of a k tile, so two groups of 8 warps work on alternate k tiles.
        // task q of a thread: flat = (tid % 256) + q * 256 -> row = flat / 4 over the staged rows (128 train rows, then this
        // block's half of the test rows), chunk = flat % 4 (8 k-values = 32 raw bytes).  Raw tiles carry the 128-byte
        // swizzle (16-byte unit u of row r sits at u ^ (r & 7)), operand tiles the 64-byte one: both the 16-byte
        // loads and the 16-byte stores of a quarter warp are conflict-free.
        const unsigned char* raw0 = smem + S * stage_bytes;
        const int group = warp / GROUP_WARPS;
        const int ch = tid % CHUNKS, row0 = (tid % GROUP_THREADS) / CHUNKS;     // task q: row0 + 64 q
        const uint32_t leader_full0 = map_to_cta(full0, 0), leader_drained = map_to_cta(drained, 0);
        bool ok = true;
        int64_t u = u0;
        Segment seg;
        int n0 = 0;                    // k tiles of the segments before
        int n = group;                 // this group's next k tile, its stage and raw slot and how often these came round
        int s = group % S, slot = group;
        uint32_t round = (uint32_t)(group / S), raw_round = 0;
        for (int i = 0; next_segment(plan.work, u, u1, seg); ++i) {
            const int64_t tn = seg.tile % plan.tiles_n, tm = seg.tile / plan.tiles_n;
            const int64_t row_a = tn * (2 * BM) + rank * BM, m0 = tm * plan.width;
            const int len = (int)(seg.k1 - seg.k0);
            while (ok && n < n0 + len) {
                ok = mbar_wait(rawfull0 + 8 * slot, raw_round & 1) && !abort_flag;      // raw tile landed
                if (!ok) break;
                float x[TASKS][8];
#pragma unroll
                for (int q = 0; q < TASKS; ++q) {
                    const int row = row0 + q * (GROUP_THREADS / CHUNKS);
                    const bool is_a = q < TASKS / 2;
                    const int r = is_a ? row : row - BM;
                    if (!is_a && r >= n_half) continue;
                    const unsigned char* rt = raw0 + slot * raw_bytes + (is_a ? 0 : RAW_A) + r * 128;
                    const float4 a = *reinterpret_cast<const float4*>(rt + (((2 * ch) ^ (r & 7)) << 4));
                    const float4 b = *reinterpret_cast<const float4*>(rt + (((2 * ch + 1) ^ (r & 7)) << 4));
                    x[q][0] = a.x; x[q][1] = a.y; x[q][2] = a.z; x[q][3] = a.w;
                    x[q][4] = b.x; x[q][5] = b.y; x[q][6] = b.z; x[q][7] = b.w;
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(rawempty0 + 8 * slot);                                      // slot may be refilled
                if (round > 0) ok = mbar_wait(empty0 + 8 * s, (round - 1) & 1) && !abort_flag;         // operand stage free
                if (!ok) break;
                unsigned char* st = smem + (size_t)s * stage_bytes;
#pragma unroll
                for (int q = 0; q < TASKS; ++q) {
                    const int row = row0 + q * (GROUP_THREADS / CHUNKS);
                    const bool is_a = q < TASKS / 2;
                    const int r = is_a ? row : row - BM;
                    if (!is_a && r >= n_half) continue;
                    uint4 hi, mid, lo;
                    split8(x[q], hi, mid, lo);
                    unsigned char* base = is_a ? st : st + 3 * A_SPLIT_BYTES;
                    const int piece = is_a ? A_SPLIT_BYTES : b_split;
                    const uint32_t off = operand_chunk_offset(r, ch);
                    *reinterpret_cast<uint4*>(base + off) = hi;
                    *reinterpret_cast<uint4*>(base + piece + off) = mid;
                    if (nprod > 4) *reinterpret_cast<uint4*>(base + 2 * piece + off) = lo;   // no product reads it otherwise
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive_operands(leader_full0 + 8 * s);
                n += GROUPS;
                s += GROUPS;
                while (s >= S) { s -= S; ++round; }
                slot += GROUPS;
                if (slot >= ring) { slot -= ring; ++raw_round; }
            }
            n0 += len;
            if (!ok) abort_flag = 1;

            // ---------------- epilogue: drain this block's accumulators ----------------
            if (ok) ok = mbar_wait(accum, (uint32_t)i & 1) && !abort_flag;
            if (!ok) abort_flag = 1;
            ok = __all_sync(0xFFFFFFFFu, ok);   // tensor-memory loads below are warp-collective
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // warp w reads TMEM lanes 32*(w%4) .. +31 (= output rows); the PWARPS/4 warps that share a lane
            // group take every (PWARPS/4)-th 32-column group
            const int lane_grp = warp & 3;
            const int64_t row = row_a + lane_grp * 32;
            const int rows = (int)((N - row) < 32 ? (N - row) : 32);
            const bool whole = seg.k0 == 0 && seg.k1 == plan.work.ktiles;
            const int cols = (int)((M - m0) < plan.width ? (M - m0) : plan.width);
            // all MMAs are done and the producers have not begun the next segment (the barrier below): the operand
            // stages serve as scratch
            float* scratch = reinterpret_cast<float*>(smem) + warp * 1024;
            for (int c0 = (warp >> 2) * 32; c0 < cols; c0 += 32 * (PWARPS / 4)) {
                uint32_t v[32];
                if (ok) {
                    uint32_t w[32];
                    const uint32_t acc0 = tmem_d + ((uint32_t)(lane_grp * 32) << 16) + (uint32_t)c0;
                    tmem_ld32_pair_wait(acc0, v, acc0 + BN, w);
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) + __uint_as_float(w[e]));
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = 0x7FC00000u;   // NaN marks an aborted tile
                }
                emit_block<32>(scratch, v, scores + row * ld_s + m0 + c0, ld_s, rows, cols - c0, out_vec_ok != 0, !whole);
            }
            asm volatile("bar.sync 1, %0;" ::"n"(PRODUCERS) : "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(leader_drained);
        }
    } else if (warp == PWARPS + 1) {
        // ---------------- TMA: raw fp32 tiles into the ring ----------------
        const uint32_t raw_u32 = smem_base + S * stage_bytes;
        bool ok = true;
        int slot = 0;
        uint32_t wrapped = 0;
        int64_t u = u0;
        Segment seg;
        while (ok && next_segment(plan.work, u, u1, seg)) {
            const int64_t tn = seg.tile % plan.tiles_n, tm = seg.tile / plan.tiles_n;
            const int32_t row_a = (int32_t)(tn * (2 * BM) + rank * BM), row_b = (int32_t)(tm * plan.width + rank * n_half);
            const int len = (int)(seg.k1 - seg.k0);
            int32_t x = (int32_t)(seg.k0 * BK);
            for (int kt = 0; kt < len; ++kt, x += BK) {
                if (wrapped > 0) ok = mbar_wait(rawempty0 + 8 * slot, (wrapped - 1) & 1) && !abort_flag;
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                if (elect_one()) {
                    const uint32_t bar = rawfull0 + 8 * slot, dst = raw_u32 + slot * raw_bytes;
                    mbar_expect_tx(bar, (uint32_t)raw_bytes);
                    tma_load_2d(dst, &map_train, x, row_a, bar);
                    tma_load_2d(dst + RAW_A, &map_test, x, row_b, bar);
                }
                __syncwarp();
                if (++slot == ring) { slot = 0; ++wrapped; }
            }
        }
        if (!ok) abort_flag = 1;
        // no copy of this block may still be in flight when it leaves (immediate unless the block gave up early)
        for (int q = 0; q < ring; ++q)                 // slot q was last filled in round wrapped (q < slot) or the one before
            if ((q < slot || wrapped > 0) && !mbar_wait(rawfull0 + 8 * q, (q < slot ? wrapped : wrapped - 1) & 1)) abort_flag = 1;
    } else if (rank == 0) {
        // ---------------- MMA issuer (leader only) ----------------
        const uint32_t idesc = make_idesc(2 * BM, (uint32_t)plan.width);
        const uint64_t desc0 = make_smem_desc(smem_base);      // addresses below are 16-byte units added to it
        bool ok = true;
        int s = 0;
        uint32_t phase = 0;
        int64_t u = u0;
        Segment seg;
        for (int i = 0; ok && next_segment(plan.work, u, u1, seg); ++i) {
            if (i > 0) ok = mbar_wait_cluster(drained, (uint32_t)(i - 1) & 1) && !abort_flag;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int len = (int)(seg.k1 - seg.k0);
            for (int kt = 0; ok && kt < len; ++kt) {
                // (what other threads hand over here are operand stores, made visible to the tensor core by their
                // fence.proxy.async and the barrier; no tensor-memory access of another thread has to be ordered)
                ok = mbar_wait(full0 + 8 * s, phase) && !abort_flag;
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                if (elect_one()) {
                    const uint64_t a0 = desc0 + (uint32_t)(s * stage_bytes >> 4), b0 = a0 + (3 * A_SPLIT_BYTES >> 4);
                    // hi*hi goes to the first accumulator, the correction terms (2^-8 and 2^-16 of it) to the second:
                    // the tensor core truncates after every accumulation, so the large sum should see as few of
                    // them as possible
#pragma unroll
                    for (int t = 0; t < 6; ++t) {
                        if (t >= nprod) break;
#pragma unroll
                        for (int ks = 0; ks < BK / 16; ++ks) {
                            const uint64_t ad = a0 + ((split_piece_a(t) * A_SPLIT_BYTES + ks * 32) >> 4);   // 16 k values on
                            const uint64_t bd = b0 + (uint32_t)((split_piece_b(t) * b_split + ks * 32) >> 4);
                            const uint32_t acc_on = (kt > 0 || ks > 0 || t > 1) ? 1u : 0u;
                            umma_bf16_pair(t == 0 ? tmem_d : tmem_d + BN, ad, bd, idesc, acc_on);
                        }
                    }
                    umma_commit_pair(empty0 + 8 * s);   // stage s of both blocks may be overwritten once these MMAs are done
                    if (kt + 1 == len) umma_commit_pair(accum);        // accumulators of both blocks complete
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
    if (warp == PWARPS) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(TMEM_COLS) : "memory");
    }
}

}  // namespace tc

// true if the tensor-core path can take these operands (TMA wants 16-byte aligned bases and row strides)
bool score_tc_supported(const float* train, int64_t ld_train, const float* test, int64_t ld_test, int64_t D)
{
    return D > 0 && ((uintptr_t)train % 16 == 0) && ((uintptr_t)test % 16 == 0) && (ld_train % 4 == 0) &&
           (ld_test % 4 == 0) && encode_tiled_fn() != nullptr;
}

grass_status launch_score_tc(const float* train, int64_t N, int64_t ld_train, const float* test, int64_t M,
                             int64_t ld_test, int64_t D, float* scores, int64_t ld_s, cudaStream_t st)
{
    if (N > 0x7FFFFFFFLL || M > 0x7FFFFFFFLL || D > 0x7FFFFFFFLL) return GRASS_ERR_UNSUPPORTED;
    int dev = 0, sms = 148;
    if (cuda_failed(cudaGetDevice(&dev))) return GRASS_ERR_CUDA;
    if (cuda_failed(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return GRASS_ERR_CUDA;
    tc::ScorePlan p;
    const int64_t tiles_m = (M + tc::BN - 1) / tc::BN;
    p.width = (int)(((M + tiles_m - 1) / tiles_m + 31) / 32 * 32);
    p.tiles_n = (N + 2 * tc::BM - 1) / (2 * tc::BM);
    const int64_t ktiles = (D + tc::BK - 1) / tc::BK;
    const int64_t run = D > 16384 ? tc::MAX_RUN : ktiles;
    // a k tile takes 0.8 us (1,536 cycles of MMAs at 256 columns)
    bool adds;
    const int64_t used = tc::plan_work(p.work, p.tiles_n * tiles_m, ktiles, run, sms / 2, 8, 10, tuning(GRASS_TUNE_SCORE_SPLITS, -1), &adds);
    // raw slots: two, four where they are small; stages: what is left
    const int n_half = p.width / 2, stage_bytes = 3 * (tc::A_SPLIT_BYTES + n_half * tc::BK * 2), raw_bytes = tc::RAW_A + n_half * tc::BK * 4;
    p.ring = p.width <= 64 ? 4 : 2;
    p.stages = std::min(tc::MAX_STAGES, (tc::SMEM_BUDGET - p.ring * raw_bytes) / stage_bytes);
    const size_t smem = (size_t)p.stages * stage_bytes + (size_t)p.ring * raw_bytes;
    CUtensorMap map_train, map_test;
    if (!make_map(&map_train, train, N, D, ld_train) || !make_map(&map_test, test, M, D, ld_test, false, n_half)) return GRASS_ERR_CUDA;
    if (cuda_failed(cudaFuncSetAttribute(tc::grass_score_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::SMEM_BUDGET)))
        return GRASS_ERR_CUDA;
    if (adds && cuda_failed(cudaMemset2DAsync(scores, (size_t)ld_s * sizeof(float), 0, (size_t)M * sizeof(float), (size_t)N, st)))
        return GRASS_ERR_CUDA;
    const int out_vec_ok = ((uintptr_t)scores % 16 == 0) && (ld_s % 4 == 0);
    int nprod = (int)tuning(GRASS_TUNE_SPLIT_PRODUCTS, tc::kSplitProductsDefault);
    if (nprod != 3 && nprod != 4) nprod = 6;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * used), 1, 1);
    cfg.blockDim = dim3(tc::THREADS, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1] = {early_launch()};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cuda_ok(cudaLaunchKernelEx(&cfg, tc::grass_score_tc_kernel, map_train, map_test, p, N, M, scores, ld_s, out_vec_ok, nprod));
}

}  // namespace grass
