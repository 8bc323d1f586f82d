// grass_score on the 5th-generation tensor cores (tcgen05 + TMEM), fp32-accurate, CTA pairs, TMA loads.
//
// scores[i, m] = <train[i, :], test[m, :]> (attribute stage, Section 2.1) is the one dense contraction
// of the path.  fp32 inputs are split exactly into three bf16 pieces, x = hi + mid + lo (8 significant
// bits each, by truncation), and the product is rebuilt from the six partial products whose weight is
// at least 2^-16 of the leading one (hi*hi, hi*mid, mid*hi, mid*mid, hi*lo, lo*hi); what is dropped is
// below 2^-23 of |x||y|, the size of one fp32 rounding.  hi*hi accumulates in one fp32 tile in tensor
// memory and the five correction terms in a second one; the epilogue adds the two.
//
// Two CTAs on neighbouring SMs (a cluster of 2) own a 256 x (<=256) output tile and run one
// tcgen05.mma.cta_group::2 (M = 256, N <= 256, K = 16) per product: each CTA stages its own 128 train
// rows and HALF of the test rows, the tensor cores of both SMs read both halves, and each CTA ends up
// with its 128 x N accumulators in its own tensor memory.
//   warp 17    one thread brings the raw fp32 tiles (128 rows x 32 k-values each, train and test) from
//              global memory into a ring of shared-memory slots with TMA (cp.async.bulk.tensor.2d, 128-byte
//              swizzle, each CTA loading only for itself); rows and k-values beyond the matrices arrive as zeros;
//   warps 0-15 producers, in two groups that take alternate k tiles: read a raw slot, split, and write the
//              bf16 pieces into shared memory in the tensor
//              core's K-major layout with the 64-byte swizzle; one lane per warp then arrives on the LEADER
//              CTA's "full" barrier (a remote arrive for the second CTA) and frees the raw slot; afterwards
//              they drain their own CTA's accumulators;
//   warp 16    allocates / frees tensor memory in both CTAs; in the leader CTA one elected thread issues
//              the MMAs and commits, multicast to both CTAs, the stage-free and accumulator-ready barriers.
// Three 48 KB operand stages and two 32 KB raw slots of 32 k-values each.  Every mbarrier wait is bounded:
// if one expires the CTA marks its tile with NaN, still frees its tensor memory, and returns; the cluster
// barriers are reached by every thread of both CTAs unconditionally.
// Long contractions, and outputs with too few tiles to fill the machine, are split over blockIdx.z: every split
// adds its partial products into the zeroed output (see launch_score_tc).
// The TMA path needs 16-byte aligned bases and row strides; other inputs take the plain FMA kernel
// (grass_score.cu).
#include <algorithm>
#include <cstdlib>

#include "score_common.cuh"

namespace grass {
namespace tc {

constexpr int BM = 128;            // train rows per CTA (the pair's MMA M is 256)
constexpr int BN = 256;            // test rows per CTA pair (MMA N, upper bound); each CTA stages half
constexpr int BNH = BN / 2;
constexpr int STAGES = 3;          // bf16 operand stages
constexpr int RING = 2;            // raw fp32 slots filled by TMA
constexpr int PRODUCERS = 512;     // threads of the producer warps
constexpr int PWARPS = PRODUCERS / 32;
constexpr int THREADS = PRODUCERS + 64;   // + the MMA / tensor-memory warp and the TMA warp
constexpr int A_SPLIT_BYTES = BM * BK * 2;    // one bf16 piece of the train tile: 8 KB
constexpr int B_SPLIT_BYTES = BNH * BK * 2;   // one bf16 piece of this CTA's half of the test tile: 8 KB
constexpr int STAGE_BYTES = 3 * (A_SPLIT_BYTES + B_SPLIT_BYTES);   // 48 KB
constexpr int CHUNKS = BK / 8;     // 16-byte chunks (8 bf16) per row per stage
constexpr int GROUPS = 2;          // producer warps work in two groups that take alternate k tiles
constexpr int GROUP_THREADS = PRODUCERS / GROUPS;
constexpr int GROUP_WARPS = PWARPS / GROUPS;
constexpr int TASKS = (BM + BNH) * CHUNKS / GROUP_THREADS;   // (row, chunk) tasks per producer per k tile = 4
// Parity waits are only unambiguous if a waiter never lags a barrier by two phases:
//  - every k tile that uses a given raw slot belongs to the same group (so a group sees all phases of its slots);
//  - a group's previous tile has already waited for an MMA at least as late as the one two rounds back on any stage.
static_assert(RING % GROUPS == 0, "all tiles of a raw slot must belong to one producer group");
static_assert(GROUPS <= STAGES, "operand-stage phases must not be skipped by a producer group");
constexpr uint32_t TMEM_COLS = 512;   // two fp32 accumulators of BN columns each
constexpr int RAW_HALF = BM * BK * 4;            // one raw fp32 tile (128 rows x 32 k-values): 16 KB
constexpr int RAW_BYTES = 2 * RAW_HALF;          // train tile + this CTA's test tile
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + RING * RAW_BYTES;
static_assert(BM == BNH, "both raw tiles use the same TMA box");
static_assert(SMEM_BYTES <= 224 * 1024 && STAGE_BYTES % 1024 == 0 && RAW_HALF % 1024 == 0, "shared memory layout");

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
grass_score_tc_kernel(const __grid_constant__ CUtensorMap map_train, const __grid_constant__ CUtensorMap map_test,
                      int64_t N, int64_t M, int64_t D, int64_t kt_split, float* __restrict__ scores, int64_t ld_s,
                      int out_vec_ok, int nprod)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long bars[2 * STAGES + 1 + 2 * RING];
    __shared__ uint32_t tmem_base_slot;
    __shared__ volatile int abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_ctarank();                       // 0 = leader (issues the MMAs)
    const int64_t n0 = (int64_t)blockIdx.x * BM;                   // this CTA's train rows
    const int64_t m0 = (int64_t)blockIdx.y * BN;
    const int64_t m_rows = (M - m0) < BN ? (M - m0) : BN;          // test rows of the pair's tile
    const uint32_t n_mma = (uint32_t)((m_rows + 15) / 16 * 16);    // MMA N (a multiple of 16 for M = 256)
    const int n_half = (int)(n_mma / 2);                           // test rows staged by each CTA
    // blockIdx.z takes k tiles [kt0, kt0 + ktiles); with more than one split the tiles add their partial
    // products into the (zeroed) output
    const int64_t kt0 = (int64_t)blockIdx.z * kt_split;
    const int64_t kt_left = (D + BK - 1) / BK - kt0;
    const int64_t ktiles = kt_left < kt_split ? (kt_left > 0 ? kt_left : 0) : kt_split;
    const bool add_out = gridDim.z > 1;

    const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[STAGES]), accum = smem_u32(&bars[2 * STAGES]);
    const uint32_t rawfull0 = smem_u32(&bars[2 * STAGES + 1]), rawempty0 = rawfull0 + 8 * RING;
    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full0 + 8 * s, 2 * GROUP_WARPS);   // one arrival per warp of the stage's group in both CTAs
            mbar_init(empty0 + 8 * s, 1);
        }
        mbar_init(accum, 1);
        for (int r = 0; r < RING; ++r) {
            mbar_init(rawfull0 + 8 * r, 1);        // the TMA thread's expect_tx arrival + the bytes
            mbar_init(rawempty0 + 8 * r, GROUP_WARPS);   // one arrival per warp of the group that read the slot
        }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == PWARPS) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();            // both CTAs' barriers are initialised before anybody arrives remotely
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_d = tmem_base_slot;
    const uint32_t smem_base = smem_u32(smem);

    if (warp < PWARPS) {
        // ---------------- producers ----------------
        // The split of one k tile is a latency chain (shared-memory loads, the arithmetic, stores, the proxy
        // fence) about as long as the MMAs of a k tile, so two groups of 8 warps work on alternate k tiles.
        // task q of a thread: flat = (tid % 256) + q * 256 -> row = flat / 4 over the 256 staged rows (128
        // train rows, then this CTA's half of the test rows), chunk = flat % 4 (8 k-values = 32 raw bytes).
        // Raw tiles carry the 128-byte swizzle (16-byte unit u of row r sits at u ^ (r & 7)), operand tiles
        // the 64-byte one: both the 16-byte loads and the 16-byte stores of a quarter warp are conflict-free.
        const unsigned char* raw0 = smem + STAGES * STAGE_BYTES;
        float x[TASKS][8];
        // raw slot -> registers (the slot can be refilled as soon as every warp of the group has done this)
        auto grab = [&](int slot) {
#pragma unroll
            for (int q = 0; q < TASKS; ++q) {
                const int flat = (tid % GROUP_THREADS) + q * GROUP_THREADS;
                const int row = flat / CHUNKS, ch = flat % CHUNKS;
                const bool is_a = row < BM;
                const int r = is_a ? row : row - BM;
                const unsigned char* rt = raw0 + slot * RAW_BYTES + (is_a ? 0 : RAW_HALF) + r * 128;
                const float4 u = *reinterpret_cast<const float4*>(rt + (((2 * ch) ^ (r & 7)) << 4));
                const float4 w = *reinterpret_cast<const float4*>(rt + (((2 * ch + 1) ^ (r & 7)) << 4));
                x[q][0] = u.x; x[q][1] = u.y; x[q][2] = u.z; x[q][3] = u.w;
                x[q][4] = w.x; x[q][5] = w.y; x[q][6] = w.z; x[q][7] = w.w;
            }
        };
        // registers -> the three bf16 pieces of operand stage s
        auto stash = [&](int s) {
            unsigned char* st = smem + (size_t)s * STAGE_BYTES;
#pragma unroll
            for (int q = 0; q < TASKS; ++q) {
                const int flat = (tid % GROUP_THREADS) + q * GROUP_THREADS;
                const int row = flat / CHUNKS, ch = flat % CHUNKS;
                const bool is_a = row < BM;
                const int r = is_a ? row : row - BM;
                uint4 hi, mid, lo;
                split8(x[q], hi, mid, lo);
                unsigned char* base = is_a ? st : st + 3 * A_SPLIT_BYTES;
                const int piece = is_a ? A_SPLIT_BYTES : B_SPLIT_BYTES;
                const uint32_t off = operand_chunk_offset(r, ch);
                *reinterpret_cast<uint4*>(base + off) = hi;
                *reinterpret_cast<uint4*>(base + piece + off) = mid;
                if (nprod > 4) *reinterpret_cast<uint4*>(base + 2 * piece + off) = lo;   // no product reads it otherwise
            }
        };
        const uint32_t leader_full0 = map_to_cta(full0, 0);
        bool ok = true;
        for (int64_t kt = warp / GROUP_WARPS; kt < ktiles; kt += GROUPS) {
            const int s = (int)(kt % STAGES), slot = (int)(kt % RING);
            const uint32_t round = (uint32_t)(kt / STAGES);
            ok = mbar_wait(rawfull0 + 8 * slot, (uint32_t)(kt / RING) & 1) && !abort_flag;      // raw tile landed
            if (!ok) break;
            grab(slot);
            __syncwarp();
            if (lane == 0) mbar_arrive(rawempty0 + 8 * slot);                                     // slot may be refilled
            if (round > 0) ok = mbar_wait(empty0 + 8 * s, (round - 1) & 1) && !abort_flag;         // operand stage free
            if (!ok) break;
            stash(s);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(leader_full0 + 8 * s);
        }
        if (!ok) abort_flag = 1;

        // ---------------- epilogue: drain this CTA's accumulators ----------------
        if (ok && ktiles > 0) ok = mbar_wait(accum, 0) && !abort_flag;
        if (!ok) abort_flag = 1;
        ok = __all_sync(0xFFFFFFFFu, ok);   // tensor-memory loads below are warp-collective
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // warp w reads TMEM lanes 32*(w%4) .. +31 (= output rows); the PWARPS/4 warps that share a lane
        // group take every (PWARPS/4)-th 32-column group
        const int lane_grp = warp & 3;
        const int64_t row = n0 + lane_grp * 32 + lane;
        for (uint32_t c0 = (warp >> 2) * 32; c0 < n_mma; c0 += 32 * (PWARPS / 4)) {
            uint32_t v[32];
            if (ok && ktiles > 0) {
                uint32_t w[32];
                tmem_ld32(tmem_d + ((uint32_t)(lane_grp * 32) << 16) + c0, v);
                tmem_ld32(tmem_d + ((uint32_t)(lane_grp * 32) << 16) + BN + c0, w);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int e = 0; e < 32; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) + __uint_as_float(w[e]));
            } else {
#pragma unroll
                for (int e = 0; e < 32; ++e) v[e] = (ktiles > 0) ? 0x7FC00000u : 0u;   // NaN marks an aborted tile
            }
            if (row < N) {
                float* dst = scores + row * ld_s + m0 + c0;
                const bool vec = out_vec_ok && (int64_t)(c0 + 32) <= m_rows;
                if (add_out) {
                    if (vec) {
#pragma unroll
                        for (int e = 0; e < 32; e += 4)
                            asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst + e),
                                         "f"(__uint_as_float(v[e])), "f"(__uint_as_float(v[e + 1])),
                                         "f"(__uint_as_float(v[e + 2])), "f"(__uint_as_float(v[e + 3]))
                                         : "memory");
                    } else {
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if ((int64_t)(c0 + e) < m_rows) atomicAdd(dst + e, __uint_as_float(v[e]));
                    }
                } else if (vec) {
#pragma unroll
                    for (int e = 0; e < 32; e += 4)
                        *reinterpret_cast<uint4*>(dst + e) = make_uint4(v[e], v[e + 1], v[e + 2], v[e + 3]);
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e)
                        if ((int64_t)(c0 + e) < m_rows) dst[e] = __uint_as_float(v[e]);
                }
            }
        }
    } else if (warp == PWARPS + 1) {
        // ---------------- TMA: raw fp32 tiles into the ring ----------------
        if (lane == 0) {
            const uint32_t raw_u32 = smem_base + STAGES * STAGE_BYTES;
            const int32_t row_a = (int32_t)n0, row_b = (int32_t)(m0 + (int64_t)rank * n_half);
            int64_t issued = 0;
            for (int64_t kt = 0; kt < ktiles; ++kt) {
                const int slot = (int)(kt % RING);
                if (kt >= RING && !(mbar_wait(rawempty0 + 8 * slot, (uint32_t)(kt / RING - 1) & 1) && !abort_flag)) {
                    abort_flag = 1;
                    break;
                }
                mbar_expect_tx(rawfull0 + 8 * slot, RAW_BYTES);
                tma_load_2d(raw_u32 + slot * RAW_BYTES, &map_train, (int32_t)((kt0 + kt) * BK), row_a, rawfull0 + 8 * slot);
                tma_load_2d(raw_u32 + slot * RAW_BYTES + RAW_HALF, &map_test, (int32_t)((kt0 + kt) * BK), row_b, rawfull0 + 8 * slot);
                issued = kt + 1;
            }
            // no copy of this CTA may still be in flight when it leaves (immediate unless the CTA gave up early)
            for (int64_t kt = issued > RING ? issued - RING : 0; kt < issued; ++kt)
                if (!mbar_wait(rawfull0 + 8 * (int)(kt % RING), (uint32_t)(kt / RING) & 1)) abort_flag = 1;
        }
    } else if (lane == 0 && rank == 0) {
        // ---------------- MMA issuer (leader CTA only) ----------------
        const uint32_t idesc = make_idesc(2 * BM, n_mma);
        bool ok = true;
        for (int64_t kt = 0; kt < ktiles && ok; ++kt) {
            const int s = (int)(kt % STAGES);
            const uint32_t round = (uint32_t)(kt / STAGES);
            ok = mbar_wait_cluster(full0 + 8 * s, round & 1) && !abort_flag;
            if (!ok) break;
            // (the only thing other threads hand over here are operand stores, made visible to the tensor core by their
            // fence.proxy.async and the barrier; no tensor-memory access of another thread has to be ordered)
            const uint32_t a0 = smem_base + s * STAGE_BYTES, b0 = a0 + 3 * A_SPLIT_BYTES;
            // hi*hi goes to the first accumulator, the correction terms (2^-8 and 2^-16 of it) to the second:
            // the tensor core truncates after every accumulation, so the large sum should see as few of
            // them as possible
#pragma unroll
            for (int t = 0; t < 6; ++t) {
                if (t >= nprod) break;
#pragma unroll
                for (int ks = 0; ks < BK / 16; ++ks) {
                    const uint64_t ad = make_smem_desc(a0 + split_piece_a(t) * A_SPLIT_BYTES + ks * 32);   // 16 k values on
                    const uint64_t bd = make_smem_desc(b0 + split_piece_b(t) * B_SPLIT_BYTES + ks * 32);
                    const uint32_t acc_on = (kt > 0 || ks > 0 || t > 1) ? 1u : 0u;
                    umma_bf16_pair(t == 0 ? tmem_d : tmem_d + BN, ad, bd, idesc, acc_on);
                }
            }
            umma_commit_pair(empty0 + 8 * s);   // stage s of both CTAs may be overwritten once these MMAs are done
        }
        if (!ok) abort_flag = 1;
        if (ok && ktiles > 0) umma_commit_pair(accum);   // accumulators of both CTAs complete
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();            // nobody leaves while the other CTA may still signal it or read its tiles
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

// Split of the contraction over blockIdx.z, for two reasons.  Accuracy: the tensor core truncates the fp32
// accumulator after every MMA, a bias that grows with the number of accumulations, so one accumulator
// never runs over more than 8,192 k-values once D exceeds 16,384 (the partial sums are then added in
// round-to-nearest fp32).  Occupancy: with fewer tile pairs than SM pairs, k is split until the machine
// is about full, in pieces of at least 256 k-values.
static grass_status plan_splits(int64_t D, int64_t pairs, int bk, int64_t* splits_out, int64_t* kt_split_out)
{
    const int64_t ktiles = (D + bk - 1) / bk;
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) != cudaSuccess) return GRASS_ERR_CUDA;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return GRASS_ERR_CUDA;
    int64_t splits = D > 16384 ? (D + 8191) / 8192 : 1;
    if (pairs > 0 && pairs * 2 <= sms / 2) splits = std::max<int64_t>(splits, std::min<int64_t>(sms / 2 / pairs, D / 256));
    splits = tuning(GRASS_TUNE_SCORE_SPLITS, splits);
    splits = std::max<int64_t>(1, std::min<int64_t>(splits, std::min<int64_t>(ktiles, 65535)));
    const int64_t kt_split = (ktiles + splits - 1) / splits;
    *splits_out = (ktiles + kt_split - 1) / kt_split;
    *kt_split_out = kt_split;
    return GRASS_OK;
}

grass_status launch_score_tc(const float* train, int64_t N, int64_t ld_train, const float* test, int64_t M,
                             int64_t ld_test, int64_t D, float* scores, int64_t ld_s, cudaStream_t st)
{
    const int64_t gx = ((N + tc::BM - 1) / tc::BM + 1) / 2 * 2;   // CTA pairs: an even number of row tiles
    const int64_t gy = (M + tc::BN - 1) / tc::BN;
    if (gx > 0x7FFFFFFFLL || gy > 65535 || N > 0x7FFFFFFFLL || M > 0x7FFFFFFFLL || D > 0x7FFFFFFFLL)
        return GRASS_ERR_UNSUPPORTED;
    CUtensorMap map_train, map_test;
    if (!make_map(&map_train, train, N, D, ld_train) || !make_map(&map_test, test, M, D, ld_test)) return GRASS_ERR_CUDA;
    const size_t smem = (size_t)tc::SMEM_BYTES + 1024;
    if (cudaFuncSetAttribute(tc::grass_score_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
        cudaSuccess)
        return GRASS_ERR_CUDA;
    int64_t splits = 1, kt_split = 1;
    if (plan_splits(D, gx / 2 * gy, tc::BK, &splits, &kt_split) != GRASS_OK) return GRASS_ERR_CUDA;
    if (splits > 1 &&
        cudaMemset2DAsync(scores, (size_t)ld_s * sizeof(float), 0, (size_t)M * sizeof(float), (size_t)N, st) != cudaSuccess)
        return GRASS_ERR_CUDA;
    dim3 grid((unsigned)gx, (unsigned)gy, (unsigned)splits);
    const int out_vec_ok = ((uintptr_t)scores % 16 == 0) && (ld_s % 4 == 0);
    int nprod = (int)tuning(GRASS_TUNE_SPLIT_PRODUCTS, tc::kSplitProductsDefault);
    if (nprod != 3 && nprod != 4) nprod = 6;
    tc::grass_score_tc_kernel<<<grid, tc::THREADS, smem, st>>>(map_train, map_test, N, M, D, kt_split, scores, ld_s,
                                                               out_vec_ok, nprod);
    return launch_status();
}

}  // namespace grass
