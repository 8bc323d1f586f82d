// Pieces shared by the score kernels: TMA loads and their barriers, operations on a pair of thread blocks, tensor maps.
#pragma once

#include <cuda.h>

#include <algorithm>

#include "grass_common.cuh"
#include "tcgen05_util.cuh"

namespace grass {
namespace tc {

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// 2-D tiled TMA load into this CTA's shared memory; x = first k-value (a multiple of 32: 128 bytes), y = first row
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int32_t x, int32_t y, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// address of the same shared-memory location in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_cta(uint32_t local_addr, uint32_t rank)
{
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local_addr), "r"(rank));
    return ra;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// the same without a cluster-scope fence, for operand tiles whose writers have already passed fence.proxy.async: each
// tensor core reads its own block's shared memory, so no other block has to see the writes (the fence costs a
// microsecond)
__device__ __forceinline__ void mbar_arrive_operands(uint32_t cluster_addr)
{
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// bounded wait with cluster-scope acquire (the arrivals come from both CTAs)
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity)
{
    for (uint32_t it = 0; it < SPIN_LIMIT; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred P;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 P, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, P;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t tmem_d, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                               uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// arrives on the barrier at this shared-memory offset in both CTAs once all MMAs issued so far are done
__device__ __forceinline__ void umma_commit_pair(uint32_t bar)
{
    const uint16_t mask = 3;
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"(mask)
                 : "memory");
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// A warp's 32 x 32 piece of an accumulator (v: row = lane, 32 columns) stored or added at dst (row stride ld; rows, cols:
// how many of each exist, from 0).  It goes through `scratch` (32 x W floats of the warp's own shared memory, W columns
// at a time) so that consecutive lanes touch consecutive addresses: with a row per lane every instruction met 32
// half-used sectors, and draining 128 x 256 took 5 us.  vec: dst and ld allow 16-byte accesses.
template <int W>
__device__ __forceinline__ void emit_block(float* scratch, const uint32_t (&v)[32], float* dst, int64_t ld, int rows, int cols,
                                           bool vec, bool add)
{
    static_assert(W == 16 || W == 32, "one or two passes");
    constexpr int U = W / 4;                   // 16-byte units per row
    const int lane = threadIdx.x & 31;
    // unit u of row r sits at u ^ swz(r): conflict-free by rows and by columns
    auto at = [](int r, int u) { return r * W + ((u ^ (W == 32 ? (r & 7) : ((r >> 1) & 3))) << 2); };
#pragma unroll
    for (int p = 0; p < 32 / W; ++p) {
        __syncwarp();
#pragma unroll
        for (int u = 0; u < U; ++u)
            *reinterpret_cast<uint4*>(scratch + at(lane, u)) =
                make_uint4(v[p * W + 4 * u], v[p * W + 4 * u + 1], v[p * W + 4 * u + 2], v[p * W + 4 * u + 3]);
        __syncwarp();
        if (vec && (p + 1) * W <= cols) {
            const int u = lane % U, r0 = lane / U;
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const int r = r0 + j * (32 / U);
                if (r >= rows) continue;
                const float4 x = *reinterpret_cast<const float4*>(scratch + at(r, u));
                float* d = dst + r * ld + p * W + 4 * u;
                if (add)
                    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(d), "f"(x.x), "f"(x.y), "f"(x.z), "f"(x.w)
                                 : "memory");
                else
                    *reinterpret_cast<float4*>(d) = x;
            }
        } else {
            const int c = lane % W, r0 = lane / W;
#pragma unroll 4
            for (int j = 0; j < W; ++j) {
                const int r = r0 + j * (32 / W);
                if (r >= rows || p * W + c >= cols) continue;
                const float x = scratch[at(r, c >> 2) + (c & 3)];
                float* d = dst + r * ld + p * W + c;
                if (add) atomicAdd(d, x);
                else *d = x;
            }
        }
    }
}

// How a contraction's (tile, k tile) units are dealt out to `pairs` pairs of blocks.
struct WorkPlan {
    int64_t ktiles;        // k tiles per tile
    int64_t units;         // tiles * ktiles
    int64_t per_pair;      // units per pair
    int64_t split;         // > 0: pair q takes piece q % split of tile q / split; 0: one contiguous range of all units
    int64_t run;           // longest accumulator run in k tiles; runs start at multiples of it within a tile
};
// pair q's range of units
__device__ __forceinline__ void pair_range(const WorkPlan& p, int64_t q, int64_t& u0, int64_t& u1)
{
    if (p.split > 0) {
        const int64_t tile = q / p.split;
        u0 = tile * p.ktiles + (q - tile * p.split) * p.per_pair;
        u1 = (tile + 1) * p.ktiles;
        u1 = u0 + p.per_pair < u1 ? u0 + p.per_pair : u1;
    } else {
        u0 = q * p.per_pair;
        u1 = u0 + p.per_pair < p.units ? u0 + p.per_pair : p.units;
    }
}
// a contiguous piece of one tile: k tiles [k0, k1)
struct Segment { int64_t tile, k0, k1; };
__device__ __forceinline__ bool next_segment(const WorkPlan& p, int64_t& u, int64_t end, Segment& s)
{
    if (u >= end) return false;
    s.tile = u / p.ktiles;
    s.k0 = u - s.tile * p.ktiles;
    int64_t k1 = (s.k0 / p.run + 1) * p.run;
    k1 = k1 < p.ktiles ? k1 : p.ktiles;
    k1 = k1 < s.k0 + (end - u) ? k1 : s.k0 + (end - u);
    s.k1 = k1;
    u += k1 - s.k0;
    return true;
}
// Chooses the cheapest of: whole tiles, pieces of tiles (one per pair), an even cut of all units.  Costs in k tiles:
// drain = emptying the pipeline and the accumulators after a segment, zero = zeroing the output that pieces are added
// into.  forced > 0: that many pieces per tile.  Returns the number of pairs; *adds: pieces are added; *least (nullable):
// the cost of the plan that was found, forced or not.
inline int64_t plan_work(WorkPlan& p, int64_t tiles, int64_t ktiles, int64_t max_run, int64_t pairs, int64_t drain, int64_t zero,
                         int64_t forced, bool* adds, int64_t* least = nullptr)
{
    p.ktiles = ktiles;
    p.units = tiles * ktiles;
    p.run = max_run < ktiles ? max_run : ktiles;
    const int64_t runs = (ktiles + p.run - 1) / p.run;
    const int64_t rounds = (tiles + pairs - 1) / pairs;
    int64_t best = rounds * (ktiles + runs * drain) + (runs > 1 ? zero : 0);
    p.split = 1;
    p.per_pair = ktiles;
    if (rounds > 1) { p.split = 0; p.per_pair = rounds * ktiles; }
    for (int64_t s = 2; s * tiles <= pairs; ++s) {
        const int64_t per = (ktiles + s - 1) / s;
        if ((ktiles + per - 1) / per != s) continue;
        const int64_t cost = per + ((per + p.run - 1) / p.run) * drain + zero;
        if (cost < best) { best = cost; p.split = s; p.per_pair = per; }
    }
    const int64_t even = (p.units + pairs - 1) / pairs;
    const int64_t segments = even / p.run + 2;             // at most
    if (even + segments * drain + zero < best) { best = even + segments * drain + zero; p.split = 0; p.per_pair = even; }
    if (least) *least = best;
    if (forced > 0) {
        p.per_pair = (ktiles + std::min(forced, ktiles) - 1) / std::min(forced, ktiles);
        p.split = (ktiles + p.per_pair - 1) / p.per_pair;
    }
    if (p.per_pair <= p.run) p.run = ktiles;               // no piece is longer than a run
    *adds = p.per_pair % ktiles != 0 || p.run < ktiles;
    return p.split > 0 ? tiles * p.split : (p.units + p.per_pair - 1) / p.per_pair;
}

}  // namespace tc

// cuTensorMapEncodeTiled through the runtime's driver entry point (the library does not link libcuda)
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_tiled_fn()
{
    static EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return (EncodeTiledFn)p;
    }();
    return fn;
}

// rows x D matrix with row stride ld, read in boxes of box_rows rows x 128 bytes with the 128-byte swizzle: 32 fp32
// k-values, or 64 bf16 k-values (then the box is an operand tile as it stands); elements outside the matrix are
// delivered as zeros
inline bool make_map(CUtensorMap* map, const void* base, int64_t rows, int64_t D, int64_t ld, bool bf16 = false,
                     int box_rows = 128)
{
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return false;
    const size_t esz = bf16 ? 2 : 4;
    const cuuint64_t gdim[2] = {(cuuint64_t)D, (cuuint64_t)rows};
    const cuuint64_t gstride[1] = {(cuuint64_t)ld * esz};
    const cuuint32_t box[2] = {(cuuint32_t)(bf16 ? 64 : 32), (cuuint32_t)box_rows};
    const cuuint32_t estride[2] = {1, 1};
    return enc(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base),
               gdim, gstride, box, estride, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace grass
