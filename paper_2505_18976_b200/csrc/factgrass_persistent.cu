// FactGraSS (Section 3.3.2) with persistent thread blocks: the gathers of the next work never wait for the projection of
// the last.
//
// The streaming kernel (factgrass.cu) gives every (layer, sample, token chunk, block tile) a thread block of its own: loads,
// then hashes, atomics and a flush, with nothing in flight meanwhile but what a neighbour on the same SM has; and a block
// above 64 x 64 is cut into tiles that gather the same columns again.  Here one thread block per SM walks an equal share
// of all 32-token steps of the launch, whole 128 x 128 blocks at a time:
//   warps 0-7   gather: thread (c, g) owns masked column c and every second 8-token group of a step, two register sets, so
//               that the loads of the next two steps are in flight while this one is written to the operand tiles (K-major,
//               64-byte swizzle) and multiplied (tcgen05.mma, accumulators in tensor memory); columns and pointers of
//               the next (layer, sample) are fetched one segment ahead;
//   warps 8-15  project the finished accumulator of the segment before (two accumulators alternate): every entry's
//               bucket and sign come from a table (written once per call for all samples), bins in shared memory, one
//               flush.  The last accumulator is projected and flushed by all sixteen warps.
// A (layer, sample) that one thread block covers alone is stored; pieces are added into zeroed rows (SJLT is linear).
// No accumulator runs over more than 8,192 tokens.
//
// What bounds it: DRAM, by the 64-byte pieces that the masks touch (a step takes what 1/148 of 6.6 TB/s gives it, whether
// one or two steps are ahead), and for short launches what lies around the gathers: 8 us until the first data are there and
// 10 us for the last projection (a shared-memory fp32 addition is a compare-and-swap, 26 cycles per warp and instruction
// here; eight projecting warps instead of four took 6 us off, four swaps per thread at a time put 30 us on).
// Measured, streaming -> persistent (us): packed fp32, 12 layers x 7 samples of 640 tokens on average, 128 x 128: 144 -> 97;
// bf16, 24 layers x 8 x 512, 128 x 128: 194 -> 103 (503 MB of pieces); fp32, the same at 96 x 96: 208 -> 132 (686 MB);
// fp32, 28 layers of a 4,096-wide model x 2 x 1,024: 182 -> 154.  64 x 64 tiles were slower here (fp32, 12 layers x 5 x
// 300: 34 -> 38) and stay with the streaming kernel.
#include "factgrass_common.cuh"

#include <algorithm>

namespace grass {
namespace fgp {

constexpr int TILE = 128;
constexpr int GATHER = 256;                    // gathering threads
constexpr int EPI_WARPS = 8;
constexpr int THREADS = GATHER + EPI_WARPS * 32;
constexpr int NBUF = 2;
constexpr int MAX_RUN = 8192 / kTokTile;       // steps per accumulator run
constexpr int MAX_VAR_B = 1024;                // samples of their own lengths whose work is shared out evenly
constexpr uint16_t NO_ENTRY = 0xFFFF;          // table entry of a position outside the k'_in x k'_out block
// fp32 operand tiles (96 KB) and the bins stay within 164 KB of shared memory.  With less than 92 KB of L1 behind them the
// gathers of one SM fall from 6.6 to 4.6 TB/s (of all SMs): L1 holds a line for every one in flight.
constexpr uint32_t MAX_K = 14336;

struct Args {
    const LayerDesc* descs;        // NULL: `single`
    int32_t L, B, T;
    const int64_t* tok_begin;
    const int32_t* tok_count;
    float* out;
    int64_t ld_out;
    const uint16_t* table;         // per layer TILE x TILE entries (bucket | sign << 15)
    uint32_t* dev_status;
    int nprod;
};

// How the steps of a launch are dealt out: layer after layer, sample after sample, an equal contiguous range per block.
struct Deal {
    int64_t per_layer, units, per_block;
};
__host__ __device__ __forceinline__ Deal deal_out(int64_t per_layer, int32_t L, int64_t blocks)
{
    Deal d;
    d.per_layer = per_layer;
    d.units = per_layer * L;
    d.per_block = (d.units + blocks - 1) / blocks;
    return d;
}

// Writes the table of every layer and zeroes the output rows that are added into: all of them for samples of their own
// lengths, else those that lie across two blocks' shares.
__global__ void __launch_bounds__(256)
prepare_kernel(const __grid_constant__ Args x, const __grid_constant__ LayerDesc single, uint16_t* __restrict__ table, int64_t steps,
               int64_t blocks)
{
    // the main kernel may start: its projecting warps wait for this grid's results before they use them
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int l = blockIdx.y;
    const LayerDesc& L = x.descs ? x.descs[l] : single;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
    for (int e = tid; e < TILE * TILE; e += stride) {
        const int a = e / TILE, c = e % TILE;
        uint16_t v = NO_ENTRY;
        if (a < L.kin && c < L.kout) {
            const uint64_t h = sjlt_hash_counter(L.seed, (uint64_t)a * (uint64_t)L.kout + (uint64_t)c + 1);
            v = (uint16_t)(sjlt_bucket(h, L.k) | ((uint32_t)h << 15));
        }
        table[(int64_t)l * (TILE * TILE) + e] = v;
    }
    const Deal d = deal_out(steps * x.B, x.L, blocks);
    for (int b = blockIdx.x; b < x.B; b += gridDim.x) {
        // first unit of (l, b), and the first block boundary behind it
        const int64_t u = (int64_t)l * d.per_layer + (int64_t)b * steps;
        const int64_t bound = (u / d.per_block + 1) * d.per_block;
        const bool shared = x.tok_count != nullptr || steps == 0 || steps > MAX_RUN || bound < u + steps || L.kin == 0 || L.kout == 0;
        if (shared)
            for (uint32_t i = threadIdx.x; i < L.k; i += blockDim.x) x.out[(int64_t)b * x.ld_out + L.out_offset + i] = 0.0f;
    }
}

struct Segment {
    int32_t l, b;
    int32_t k0, k1;        // steps of the sample
    bool whole;            // all of the sample's steps
};

// walks the segments of a range of units; every thread runs its own copy
struct Walk {
    int64_t u, end;
    int32_t per_layer_steps;       // steps per sample, or 0: prefix[]
    const int32_t* prefix;         // B + 1 entries (shared memory) where samples have their own lengths
    int32_t B;
    int64_t per_layer;
    __device__ __forceinline__ bool next(Segment& s)
    {
        if (u >= end) return false;
        s.l = (int32_t)(u / per_layer);
        const int32_t r = (int32_t)(u - (int64_t)s.l * per_layer);
        int32_t n, r0;
        if (per_layer_steps > 0) {
            s.b = r / per_layer_steps;
            r0 = s.b * per_layer_steps;
            n = per_layer_steps;
        } else {
            int32_t lo = 0, hi = B;                        // the last b with prefix[b] <= r
            while (hi - lo > 1) {
                const int32_t mid = (lo + hi) >> 1;
                if (prefix[mid] <= r) lo = mid; else hi = mid;
            }
            s.b = lo;
            r0 = prefix[lo];
            n = prefix[lo + 1] - r0;
        }
        s.k0 = r - r0;
        int32_t k1 = (s.k0 / MAX_RUN + 1) * MAX_RUN;
        k1 = min(k1, n);
        if (end - u < (int64_t)(k1 - s.k0)) k1 = s.k0 + (int32_t)(end - u);
        s.k1 = k1;
        s.whole = s.k0 == 0 && k1 == n;
        u += k1 - s.k0;
        return true;
    }
};

template <bool F32>
__global__ void __launch_bounds__(THREADS, 1)
factgrass_persistent_kernel(const __grid_constant__ Args x, const __grid_constant__ LayerDesc single, uint32_t max_k)
{
    using elem_t = typename in_elem<F32>::type;
    constexpr int NP = F32 ? 3 : 1;                        // bf16 pieces per operand
    constexpr int PIECE = TILE * (int)tc::ROW_BYTES;       // one piece of an operand tile (TILE rows x 32 tokens)
    constexpr int STAGE = 2 * NP * PIECE;
    constexpr int GROUPS = GATHER / TILE;                  // 8-token groups covered by one pass
    constexpr int PASS = 4 / GROUPS;                       // passes per step
    constexpr uint32_t ACC = F32 ? 2 * TILE : TILE;        // tensor-memory columns per accumulator
    constexpr uint32_t COLS = 2 * ACC;

    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long bars[NBUF + 4];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    __shared__ int32_t prefix[MAX_VAR_B + 1];
    float* bins = reinterpret_cast<float*>(smem + NBUF * STAGE);

    const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
    // stage[b]: the MMAs that read operand buffer b are done; full[a]: accumulator a is complete; empty[a]: it was read
    const uint32_t stage0 = tc::smem_u32(&bars[0]), full0 = tc::smem_u32(&bars[NBUF]), empty0 = tc::smem_u32(&bars[NBUF + 2]);
    if (tid == 0) {
        for (int i = 0; i < NBUF; ++i) tc::mbar_init(stage0 + 8 * i, 1);
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(full0 + 8 * i, 1);
            tc::mbar_init(empty0 + 8 * i, EPI_WARPS);
        }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&tmem_slot)), "r"(COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // a sample's tokens: Tb = T and row0 = b * T without the per-sample arrays; a length outside [0, T] is clamped
    auto tokens_of = [&](int b) {
        int n = x.T;
        if (x.tok_count) {
            n = __ldg(x.tok_count + b);
            n = n < 0 ? 0 : min(n, x.T);
        }
        return n;
    };
    const bool var = x.tok_count != nullptr;
    if (var && warp == GATHER / 32) {
        int32_t carry = 0;
        for (int b0 = 0; b0 < x.B; b0 += 32) {
            const int b = b0 + lane;
            const int32_t v = b < x.B ? (tokens_of(b) + kTokTile - 1) / kTokTile : 0;
            int32_t incl = v;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, d);
                if (lane >= d) incl += t;
            }
            if (b < x.B) prefix[b + 1] = carry + incl;
            carry += __shfl_sync(0xFFFFFFFFu, incl, 31);
        }
        if (lane == 0) prefix[0] = 0;
    }
    if (x.tok_count && x.dev_status && blockIdx.x == 0 && warp == 0)
        for (int b = lane; b < x.B; b += 32) {
            const int n = __ldg(x.tok_count + b);
            if (n < 0 || n > x.T) atomicOr(x.dev_status, GRASS_DEV_BAD_LENGTH);
        }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_d = tmem_slot;
    Walk walk;
    {
        walk.per_layer_steps = var ? 0 : (x.T + kTokTile - 1) / kTokTile;
        walk.prefix = prefix;
        walk.B = x.B;
        const Deal d = deal_out(var ? (int64_t)prefix[x.B] : (int64_t)walk.per_layer_steps * x.B, x.L, gridDim.x);
        walk.per_layer = d.per_layer;
        walk.u = (int64_t)blockIdx.x * d.per_block;
        walk.end = walk.u + d.per_block < d.units ? walk.u + d.per_block : d.units;
    }

    // adds columns 32 * part + .., every parts-th piece of 32, of a finished accumulator to the bins
    auto project = [&](const Segment& g, int seg, int part, int parts, bool ok) {
        const int acc = seg & 1, a = (warp & 3) * 32 + lane;      // accumulator row a sits in tensor-memory lane a
        const uint16_t* row = x.table + (int64_t)g.l * (TILE * TILE) + a * TILE;
        ok = ok && tc::mbar_wait(full0 + 8 * acc, (uint32_t)(seg / 2) & 1u);
        ok = __all_sync(0xFFFFFFFFu, ok);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t d0 = tmem_d + acc * ACC + ((uint32_t)((warp & 3) * 32) << 16);
        auto add = [&](uint32_t entry, uint32_t v) {
            if (entry != NO_ENTRY && __uint_as_float(v) != 0.0f)
                atomicAdd(bins + (entry & 0x7FFFu), __uint_as_float(v ^ ((entry & 0x8000u) << 16)));
        };
#pragma unroll 1
        for (int c0 = 32 * part; c0 < TILE; c0 += 32 * parts) {
            uint4 t4[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) t4[q] = *reinterpret_cast<const uint4*>(row + c0 + 8 * q);
            uint32_t v[32];
            if (ok) {
                tc::tmem_ld32_wait(d0 + (uint32_t)c0, v);
                if constexpr (F32) {
                    uint32_t w[32];
                    tc::tmem_ld32_wait(d0 + (uint32_t)(TILE + c0), w);
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) + __uint_as_float(w[e]));
                }
            } else {
#pragma unroll
                for (int e = 0; e < 32; ++e) v[e] = 0u;
            }
            if (parts == EPI_WARPS / 4 && c0 + 32 * parts >= TILE) {     // everything that this warp reads has been read
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(empty0 + 8 * acc);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t w4[4] = {t4[q].x, t4[q].y, t4[q].z, t4[q].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    add(w4[e] & 0xFFFFu, v[8 * q + 2 * e]);
                    add(w4[e] >> 16, v[8 * q + 2 * e + 1]);
                }
            }
        }
        return ok;
    };
    auto flush = [&](const Segment& g, int first, int stride) {
        const LayerDesc& L = x.descs ? x.descs[g.l] : single;
        float* orow = x.out + (int64_t)g.b * x.ld_out + L.out_offset;
        for (uint32_t i = first; i < L.k; i += stride) {
            const float v = bins[i];
            bins[i] = 0.0f;
            if (g.whole) orow[i] = v;
            else if (v != 0.0f) atomicAdd(orow + i, v);
        }
    };

    if (warp < GATHER / 32) {
        // ---------------- gather and contract ----------------
        const int col = tid % TILE, grp = tid / TILE;
        bool bad = false;
        // what this thread needs to read its two columns of a segment
        struct Source {
            const elem_t *A, *G;       // token 0 of the sample, column 0
            int64_t d_in, d_out;
            uint32_t ca, cg;           // masked columns
            int32_t t, t_end;          // next step's first token; the segment's end (0, -1: no segment)
            bool has_a, has_g;
        };
        Walk ahead = walk;
        auto open = [&]() {
            Source r;
            Segment g;
            r.t = 0;
            r.t_end = -1;
            if (!ahead.next(g)) return r;
            const LayerDesc& L = x.descs ? x.descs[g.l] : single;
            const int64_t row0 = x.tok_begin ? __ldg(x.tok_begin + g.b) : (int64_t)g.b * x.T;
            r.d_in = L.d_in;
            r.d_out = L.d_out;
            r.has_a = col < L.kin && L.kout > 0;
            r.has_g = col < L.kout && L.kin > 0;
            r.ca = r.has_a ? (L.mask_in ? __ldg(L.mask_in + col) : (uint32_t)col) : 0u;
            r.cg = r.has_g ? (L.mask_out ? __ldg(L.mask_out + col) : (uint32_t)col) : 0u;
            r.A = reinterpret_cast<const elem_t*>(L.A) + row0 * r.d_in;
            r.G = reinterpret_cast<const elem_t*>(L.G) + row0 * r.d_out;
            r.t = g.k0 * kTokTile;
            r.t_end = min(g.k1 * kTokTile, tokens_of(g.b));
            return r;
        };
        Source cur = open(), nxt;
        auto check = [&](Source& r) {
            if (r.has_a && (int64_t)r.ca >= r.d_in) { bad = true; r.has_a = false; r.ca = 0; }
            if (r.has_g && (int64_t)r.cg >= r.d_out) { bad = true; r.has_g = false; r.cg = 0; }
            r.A += r.ca;
            r.G += r.cg;
        };
        if (cur.t_end > 0) check(cur);
        auto load1 = [](const elem_t* p) -> uint32_t {
            if constexpr (F32) return gather_u32(p); else return (uint32_t)gather_u16(p);
        };
        // issues the loads of the next step (zeros behind the last)
        auto fetch = [&](uint32_t (&ra)[PASS][8], uint32_t (&rg)[PASS][8]) {
            if (cur.t >= cur.t_end && cur.t_end > 0) {
                cur = nxt;
                if (cur.t_end > 0) {
                    check(cur);
                    nxt = open();
                }
            }
            const int t0 = cur.t;
            const bool full = t0 + kTokTile <= cur.t_end;
#pragma unroll
            for (int ps = 0; ps < PASS; ++ps) {
                const int t = t0 + (ps * GROUPS + grp) * 8;
                const elem_t* pa = cur.A + (int64_t)t * cur.d_in;
                const elem_t* pg = cur.G + (int64_t)t * cur.d_out;
                if (full) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) ra[ps][i] = cur.has_a ? load1(pa + i * cur.d_in) : 0u;
#pragma unroll
                    for (int i = 0; i < 8; ++i) rg[ps][i] = cur.has_g ? load1(pg + i * cur.d_out) : 0u;
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i) ra[ps][i] = (cur.has_a && t + i < cur.t_end) ? load1(pa + i * cur.d_in) : 0u;
#pragma unroll
                    for (int i = 0; i < 8; ++i) rg[ps][i] = (cur.has_g && t + i < cur.t_end) ? load1(pg + i * cur.d_out) : 0u;
                }
            }
            cur.t += kTokTile;
        };
        // registers -> operand tile: row = masked column, 16-byte chunk = 8-token group
        auto put = [&](unsigned char* tile0, int ch, const uint32_t (&v)[8]) {
            const uint32_t off = tc::operand_chunk_offset(col, ch);
            if constexpr (F32) {
                float f[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) f[i] = __uint_as_float(v[i]);
                uint4 hi, mid, lo;
                tc::split8(f, hi, mid, lo);
                *reinterpret_cast<uint4*>(tile0 + off) = hi;
                *reinterpret_cast<uint4*>(tile0 + PIECE + off) = mid;
                *reinterpret_cast<uint4*>(tile0 + 2 * PIECE + off) = lo;
            } else {
                *reinterpret_cast<uint4*>(tile0 + off) = pack8_bf16(v);
            }
        };
        const uint64_t desc0 = tc::make_smem_desc(tc::smem_u32(smem));
        const uint32_t idesc = tc::make_idesc(TILE, TILE);
        bool ok = true;
        int n = 0;
        uint32_t ra0[PASS][8], rg0[PASS][8], ra1[PASS][8], rg1[PASS][8];
        // the first loads leave before the second segment is looked up
        nxt.t = 0;
        nxt.t_end = -1;
        fetch(ra0, rg0);
        nxt = open();
        fetch(ra1, rg1);
        auto step = [&](uint32_t (&ra)[PASS][8], uint32_t (&rg)[PASS][8], int seg, bool first, bool last) {
            const int buf = n % NBUF, acc = seg & 1;
            // the MMAs that read this buffer NBUF steps ago must have finished before it is overwritten
            if (n >= NBUF) ok = ok && tc::mbar_wait(stage0 + 8 * buf, (uint32_t)(n / NBUF - 1) & 1u);
            unsigned char* sa = smem + buf * STAGE;
#pragma unroll
            for (int ps = 0; ps < PASS; ++ps) {
                put(sa, ps * GROUPS + grp, ra[ps]);
                put(sa + NP * PIECE, ps * GROUPS + grp, rg[ps]);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            fetch(ra, rg);
            asm volatile("bar.sync 1, %0;" ::"n"(GATHER) : "memory");
            if (warp == 0) {
                if (first && seg >= 2) ok = ok && tc::mbar_wait(empty0 + 8 * acc, (uint32_t)(seg / 2 - 1) & 1u);
                __syncwarp();
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (tc::elect_one()) {
                    // addresses in 16-byte units on top of the first descriptor
                    const uint64_t a0 = desc0 + (uint32_t)(buf * (STAGE >> 4)), g0 = a0 + (NP * PIECE >> 4);
                    const uint32_t d0 = tmem_d + acc * ACC;
#pragma unroll
                    for (int ks = 0; ks < kTokTile / 16; ++ks) {
                        if constexpr (F32) {
                            // hi*hi goes to the first accumulator, the correction terms to the second (the tensor core
                            // truncates after every accumulation, so the large sum sees as few of them as possible)
#pragma unroll
                            for (int q = 0; q < 6; ++q) {
                                if (q >= x.nprod) break;
                                tc::umma_bf16(q == 0 ? d0 : d0 + TILE, a0 + ((tc::split_piece_a(q) * PIECE + ks * 32) >> 4),
                                              g0 + ((tc::split_piece_b(q) * PIECE + ks * 32) >> 4), idesc,
                                              (!first || ks > 0 || q > 1) ? 1u : 0u);
                            }
                        } else {
                            tc::umma_bf16(d0, a0 + (ks * 32 >> 4), g0 + (ks * 32 >> 4), idesc, (!first || ks > 0) ? 1u : 0u);
                        }
                    }
                    tc::umma_commit(stage0 + 8 * buf);             // buffer free once these MMAs have read it
                    if (last) tc::umma_commit(full0 + 8 * acc);    // accumulator complete
                }
                __syncwarp();
            }
            ++n;
        };
        Segment g;
        int segs = 0;
        for (; walk.next(g); ++segs)
            for (int k = g.k0; k < g.k1; ++k) {
                if (n & 1) step(ra1, rg1, segs, k == g.k0, k + 1 == g.k1);
                else step(ra0, rg0, segs, k == g.k0, k + 1 == g.k1);
            }
        if (segs > 0) {
            // nothing left to gather: the last accumulator is everybody's work
            asm volatile("griddepcontrol.wait;" ::: "memory");
            asm volatile("bar.sync 2, %0;" ::"n"(THREADS) : "memory");
            ok = project(g, segs - 1, warp / 4, THREADS / 128, ok);
            asm volatile("bar.sync 2, %0;" ::"n"(THREADS) : "memory");
            flush(g, tid, THREADS);
        }
        if (bad && x.dev_status) atomicOr(x.dev_status, GRASS_DEV_BAD_INDEX);
        if (!ok) abort_flag = 1;
    } else {
        // ---------------- project ----------------
        const int et = tid - GATHER;
        for (uint32_t i = et; i < max_k; i += EPI_WARPS * 32) bins[i] = 0.0f;
        // the table and the zeroed rows are complete
        asm volatile("griddepcontrol.wait;" ::: "memory");
        bool ok = true;
        Segment g;
        for (int seg = 0; walk.next(g); ++seg) {
            if (walk.u >= walk.end) {
                asm volatile("bar.sync 2, %0;" ::"n"(THREADS) : "memory");      // bins are clear
                ok = project(g, seg, warp / 4, THREADS / 128, ok);
                asm volatile("bar.sync 2, %0;" ::"n"(THREADS) : "memory");
                flush(g, tid, THREADS);
                break;
            }
            asm volatile("bar.sync 3, %0;" ::"n"(EPI_WARPS * 32) : "memory");   // bins are clear
            ok = project(g, seg, warp / 4 - GATHER / 128, EPI_WARPS / 4, ok);
            asm volatile("bar.sync 3, %0;" ::"n"(EPI_WARPS * 32) : "memory");
            flush(g, et, EPI_WARPS * 32);
        }
        if (!ok) abort_flag = 1;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (abort_flag && tid == 0 && x.dev_status) atomicOr(x.dev_status, GRASS_DEV_TIMEOUT);
    if (warp == 0) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(COLS) : "memory");
    }
}

}  // namespace fgp

size_t persistent_table_bytes(int32_t L) { return (size_t)L * fgp::TILE * fgp::TILE * sizeof(uint16_t); }

bool persistent_fits(const LayerDesc* d, int32_t L, int32_t B, const int32_t* tok_count)
{
    using namespace fgp;
    if (tok_count && B > MAX_VAR_B) return false;
    for (int l = 0; l < L; ++l)
        if (d[l].kin > TILE || d[l].kout > TILE || d[l].s != 1 || d[l].k > MAX_K) return false;
    return true;
}

grass_status launch_persistent(const LayerDesc* dev_descs, const LayerDesc& single, uint32_t max_k, bool f32, int32_t L, int32_t B,
                               int32_t T, const int64_t* tok_begin, const int32_t* tok_count, float* out, int64_t ld_out, void* table,
                               uint32_t* dev_status, int sms, cudaStream_t st)
{
    using namespace fgp;
    const int64_t steps = (T + kTokTile - 1) / kTokTile, units = steps * B * L;
    // An equal share for every SM.  Where samples are longer than that and a share of one or two steps more divides a
    // sample evenly, it is taken: a share that runs into the next sample pays for a second projection (8,192 tokens of 32
    // samples at 128 x 128 fp32: 70 us in shares of 7 steps, 62 in shares of 8).
    const int64_t per = (units + sms - 1) / sms, pieces = steps / per;
    const bool even = !tok_count && pieces > 0 && steps % pieces == 0 && steps / pieces <= per + 2;
    const int64_t blocks = even ? pieces * B * L : std::min<int64_t>(sms, units);
    Args x;
    x.descs = dev_descs;
    x.L = L;
    x.B = B;
    x.T = T;
    x.tok_begin = tok_begin;
    x.tok_count = tok_count;
    x.out = out;
    x.ld_out = ld_out;
    x.table = (const uint16_t*)table;
    x.dev_status = dev_status;
    x.nprod = (int)tuning(GRASS_TUNE_SPLIT_PRODUCTS, tc::kSplitProductsDefault);
    if (x.nprod != 3 && x.nprod != 4) x.nprod = 6;
    prepare_kernel<<<dim3((unsigned)std::min(std::max(B, 8), 64), (unsigned)L, 1), 256, 0, st>>>(x, single, (uint16_t*)table, steps, blocks);
    if (launch_status() != GRASS_OK) return GRASS_ERR_CUDA;
    auto launch = [&](auto kern, int pieces) -> grass_status {
        const size_t smem = (size_t)NBUF * 2 * pieces * TILE * tc::ROW_BYTES + (size_t)max_k * 4;
        // the same limit in every call (96 KB of tiles and the longest bins): another thread may be between this and its launch
        if (cuda_failed(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024 + (int)MAX_K * 4))) return GRASS_ERR_CUDA;
        // what shared memory does not need is L1, where gathered loads wait
        int carve = 100;
        for (int kb : {64, 100, 132, 164, 196, 228})
            if ((size_t)kb * 1024 >= smem + 7 * 1024) { carve = (kb * 100 + 227) / 228; break; }
        carve = (int)tuning(GRASS_TUNE_FACTGRASS_CARVEOUT, carve);
        if (cuda_failed(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, carve))) return GRASS_ERR_CUDA;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)blocks, 1, 1);
        cfg.blockDim = dim3(THREADS, 1, 1);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, x, single, max_k);
        return cuda_ok(e);
    };
    return f32 ? launch(factgrass_persistent_kernel<true>, 3) : launch(factgrass_persistent_kernel<false>, 1);
}

}  // namespace grass
