// Plain SJLT (identity mask, the k' = p case of Section 3.3.1) through a table of the projection.
//
// All samples of a call share one projection.  The streamed path of grass_compress.cu hashes every position anew for every
// two samples (about 45 integer instructions) and is bound by that; here a first kernel writes the call's (bucket, sign)
// table once, 16 bits a position, into the caller's scratch, and the second kernel looks it up.
//   One block per SM.  Rows stream through a ring of chunks in shared memory (bulk copies, one loading warp); S = 2 rows
//   share a chunk of the table.  31 warps walk the chunk 128 positions at a time and add the non-zero values into k bins
//   per row in shared memory; the cost of that follows the non-zeros (Section 3.1).  The (rows, chunk) units are cut
//   evenly over the blocks, so there is no last wave; a row that two blocks share is added into zeroes.
// What bounds it: for dense inputs the shared-memory fp32 additions, each a compare-and-swap; HBM for sparse ones (99 % zeros: 5.5
// TB/s).  In between the additions, the rows and the table share the pipe to shared memory: at 70 % zeros it is busy for 73 % of the
// cycles (DRAM 44 %), 70 % of that with additions (a warp's takes 5.4 cycles for ten active lanes: one to read, four to swap, and
// repeats) and 29 % with rows and table; the warps wait for its answers.
// 1,024 x 131,072, k = 4,096, against the streamed path: fp32 230 -> 154 us at 70 % zeros, 109 -> 97 at 99 %;
// bf16 303 -> 139; k = 32,768 615 -> 202.
// (Turning the projection around instead, lists of positions per bucket summed without atomics, was built and measured:
// its 16-bit lists cost 30 instructions per 32 buckets and chunk and it ran at 260 us whatever the sparsity.)
#include "grass_common.cuh"
#include "tcgen05_util.cuh"

#include <algorithm>

namespace grass {
namespace sjlt {

constexpr int WARPS = 31;                        // warps that project; one more loads
constexpr int CONSUMERS = WARPS * 32;
constexpr int THREADS = CONSUMERS + 32;
constexpr int STEP = CONSUMERS * 4;              // positions that the block takes at a time, four per thread
constexpr int MAX_STAGES = 6;
constexpr int SLACK = 16;                        // elements per staged row beyond a chunk: the row's shift against 16 bytes
constexpr int SMEM_BUDGET = 224 * 1024;
constexpr uint32_t MAX_K = 32768;                // a bucket is 15 bits

struct Layout {
    int64_t p, nchunks;
    uint32_t chunk;        // positions per chunk, a multiple of 128
    uint32_t k;
    int rows;              // rows per unit (1 or 2)
    int copies;            // bins per bucket, one per lane modulo copies (a power of two)
    int stages;
    uint32_t row_elems;    // elements per staged row
    uint32_t stage_bytes;  // rows, then the table's chunk
};

// false: the bins leave no room
static bool layout_of(Layout& t, int64_t p, uint32_t k, size_t elem_bytes)
{
    if (k > MAX_K) return false;
    t.p = p;
    t.k = k;
    t.rows = (size_t)k * 8 <= 96 * 1024 ? 2 : 1;
    // Lanes of a warp that meet in one bin repeat their compare-and-swap: few bins come in copies (k = 600, dense fp32: the
    // repeats cost a sixth).
    t.copies = k <= 1024 ? 4 : (k <= 2048 ? 2 : 1);
    const size_t room = SMEM_BUDGET - (size_t)t.rows * t.copies * k * 4;
    // Chunks of up to four steps in three stages (a turn costs every warp 400 cycles of waiting, so long chunks), of about
    // equal length.
    const size_t per_pos = (size_t)t.rows * elem_bytes + 2;
    const int64_t fit = ((int64_t)(room / 3) - t.rows * SLACK * (int64_t)elem_bytes - 128) / (int64_t)per_pos / 128 * 128;
    const int64_t longest = std::min<int64_t>(fit, 4 * STEP / 128 * 128);
    if (longest < 1024) return false;
    t.nchunks = (p + longest - 1) / longest;
    t.chunk = (uint32_t)(((p + t.nchunks - 1) / t.nchunks + 127) / 128 * 128);
    t.row_elems = t.chunk + SLACK;
    t.stage_bytes = (uint32_t)(((size_t)t.rows * t.row_elems * elem_bytes + (size_t)t.chunk * 2 + 127) / 128 * 128);
    t.stages = (int)std::min<size_t>(MAX_STAGES, room / t.stage_bytes);
    return t.stages >= 3;
}

// entry = bucket | sign << 15 for every position (padded to whole chunks); and zeroes the output rows that two blocks of the
// main kernel share
__global__ void __launch_bounds__(256)
build_kernel(uint16_t* __restrict__ table, int64_t padded, uint32_t k, uint64_t seed, float* __restrict__ out, int64_t ld_out,
             int64_t n, int rows, int64_t nchunks, int64_t units, int64_t per_block, int blocks)
{
    // the main kernel may start: it waits for this grid's results before it uses them
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < padded; j += stride) {
        const uint64_t h = sjlt_hash_counter(seed, (uint64_t)j + 1);
        table[j] = (uint16_t)(sjlt_bucket(h, k) | ((uint32_t)h << 15));
    }
    // boundary c lies between blocks c and c + 1 of the main kernel
    for (int64_t c = blockIdx.x; c + 1 < blocks; c += gridDim.x) {
        const int64_t u = (c + 1) * per_block;
        if (u >= units || u % nchunks == 0) continue;
        for (int r = 0; r < rows; ++r) {
            const int64_t i = u / nchunks * rows + r;
            if (i >= n) break;
            for (uint32_t b = threadIdx.x; b < k; b += blockDim.x) out[i * ld_out + b] = 0.0f;
        }
    }
}

__device__ __forceinline__ uint32_t bits_of(const float* p) { return __float_as_uint(*p); }
__device__ __forceinline__ uint32_t bits_of(const __nv_bfloat16* p) { return (uint32_t)*reinterpret_cast<const uint16_t*>(p) << 16; }
// four consecutive elements of a staged row, as fp32 bits
__device__ __forceinline__ void load4(const float* p, uint32_t (&v)[4])
{
    const uint4 t = *reinterpret_cast<const uint4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void load4(const __nv_bfloat16* p, uint32_t (&v)[4])
{
    const uint2 t = *reinterpret_cast<const uint2*>(p);
    v[0] = t.x << 16; v[1] = t.x & 0xFFFF0000u; v[2] = t.y << 16; v[3] = t.y & 0xFFFF0000u;
}

template <typename T, int S>
__global__ void __launch_bounds__(THREADS, 1)
project_kernel(const T* __restrict__ g, int64_t n, int64_t ld, const uint16_t* __restrict__ table, const __grid_constant__ Layout lay,
               float* __restrict__ out, int64_t ld_out, int64_t units, int64_t per_block, int out_bf16, uint32_t* dev_status)
{
    constexpr int PER16 = 16 / (int)sizeof(T);
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) unsigned long long bars[2 * MAX_STAGES];
    __shared__ volatile int abort_flag;
    __shared__ int2 meta[MAX_STAGES];            // per stage: shift of row 0 | shift of row 1 << 8 | rows << 16, positions
    const int STAGES = lay.stages;
    float* bins = reinterpret_cast<float*>(smem + (size_t)STAGES * lay.stage_bytes);    // S x copies x k
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t k = lay.k, chunk = lay.chunk;
    const int64_t u0 = (int64_t)blockIdx.x * per_block;
    const int64_t u1 = u0 + per_block < units ? u0 + per_block : units;
    const uint32_t full0 = tc::smem_u32(&bars[0]), empty0 = tc::smem_u32(&bars[MAX_STAGES]);
    const uint32_t table_off = S * lay.row_elems * (uint32_t)sizeof(T);

    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            tc::mbar_init(full0 + 8 * s, 32);        // the loading warp's lanes, and the bytes
            tc::mbar_init(empty0 + 8 * s, WARPS);
        }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const int copies = lay.copies;
    const uint32_t row_bins = copies * k;
    for (uint32_t b = tid; b < S * row_bins; b += THREADS) bins[b] = 0.0f;
    __syncthreads();
    // table and zeroed rows are complete (until here only this block's own shared memory was touched)
    asm volatile("griddepcontrol.wait;" ::: "memory");

    if (warp == WARPS) {
        // ---------------- loads ----------------
        // Lane r < S copies row r of every unit, lane S the table's chunk.  A row may start anywhere inside a 16-byte granule;
        // element i of a chunk lies at i + shift of its stage, so that the granules which lie wholly inside the chunk keep
        // their alignment and one bulk copy brings them; the few elements before and behind are loaded one by one, half of
        // the warp's lanes before and half behind.  Every lane arrives once its elements are stored.
        int64_t pair = u0 / lay.nchunks, c = u0 - pair * lay.nchunks;
        int s = 0;
        uint32_t round = 0;
        bool ok = true;
        const T* row = nullptr;    // lane r < S: its row's chunk; NULL beyond the matrix
        bool fresh = true;
        for (int64_t u = u0; u < u1; ++u) {
            if (fresh) row = (lane < S && pair * S + lane < n) ? g + (pair * S + lane) * ld + c * chunk : nullptr;
            const int len = (int)(lay.p - c * chunk < chunk ? lay.p - c * chunk : chunk);
            const int shift = row ? (int)(((uintptr_t)row & 15) / sizeof(T)) : 0;
            const int head = min(shift ? PER16 - shift : 0, len);
            const int bulk = row ? (len - head) / PER16 * PER16 : 0;
            const uint32_t bytes = lane == S ? chunk * 2 : (uint32_t)(bulk * sizeof(T));
            const void* src = lane == S ? (const void*)(table + c * chunk) : (const void*)(row + head);
            const uint32_t dst = lane == S ? table_off : (uint32_t)((lane * lay.row_elems + shift + head) * sizeof(T));
            if (round > 0) ok = tc::mbar_wait(empty0 + 8 * s, (round - 1) & 1) && !abort_flag;
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            unsigned char* st = smem + s * lay.stage_bytes;
            const uint32_t bar = full0 + 8 * s;
            if (lane <= S) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                // the bytes may be counted before they are expected: the phase cannot end before this lane arrives
                if (bytes > 0) tc::bulk_copy(tc::smem_u32(st) + dst, src, bytes, bar);
            }
            int packed = 0;
#pragma unroll
            for (int r = 0; r < S; ++r) packed |= __shfl_sync(0xFFFFFFFFu, shift, r) << (8 * r);
            if (packed != 0 || len % PER16 != 0) {
#pragma unroll
                for (int r = 0; r < S; ++r) {
                    const T* rp = (const T*)(uintptr_t)__shfl_sync(0xFFFFFFFFu, (unsigned long long)(uintptr_t)row, r);
                    const int rh = __shfl_sync(0xFFFFFFFFu, head, r), rb = __shfl_sync(0xFFFFFFFFu, bulk, r);
                    const int e = lane < 16 ? lane : rh + rb + lane - 16;
                    if (rp && (lane < 16 ? e < rh : e < len))
                        reinterpret_cast<T*>(st)[r * lay.row_elems + ((packed >> (8 * r)) & 0xFF) + e] = rp[e];
                }
            }
            if (lane == 0) meta[s] = make_int2(packed | (n - pair * S < S ? (int)(n - pair * S) : S) << 16, len);
            if (lane <= S) tc::expect_tx(bar, bytes);
            else tc::mbar_arrive(bar);
            fresh = false;
            if (row) row += chunk;
            if (++c == lay.nchunks) { c = 0; ++pair; fresh = true; }
            if (++s == STAGES) { s = 0; ++round; }
        }
        if (!ok) abort_flag = 1;
        // no copy may still be in flight when the block leaves
        for (int q = 0; q < STAGES; ++q)                   // stage q was last filled in round `round` (q < s) or the one before
            if ((q < s || round > 0) && !tc::mbar_wait(full0 + 8 * q, (q < s ? round : round - 1) & 1)) abort_flag = 1;
    } else {
        // ---------------- projection ----------------
        int64_t pair = u0 / lay.nchunks;
        int c = (int)(u0 - pair * lay.nchunks);
        const int64_t whole_from = c == 0 ? pair : pair + 1;       // first rows that this block sees from their first chunk on
        int s = 0;
        uint32_t phase = 0;
        bool ok = true;
        const bool vec_out = !out_bf16 && k % 4 == 0 && ld_out % 4 == 0 && (uintptr_t)out % 16 == 0;
        // a chunk's groups of 128 positions go round the warps; the next chunk carries on where this one stopped
        int turn = warp;
        const int groups_mod = (int)(chunk / 128 % WARPS);
        float* my_bins = bins + (lane & (copies - 1)) * k;
        for (int64_t u = u0; u < u1; ++u) {
            if (ok) ok = tc::mbar_wait(full0 + 8 * s, phase) && !abort_flag;
            const unsigned char* st = smem + s * lay.stage_bytes;
            const int2 m = meta[s];
            const int rows = m.x >> 16;
            auto add = [&](int r, uint32_t entry, uint32_t v) {
                if (__uint_as_float(v) != 0.0f)
                    atomicAdd(my_bins + r * row_bins + (entry & 0x7FFFu), __uint_as_float(v ^ ((entry & 0x8000u) << 16)));
            };
            if (ok && (m.x & 0xFFFF) == 0) {
                // aligned rows: four positions per lane
                for (int j = 128 * turn + 4 * lane; j < m.y; j += STEP) {
                    const uint2 t2 = *reinterpret_cast<const uint2*>(st + table_off + 2 * j);
                    const uint32_t e[4] = {t2.x, t2.x >> 16, t2.y, t2.y >> 16};
                    uint32_t v[S][4];
#pragma unroll
                    for (int r = 0; r < S; ++r) load4(reinterpret_cast<const T*>(st) + r * lay.row_elems + j, v[r]);
                    if (j + 4 > m.y) {                     // the last positions of a row
#pragma unroll
                        for (int r = 0; r < S; ++r)
#pragma unroll
                            for (int q = 1; q < 4; ++q)
                                if (j + q >= m.y) v[r][q] = 0u;
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int r = 0; r < S; ++r)
                            if (r < rows) add(r, e[q], v[r][q]);
                }
            } else if (ok) {
                const uint16_t* tab = reinterpret_cast<const uint16_t*>(st + table_off);
#pragma unroll 2
                for (int j = tid; j < m.y; j += CONSUMERS) {
                    const uint32_t e = tab[j];
#pragma unroll
                    for (int r = 0; r < S; ++r)
                        if (r < rows) add(r, e, bits_of(reinterpret_cast<const T*>(st) + r * lay.row_elems + ((m.x >> (8 * r)) & 0xFF) + j));
                }
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(empty0 + 8 * s);
            turn -= groups_mod;
            if (turn < 0) turn += WARPS;
            if (++s == STAGES) { s = 0; phase ^= 1; }
            if (++c == (int)lay.nchunks || u + 1 == u1) {
                // the rows, or this block's part of them, are complete
                asm volatile("bar.sync 1, %0;" ::"n"(CONSUMERS) : "memory");
                const bool whole = pair >= whole_from && c == (int)lay.nchunks;
#pragma unroll
                for (int r = 0; r < S; ++r) {
                    const int64_t orow = (pair * S + r) * ld_out;
                    if (whole && vec_out) {
                        for (uint32_t b = 4 * tid; b < k; b += 4 * CONSUMERS) {
                            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                            for (int q = 0; q < copies; ++q) {
                                float4* bin = reinterpret_cast<float4*>(bins + r * row_bins + q * k + b);
                                const float4 x = *bin;
                                v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
                                *bin = make_float4(0.f, 0.f, 0.f, 0.f);
                            }
                            if (r < rows) *reinterpret_cast<float4*>(out + orow + b) = v;
                        }
                        continue;
                    }
                    for (uint32_t b = tid; b < k; b += CONSUMERS) {
                        float v = 0.0f;
                        for (int q = 0; q < copies; ++q) {
                            v += bins[r * row_bins + q * k + b];
                            bins[r * row_bins + q * k + b] = 0.0f;
                        }
                        if (r >= rows) continue;
                        if (whole) store_out(out, orow + b, v, out_bf16);
                        else if (v != 0.0f) atomicAdd(out + orow + b, v);
                    }
                }
                asm volatile("bar.sync 1, %0;" ::"n"(CONSUMERS) : "memory");
                c = 0;
                ++pair;
            }
        }
        if (!ok) {
            abort_flag = 1;
            if (lane == 0 && dev_status) atomicOr(dev_status, GRASS_DEV_TIMEOUT);
        }
    }
}

}  // namespace sjlt

size_t sjlt_table_bytes(int64_t n, int64_t p, uint32_t k, uint32_t s, size_t elem_bytes)
{
    // The table costs a launch of its own; below about 4 M values the streamed path is done by then.
    const int64_t forced = tuning(GRASS_TUNE_COMPRESS_DENSE, -1);
    if (s != 1 || n <= 0 || p <= 0 || forced == 0 || forced == 1) return 0;
    if (forced != 2 && (n < 32 || n * p < ((int64_t)4 << 20))) return 0;
    sjlt::Layout t;
    return sjlt::layout_of(t, p, k, elem_bytes) ? (size_t)t.nchunks * t.chunk * 2 : 0;
}

template <typename T>
static grass_status launch_t(const T* g, int64_t n, int64_t p, int64_t ld, const grass_sjlt_spec& sp, float* out, int64_t ld_out,
                             void* table, uint32_t* dev_status, cudaStream_t st, int out_bf16)
{
    using namespace sjlt;
    Layout t;
    if (!layout_of(t, p, sp.k, sizeof(T))) return GRASS_ERR_UNSUPPORTED;
    int dev = 0, sms = 148;
    if (cuda_failed(cudaGetDevice(&dev))) return GRASS_ERR_CUDA;
    if (cuda_failed(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return GRASS_ERR_CUDA;
    const int64_t pairs = (n + t.rows - 1) / t.rows, units = pairs * t.nchunks;
    if (t.nchunks > 0x7FFFFFFF) return GRASS_ERR_UNSUPPORTED;
    int64_t per_block = (units + sms - 1) / sms;
    if (out_bf16) per_block = (per_block + t.nchunks - 1) / t.nchunks * t.nchunks;      // a bf16 row is rounded once: whole rows
    const int64_t blocks = (units + per_block - 1) / per_block;
    const int64_t padded = t.nchunks * t.chunk;
    build_kernel<<<(unsigned)std::min<int64_t>((padded + 255) / 256, 2 * sms), 256, 0, st>>>(
        (uint16_t*)table, padded, sp.k, sp.seed, out, ld_out, n, t.rows, t.nchunks, units, per_block, (int)blocks);
    if (launch_status() != GRASS_OK) return GRASS_ERR_CUDA;
    const size_t psm = (size_t)t.stages * t.stage_bytes + (size_t)t.rows * t.copies * t.k * 4;
    auto launch = [&](auto kern) -> grass_status {
        if (cuda_failed(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDynSmemLimit))) return GRASS_ERR_CUDA;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)blocks, 1, 1);
        cfg.blockDim = dim3(THREADS, 1, 1);
        cfg.dynamicSmemBytes = psm;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, g, n, ld, (const uint16_t*)table, t, out, ld_out, units, per_block, out_bf16,
                                                 dev_status);
        return cuda_ok(e);
    };
    return t.rows == 2 ? launch(project_kernel<T, 2>) : launch(project_kernel<T, 1>);
}

grass_status launch_sjlt_table(const void* g, grass_dtype dt, int64_t n, int64_t p, int64_t ld, const grass_sjlt_spec& sp, float* out,
                               int64_t ld_out, void* table, uint32_t* dev_status, cudaStream_t st, int out_bf16)
{
    if (dt == GRASS_F32) return launch_t((const float*)g, n, p, ld, sp, out, ld_out, table, dev_status, st, out_bf16);
    return launch_t((const __nv_bfloat16*)g, n, p, ld, sp, out, ld_out, table, dev_status, st, out_bf16);
}

}  // namespace grass
