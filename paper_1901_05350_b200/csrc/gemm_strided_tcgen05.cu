// Tensor-core GEMM with fp32 accuracy on operands as they lie in memory:  C[M,N] = act( A . B + bias ),  one product or
// a batch of them, every operand with either of its two dimensions contiguous, any sizes and any 4-byte alignment.
//
// The bulk copy unit wants rows that start on 16 bytes and delivers K-contiguous tiles only from K-contiguous memory.
// Here eight loader warps fetch the tiles instead: they read global memory in runs of 32 floats along whichever dimension
// is contiguous, the next k-block's values as soon as this one's are stored, and write the K-major, 128-byte-swizzled operand
// tiles that tcgen05.mma reads (K-contiguous: a warp's 32 floats are one row, or, where rows are whole quads, four k per lane
// and four rows per warp; otherwise a lane collects four k of its own row and stores 16 bytes; all free of bank conflicts).
//
// An operand value is stored as two TF32 values, and the large products are summed in segments (umma_tile.cuh), which the
// loader warps add up between two k-blocks.  Error against 64 bits, and of fp32 multiply-adds: 1.2e-7 and 1.4e-7 at K = 64,
// 2.7e-7 and 8.0e-7 at 2001; sums of one sign 4.2e-7 and 6.6e-7 at 2001, 1.9e-6 and 2.2e-6 at 20001.
//
// A tile is 128 x BN (BN 32, 64) of C or of its transpose, whichever wastes fewer rows.  Small products are a chain of one
// load, a few MMAs and the store, so two CTAs share an SM and cover each other's latency.  With fewer tiles than CTAs fit
// the K loop is cut over a cluster of 2, 4 or 8: each CTA leaves its partial tile in its shared memory, and after a cluster
// barrier every CTA adds one band of rows from all of them, in rank order, and stores it.
//
// Bound by the loaders: a k-block costs a CTA about 2500 cycles (address arithmetic, 4-byte loads and stores) against 400
// of MMAs, fewer with 16-byte loads (64 products [199,64] . [64,199]^T 18.8 -> 16.6 us, 2001 x 2000 x 2001 203 -> 166);
// sixteen loader warps per CTA were slower (2001^3: 297 us against 220), and so was fetching the next values before
// this k-block's are stored, which takes twice the registers (2001^3: 275 us against 205).  64 products [199,64] . [64,199]:
// 1179 us as 64 launches of the CUDA-core kernel, 18.6 us here; [64,1024] . [1024,101]: 201 us and 10.5 us.
#include <algorithm>

#include "common.cuh"
#include "ptx_sm100.cuh"
#include "umma_tile.cuh"

namespace tfjsb {

using namespace ptx;
using namespace tile;

namespace {

constexpr int LOADERS = 8;
constexpr int GS_THREADS = 32 + LOADERS * 32;
constexpr int GS_MAX_STAGES = 2;  // what fits beside a second CTA, for tiles of 64 and of 32 columns
constexpr int GS_MAX_CLUSTER = 8;

// One operand: element (row, k) of product b at ptr[b * batch_stride + row * row_stride + k * k_stride].
struct Side {
    const float* ptr;
    int row_stride, k_stride;
    int rows;
    int quads;  // K-contiguous, and every row starts on 16 bytes: four k per load
    long long batch_stride;
};

struct StridedArgs {
    Side p, q;          // p: the 128 rows of a tile, q: its BN columns
    int K, num_kb, stages, splits;
    int segment;        // k-blocks per accumulator of the large products
    int p_tiles, q_tiles;
    float* c;           // element (row of p, row of q) of product b
    long long c_p, c_q, c_batch;
    const float* bias;  // along p if bias_p, else along q
    int bias_p, act;
    unsigned int* dev_status;
};

// What one loader thread fetches of a k-block of ROWS rows, and where it stores it.
template <int ROWS, bool QUADS>
struct Fetch {
    float v[ROWS / 8];

    // Rows past the last are read as the last one: their results are not stored.  k past K must be zero.
    __device__ __forceinline__ void load(const Side& s, const float* base, int r0, int k0, int K, int w, int lane) {
        const int last = s.rows - 1;
        if (QUADS && s.quads) {        // lane = 4 k of one of four rows, row 32 i + 4 w + lane / 8
            const bool ok = k0 + 4 * (lane & 7) < K;  // K % 4 == 0
            const float* at = base + k0 + 4 * (lane & 7);
#pragma unroll
            for (int i = 0; i < ROWS / 32; ++i) {
                float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
                if (ok) q = ld_global4(at + (long long)min(r0 + 32 * i + 4 * w + (lane >> 3), last) * s.row_stride);
                v[4 * i] = q.x; v[4 * i + 1] = q.y; v[4 * i + 2] = q.z; v[4 * i + 3] = q.w;
            }
        } else if (s.k_stride == 1) {  // lane = k, row w + 8 i
            const bool ok = k0 + lane < K;
            const float* at = base + k0 + lane;
#pragma unroll
            for (int i = 0; i < ROWS / 8; ++i) v[i] = ok ? ld_global(at + (long long)min(r0 + w + 8 * i, last) * s.row_stride) : 0.f;
        } else {                // lane = row of block i, k = 4 w + e; rows are contiguous
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int k = k0 + 4 * w + e;
                const float* at = base + (long long)k * s.k_stride;
#pragma unroll
                for (int i = 0; i < ROWS / 32; ++i) v[4 * i + e] = k < K ? ld_global(at + min(r0 + 32 * i + lane, last)) : 0.f;
            }
        }
    }
    // four k of one row in every 32
    __device__ __forceinline__ void store_quads(uint32_t at, uint32_t lo_offset) const {
#pragma unroll
        for (int i = 0; i < ROWS / 32; ++i) {
            float hi[4], lo[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) tf32_split(v[4 * i + e], hi[e], lo[e]);
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at + (uint32_t)i * 4096u), "f"(hi[0]), "f"(hi[1]), "f"(hi[2]), "f"(hi[3]) : "memory");
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at + lo_offset + (uint32_t)i * 4096u), "f"(lo[0]), "f"(lo[1]), "f"(lo[2]), "f"(lo[3]) : "memory");
        }
    }
    __device__ __forceinline__ void store(const Side& s, uint32_t tile, uint32_t lo_offset, int w, int lane) const {
        if (QUADS && s.quads) {
            const int row = 4 * w + (lane >> 3);
            store_quads(tile + (uint32_t)(row * 128 + (((lane ^ row) & 7) << 4)), lo_offset);
        } else if (s.k_stride == 1) {
            const uint32_t at = tile + (uint32_t)(w * 128 + (((lane >> 2) ^ w) << 4) + (lane & 3) * 4);
#pragma unroll
            for (int i = 0; i < ROWS / 8; ++i) {
                float hi, lo;
                tf32_split(v[i], hi, lo);
                asm volatile("st.shared.f32 [%0], %1;" ::"r"(at + (uint32_t)i * 1024u), "f"(hi) : "memory");
                asm volatile("st.shared.f32 [%0], %1;" ::"r"(at + lo_offset + (uint32_t)i * 1024u), "f"(lo) : "memory");
            }
        } else {
            store_quads(tile + (uint32_t)(lane * 128 + ((w ^ (lane & 7)) << 4)), lo_offset);
        }
    }
};

// One element over k0 .. k1 by fp32 multiply-adds.
__device__ __noinline__ float sum_in_fp32(const float* p, const float* q, int p_step, int q_step, int k0, int k1) {
    float acc = 0.f;
    for (int k = k0; k < k1 && acc == acc; ++k) acc = fmaf(ld_global(p + (long long)k * p_step), ld_global(q + (long long)k * q_step), acc);
    return acc;
}

// QUADS: an operand has rows of whole quads (an instance of its own: the code for them cost the others 7 %)
template <int BN, bool QUADS>
__global__ void __launch_bounds__(GS_THREADS, 2)
gemm_strided_kernel(const StridedArgs g) {
    constexpr int OPERANDS = A_STAGE_BYTES + BN * 128;  // hi (or lo) of one stage
    constexpr int STAGE_BYTES = OPERANDS * 2;
    constexpr uint32_t TMEM_COLS = 4 * BN;              // [large 0 | large 1 | small | sum]
    // Segment j has been multiplied when its last stage comes free, `stages` k-blocks later, and the loaders add it to the
    // sum before they hand over the first k-block of segment j + 2, which takes its accumulator: no barriers of its own.
    static_assert(GS_MAX_STAGES <= 2, "a segment of one k-block is added up before its accumulator is used again");
    constexpr int PITCH = BN + 1;                       // words per row of the partial tile in shared memory
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[GS_MAX_STAGES], bar_empty[GS_MAX_STAGES], bar_acc, bar_drain;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag_s;
    volatile int* abort_flag = &abort_flag_s;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    if (threadIdx.x == 0) {
        for (int s = 0; s < g.stages; ++s) {
            mbar_init(smem_u32(&bar_full[s]), LOADERS);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        mbar_init(smem_u32(&bar_acc), 1);
        mbar_init(smem_u32(&bar_drain), 1);
        abort_flag_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    pdl_wait();

    const int rank = g.splits > 1 ? (int)(blockIdx.x % (unsigned)g.splits) : 0;
    int t = (int)(blockIdx.x / (unsigned)g.splits);
    const int qt = t % g.q_tiles;
    t /= g.q_tiles;
    const int pt = t % g.p_tiles, batch = t / g.p_tiles;
    const int p0 = pt * BLOCK_M, q0 = qt * BN;
    const int kb0 = (int)((long long)g.num_kb * rank / g.splits), kb1 = (int)((long long)g.num_kb * (rank + 1) / g.splits);
    const int segments = (kb1 - kb0 + g.segment - 1) / g.segment;  // never zero (splits <= num_kb)

    if (warp == 0) {
        const uint32_t idesc = make_idesc_tf32(BLOCK_M, BN);
        const uint32_t small = tmem + 2 * BN;
        int stage = 0, in_seg = 0;
        uint32_t phase = 0, large = tmem;
        const bool leader = elect_one();
        bool ok = true, issued = false;  // the leader's
        for (int kb = kb0; kb < kb1; ++kb) {
            const uint32_t hi = base + (uint32_t)(stage * STAGE_BYTES), lo = hi + OPERANDS;
            const uint64_t ah = make_kmajor_sw128_desc(hi), bh = make_kmajor_sw128_desc(hi + A_STAGE_BYTES);
            const uint64_t al = make_kmajor_sw128_desc(lo), bl = make_kmajor_sw128_desc(lo + A_STAGE_BYTES);
            if (leader && ok && (ok = bounded_wait(smem_u32(&bar_full[stage]), phase, abort_flag))) {
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint64_t o = (uint64_t)(2 * k);
                    tc_mma_tf32(large, ah + o, bh + o, idesc, (in_seg | k) != 0 ? 1u : 0u);
                    tc_mma_tf32(small, ah + o, bl + o, idesc, (kb != kb0 || k != 0) ? 1u : 0u);
                    tc_mma_tf32(small, al + o, bh + o, idesc, 1u);
                }
                issued = true;
                tc_commit(smem_u32(&bar_empty[stage]));
            }
            if (++stage == g.stages) { stage = 0; phase ^= 1u; }
            if (++in_seg == g.segment) { in_seg = 0; large = tmem + (large == tmem ? BN : 0); }
        }
        if (leader && ok) tc_commit(smem_u32(&bar_acc));
        if (!ok) {
            if (!*abort_flag) {
                *abort_flag = 1;
                atomicOr(g.dev_status, DEV_STATUS_TIMEOUT_MMA);
            }
            if (issued) {
                tc_commit(smem_u32(&bar_drain));
                const unsigned long long t0 = global_ns();
                while (!mbar_try_wait(smem_u32(&bar_drain), 0u))
                    if (global_ns() - t0 > WAIT_LIMIT_NS) {
                        atomicOr(g.dev_status, DEV_STATUS_TIMEOUT_DRAIN);
                        break;
                    }
            }
        }
        __syncwarp();
    } else {
        const int w = warp - 1;
        const float* pb = g.p.ptr + batch * g.p.batch_stride;
        const float* qb = g.q.ptr + batch * g.q.batch_stride;
        bool ok = true;
        Fetch<BLOCK_M, QUADS> fp;
        Fetch<BN, QUADS> fq;
        fp.load(g.p, pb, p0, kb0 * BLOCK_K, g.K, w, lane);
        fq.load(g.q, qb, q0, kb0 * BLOCK_K, g.K, w, lane);
        // the sum: the two warps of a lane quadrant take 32 columns each
        const int quad = warp & 3, c0 = (w >> 2) * 32;
        const uint32_t lanes = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)c0;
        int added = 0;                                        // segments that are in the sum
        int add_at = kb0 + g.segment - 1 + g.stages;          // the k-block before which the next is added
        auto add = [&](bool last) {
            tc_fence_after();
            if (c0 < BN) add_segment<16>(lanes + (uint32_t)((added & 1) * BN), lanes + 2 * BN, lanes + 3 * BN, 32, added == 0, last);
            tc_fence_before();
            ++added;
        };
        int stage = 0;
        uint32_t phase = 0;
        for (int kb = kb0; kb < kb1; ++kb) {
            const bool got = bounded_wait(smem_u32(&bar_empty[stage]), phase ^ 1u, abort_flag);
            if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
            const uint32_t hi = base + (uint32_t)(stage * STAGE_BYTES);
            fp.store(g.p, hi, OPERANDS, w, lane);
            fq.store(g.q, hi + A_STAGE_BYTES, OPERANDS, w, lane);
            if (kb == add_at) {  // before the next values are fetched: it wants their registers
                add(false);
                add_at += g.segment;
            }
            if (kb + 1 < kb1) {
                fp.load(g.p, pb, p0, (kb + 1) * BLOCK_K, g.K, w, lane);
                fq.load(g.q, qb, q0, (kb + 1) * BLOCK_K, g.K, w, lane);
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bar_full[stage]));
            if (++stage == g.stages) { stage = 0; phase ^= 1u; }
        }
        ok = ok && bounded_wait(smem_u32(&bar_acc), 0u, abort_flag);
        if (!__all_sync(0xffffffffu, ok)) {
            if (lane == 0 && !*abort_flag) {
                *abort_flag = 1;
                atomicOr(g.dev_status, DEV_STATUS_TIMEOUT_EPILOGUE);
            }
        } else {
            // the rest of the sum (one segment or two), and the sum -> partial tile in shared memory (all operand reads are
            // done: bar_acc)
            while (added < segments) add(added + 1 == segments);
            if (c0 < BN) {
                uint32_t u[32];
                tc_ld_32x32(lanes + 3 * BN, u);
                tc_ld_wait();
                const uint32_t row = base + (uint32_t)(((quad * 32 + lane) * PITCH + c0) * 4);
                bool odd = false;
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                    odd = odd || not_finite(u[e]);
                    asm volatile("st.shared.b32 [%0], %1;" ::"r"(row + 4u * e), "r"(u[e]) : "memory");
                }
                const int pr = p0 + quad * 32 + lane;
                for (int e = 0; odd && pr < g.p.rows && e < min(32, g.q.rows - q0 - c0); ++e) {
                    uint32_t bits;
                    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(bits) : "r"(row + 4u * e) : "memory");
                    if (!not_finite(bits)) continue;
                    const float again = sum_in_fp32(pb + (long long)pr * g.p.row_stride, qb + (long long)(q0 + c0 + e) * g.q.row_stride, g.p.k_stride,
                                                    g.q.k_stride, kb0 * BLOCK_K, min(g.K, kb1 * BLOCK_K));
                    asm volatile("st.shared.f32 [%0], %1;" ::"r"(row + 4u * e), "f"(again) : "memory");
                }
            }
            tc_fence_before();
        }
    }
    // The next kernel may start now and no earlier: two CTAs fit an SM, and those of a next product that come while this one still
    // multiplies are put in pairs where they would have an SM each ([24,266].[266,3975], 128 CTAs, one after the other: 14.6 us
    // without an early start, 16.8 with one at the top, 12.6 here; [1702,1276].[1276,1679] 113, 114 to 117, 110).
    pdl_launch_dependents();
    if (g.splits > 1) {
        cluster_arrive();
        cluster_wait();
    } else {
        __syncthreads();
    }
    if (!*abort_flag && warp > 0) {
        // 256 threads, consecutive ones along the contiguous dimension of C, each walking the other dimension
        const int tid = (int)threadIdx.x - 32, band_log = 7 - (31 - __clz(g.splits)), band = 1 << band_log, r0 = rank * band;
        const bool along_p = g.c_p == 1;
        const int row = along_p ? tid & (band - 1) : tid / BN, col = along_p ? tid >> band_log : tid % BN;
        const int row_step = along_p ? 0 : 256 / BN, col_step = along_p ? 256 >> band_log : 0;
        const int p = p0 + r0 + row, q = q0 + col;
        const int limit = along_p ? min(BN, g.q.rows - q0) : min(band, g.p.rows - p0 - r0);  // of the walked dimension
        const int step = along_p ? col_step : row_step;
        const bool live = along_p ? p < g.p.rows : q < g.q.rows;
        float* out = g.c + batch * g.c_batch + (long long)p * g.c_p + (long long)q * g.c_q;
        const long long out_step = (long long)step * (along_p ? g.c_q : g.c_p);
        uint32_t at = base + (uint32_t)(((r0 + row) * PITCH + col) * 4);
        const uint32_t at_step = (uint32_t)((row_step * PITCH + col_step) * 4);
        // the bias is either one value per thread or walked along
        const bool one_bias = g.bias != nullptr && along_p == (g.bias_p != 0);
        const float b0 = one_bias && live ? ld_global(g.bias + (along_p ? p : q)) : 0.f;
        const float* bias = g.bias != nullptr && !one_bias ? g.bias + (along_p ? q0 : p0 + r0) : nullptr;
#pragma unroll 4
        for (int i = along_p ? col : row; i < (live ? limit : 0); i += step, at += at_step, out += out_step) {
            float v;
            if (g.splits == 1) {
                asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(at) : "memory");
            } else {
                float part[GS_MAX_CLUSTER];
#pragma unroll
                for (int s = 0; s < GS_MAX_CLUSTER; ++s)
                    if (s < g.splits) asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(part[s]) : "r"(map_to_cta(at, (uint32_t)s)) : "memory");
                v = part[0];
#pragma unroll
                for (int s = 1; s < GS_MAX_CLUSTER; ++s)
                    if (s < g.splits) v += part[s];
            }
            if (g.bias) v += bias ? ld_global(bias + i) : b0;
            *out = apply_act(v, g.act);
        }
    }
    if (g.splits > 1) {  // nobody leaves while its shared memory is being read
        cluster_arrive();
        cluster_wait();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

template <int BN>
cudaError_t launch_instance(StridedArgs a, int64_t tiles, cudaStream_t s) {
    auto kernel = a.p.quads || a.q.quads ? gemm_strided_kernel<BN, true> : gemm_strided_kernel<BN, false>;
    constexpr int STAGE_BYTES = (A_STAGE_BYTES + BN * 128) * 2;
    constexpr int LIMIT = 110 * 1024;  // two CTAs per SM
    cudaError_t e = smem_attr_once(reinterpret_cast<const void*>(kernel), LIMIT);
    if (e != cudaSuccess) return e;
    a.stages = (LIMIT - 1024) / STAGE_BYTES;
    if (a.stages > GS_MAX_STAGES) a.stages = GS_MAX_STAGES;
    const int own_kb = (a.num_kb + a.splits - 1) / a.splits;
    if (a.stages > own_kb) a.stages = own_kb;
    size_t smem = (size_t)a.stages * STAGE_BYTES;
    const size_t partial = (size_t)BLOCK_M * (BN + 1) * 4;
    if (smem < partial) smem = partial;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * a.splits));
    cfg.blockDim = dim3(GS_THREADS);
    cfg.dynamicSmemBytes = smem + 1024;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (a.splits > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = (unsigned)a.splits;
        attr[n].val.clusterDim.y = 1;
        attr[n].val.clusterDim.z = 1;
        ++n;
    }
    if (g_launch_pdl) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, a);
}

// Cycles of one k-block (two CTAs sharing the SM) and of everything around the K loop, as measured; used to choose
// between shapes only.
constexpr int64_t FIXED_CYCLES = 8000, CLUSTER_CYCLES = 2000;
int64_t kb_cycles(int bn) { return bn == 64 ? 1100 : 800; }

struct Choice {
    bool swap = false;
    int bn = 0, splits = 1;
    int64_t tiles = 0, cycles = INT64_MAX;
};
Choice choose(int64_t batches, int64_t M, int64_t N, int64_t K, int sm_count) {
    Choice best;
    const int64_t nkb = (K + BLOCK_K - 1) / BLOCK_K, capacity = 2 * (int64_t)sm_count;
    for (int swap = 0; swap < 2; ++swap) {
        const int64_t P = swap ? N : M, Q = swap ? M : N;
        for (int bn = 32; bn <= 64; bn <<= 1) {
            const int64_t tiles = batches * ((P + BLOCK_M - 1) / BLOCK_M) * ((Q + bn - 1) / bn);
            for (int s = 1; s <= GS_MAX_CLUSTER; s <<= 1) {
                if (s > 1 && (tiles * s > capacity || nkb < 2 * s)) break;
                const int64_t rounds = (tiles * s + capacity - 1) / capacity;
                const int64_t cycles = rounds * ((nkb + s - 1) / s * kb_cycles(bn) + FIXED_CYCLES) + (s > 1 ? CLUSTER_CYCLES : 0);
                if (cycles < best.cycles) {
                    best.swap = swap != 0;
                    best.bn = bn;
                    best.splits = s;
                    best.tiles = tiles;
                    best.cycles = cycles;
                }
            }
            if (bn >= Q) break;
        }
    }
    return best;
}

// One product over 16 terms or fewer, a single k-block of the CUDA-core kernel, takes what its tiles and their stores take:
// there 128 x 128 tiles, here 128 x 64.  The CUDA cores are faster while an SM has one of the larger tiles at most (60 products
// 5.0 to 7.3 us here and mostly 0.7 to 0.95 of that there: [1,3].[3,1] 5.1 and 4.4, [254,9].[9,3] 5.7 and 5.0, [16000,7].[7,13] 6.6
// and 5.9; [20000,7].[7,9], 157 tiles, 7.6 and 9.7), and beyond that where the smaller tiles are 1.6 times as many or more
// ([30000,7].[7,101] 15.3 and 12.0, [704,15].[15,6921] 19.8 and 18.0, [9000,7].[7,260] 13.7 and 12.9, but
// [100000,7].[7,33] 21.7 and 28.4, [20000,7].[7,130] 15.2 and 16.3, [1000000,3].[3,1] 133 and 268).  55 products of 17 to 50 terms
// take 0.5 to 0.9 of the time of the CUDA cores ([2,17].[17,5] 5.0 and 6.6, [3235,19].[19,7969] 75 and 107).  Batches have
// one launch here and one per product there.
bool short_sum_on_cuda_cores(int64_t M, int64_t N, int64_t K, int sm_count) {
    if (K > 16) return false;
    const int64_t wide = ((M + 127) / 128) * ((N + 127) / 128);
    const int64_t narrow = std::min(((M + 127) / 128) * ((N + 63) / 64), ((N + 127) / 128) * ((M + 63) / 64));
    return wide <= sm_count || 5 * narrow >= 8 * wide;
}

}  // namespace

bool gemm_strided_supported(int64_t batches, int64_t M, int64_t N, int64_t K, int sm_count) {
    constexpr int64_t LIM = (1LL << 31) - 256;
    if (batches == 1 && short_sum_on_cuda_cores(M, N, K, sm_count)) return false;
    return batches >= 1 && M >= 1 && N >= 1 && K >= 1 && M < LIM && N < LIM && K <= SPLIT_MAX_K && batches < LIM &&
           (double)batches * (double)((M + 31) / 32) * (double)((N + 31) / 32) < 1e9;
}

cudaError_t launch_gemm_strided(const float* a, int64_t a_rs, int64_t a_ks, const float* b, int64_t b_ks, int64_t b_cs, const float* bias,
                                int act, float* c, int64_t batches, int64_t M, int64_t N, int64_t K, int sm_count,
                                unsigned int* dev_status, cudaStream_t s, int64_t* launches) {
    if (M == 0 || N == 0 || batches == 0) return cudaSuccess;
    const Choice ch = choose(batches, M, N, K, sm_count);
    const bool aligned = K % 4 == 0;  // and so are the products of a batch
    const bool a_quads = aligned && a_ks == 1 && a_rs % 4 == 0 && (reinterpret_cast<uintptr_t>(a) & 15u) == 0;
    const bool b_quads = aligned && b_ks == 1 && b_cs % 4 == 0 && (reinterpret_cast<uintptr_t>(b) & 15u) == 0;
    const Side sa{a, (int)a_rs, (int)a_ks, (int)M, a_quads, M * K}, sb{b, (int)b_cs, (int)b_ks, (int)N, b_quads, K * N};
    StridedArgs g{};
    g.p = ch.swap ? sb : sa;
    g.q = ch.swap ? sa : sb;
    g.K = (int)K;
    g.num_kb = (int)((K + BLOCK_K - 1) / BLOCK_K);
    g.splits = ch.splits;
    g.segment = split_segment(K);
    g.p_tiles = (g.p.rows + BLOCK_M - 1) / BLOCK_M;
    g.q_tiles = (g.q.rows + ch.bn - 1) / ch.bn;
    g.c = c;
    g.c_p = ch.swap ? 1 : N;
    g.c_q = ch.swap ? N : 1;
    g.c_batch = M * N;
    g.bias = bias;
    g.bias_p = ch.swap;
    g.act = act;
    g.dev_status = dev_status;
    ++*launches;
    return ch.bn == 32 ? launch_instance<32>(g, ch.tiles, s) : launch_instance<64>(g, ch.tiles, s);
}

}  // namespace tfjsb
