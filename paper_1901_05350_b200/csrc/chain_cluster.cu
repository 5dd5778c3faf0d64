// The layers of a small model as one kernel: a cluster of thread blocks takes an image from the first convolution to the
// class probabilities.
//
// A MobileNet of 14 MFLOP an image is not bound by arithmetic or by bytes but by its chain of 30 kernels, each of which
// costs about 4 us from its start to its results being visible however little it does.  Here a step between two layers
// is a hardware cluster barrier (well under 1 us), the next layer's filter is on its way to shared memory before the
// barrier, and a depthwise layer and the pointwise layer after it are one step: a block computes the depthwise result of
// its pixels for all channels into shared memory, and multiplies it with its columns of the pointwise filter.  Where a
// layer has fewer pixels than the cluster has blocks' worth, the columns are divided and the depthwise part is repeated.
// Images are independent, so a batch is spread over clusters, and the cluster gets smaller as the batch grows: 16 blocks
// for one image, down to single blocks (whose steps are separated by __syncthreads alone) for more than a hundred.
//
// The products are m16n8k8 TF32 mma.sync: a step multiplies 16 to 256 rows, most often 16 or 32, and needs its result in
// registers at once.  A tcgen05 tile has at least 64 rows and a round trip through tensor memory that costs as much as the
// whole step here; large models, where the tensor core's rate counts, stay with the separate kernels.  Measured, whole model in the kernels
// of the layers and here: width 0.25, 128 x 128, 1 image 102 and 56 us, 8 images 113 and 71, 32 images 132 and 97; 224 x 224,
// 1 image 112 and 91; width 0.5, 128 x 128, 1 image 112 and 81.  And where it loses and is not chosen: width 0.5, 224 x 224,
// 1 image 120 and 161; width 1, 96 x 96, 120 and 150; width 0.25, 160 x 160, 64 images 186 and 241.
//
// What bounds a step of about 5500 clocks (16 blocks, one image): its stores' way to L2 before the barrier (1500), the
// latency of the depthwise windows (1300), of 4 to 8 dependent products (900), of the epilogue (1000) and the fetch of
// instructions that run once.  The copying warp needs whole chunks in one copy: row by row, 128 copies of 128 bytes took
// 7700 clocks and held the barriers up.
//
// Intermediate tensors are in a workspace of the cluster's own and stay in L2; each has a buffer of its own whose border of
// zeros, set once, is the next layer's padding.  Layer outputs that can be read after the run are also written to the
// buffers where the separate kernels leave them (an instance of its own: the code costs a small model 2 us of 55).
// Convolutions multiply as the separate kernels do: TF32 operands (exact for bfloat16 values), fp32 sums in another order.
// The dense layer multiplies fp32 values on the CUDA cores.  In the bfloat16 storage mode every stored value and the depthwise
// result are rounded to bfloat16 at the same places.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "chain_copy.cuh"
#include "common.cuh"
#include "ptx_sm100.cuh"

namespace tfjsb {

namespace {

constexpr int THREADS = 256, WARPS = THREADS / 32;  // and one warp that copies the filters
constexpr int D_FLOATS = 20480;    // depthwise results of a unit's pixels, [pixel][C + 4]
constexpr int F_FLOATS = 10240;    // the depthwise filter and bias, [10][C]
constexpr int W_FLOATS = 8192;     // a chunk of filter rows, then the tile's bias; twice
constexpr int RED_FLOATS = 8192;   // partial sums where the warps divide K
constexpr int SMEM_BYTES = (D_FLOATS + F_FLOATS + 2 * W_FLOATS + RED_FLOATS) * 4 + CHAIN_MAX_OPS * (int)sizeof(ChainOp);

// The computing threads of the block.
__device__ __forceinline__ void block_sync() { asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory"); }
// Every thread of the cluster, the copying warps included.  The aligned forms want the warp's threads together: a warp that
// comes out of a wait or of one thread's work executes __syncwarp() first.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
    cluster_arrive();
    cluster_wait();
}
// Activations are written by other blocks of the cluster during the kernel: ld_global, never the read-only path.
// `bytes` (a multiple of 16) to shared memory, counted on `bar`.
__device__ __forceinline__ void bulk_copy(uint32_t dst, const float* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float round_bf16(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
// relu and relu6 as bounds (none: infinite ones); NaN stays NaN
__device__ __forceinline__ float bounded(float v, float lo, float hi) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;\n\tmin.NaN.f32 %0, %0, %3;" : "=&f"(r) : "f"(v), "f"(lo), "f"(hi));
    return r;
}
// n / d from ceil(2^32 / d): exact while n d < 2^32
__device__ __forceinline__ int div_by(int n, unsigned int magic) { return magic ? (int)__umulhi((unsigned)n, magic) : n; }

// Waits of a converged warp, which comes out of them converged (mma.sync, bar.sync and barrier.cluster follow); after the
// limit the kernel notes it and the warp goes on without waiting, to the kernel's end.  Threads that spin and leave on their
// own would leave at different times, and only some of them on giving up.
struct Waiter {
    unsigned int* dev_status;
    bool off;  // the same in all threads of the warp
    __device__ __forceinline__ void wait(uint32_t bar, uint32_t parity) {
        if (off || __all_sync(0xffffffffu, ptx::mbar_try_wait(bar, parity))) return;
        const unsigned long long t0 = ptx::global_ns();
        while (!__all_sync(0xffffffffu, ptx::mbar_try_wait(bar, parity)))
            if (__any_sync(0xffffffffu, ptx::global_ns() - t0 > ptx::WAIT_LIMIT_NS)) {
                if ((threadIdx.x & 31) == 0) atomicOr(dev_status, DEV_STATUS_TIMEOUT_PRODUCER);
                off = true;
                return;
            }
    }
};

// The copying warp's side of chain_copy_filters.
struct CopyPort {
    unsigned int* dev_status;
    uint32_t bars, w_sm, f_sm;
    int rank;
    __device__ __forceinline__ bool wants(const ChainOp& o) const { return o.kind == CHAIN_BLOCK && rank < o.units; }
    __device__ __forceinline__ int group(const ChainOp& o, int u) const { return u - div_by(u, o.by_groups) * o.groups; }
    __device__ __forceinline__ bool wait(int bar, uint32_t parity) const {
        Waiter w{dev_status, false};  // of this one wait: one that gave up says nothing about the next
        w.wait(bars + 8 * bar, parity);
        return !w.off;
    }
    __device__ __forceinline__ void copy_filter(const ChainOp& o) const {
        if ((threadIdx.x & 31) == 0) {
            ptx::mbar_arrive_expect_tx(bars + 8 * CHAIN_F_FULL, 10 * o.C * 4);
            bulk_copy(f_sm, o.f1, 10 * o.C * 4, bars + 8 * CHAIN_F_FULL);
        }
    }
    __device__ __forceinline__ void copy_chunk(const ChainOp& o, int64_t from, int buf) const {
        if ((threadIdx.x & 31) == 0) {
            ptx::mbar_arrive_expect_tx(bars + 8 * (CHAIN_FULL0 + buf), o.chunk_floats * 4);
            bulk_copy(w_sm + (uint32_t)buf * W_FLOATS * 4, o.f2 + from, o.chunk_floats * 4, bars + 8 * (CHAIN_FULL0 + buf));
        }
    }
    __device__ __forceinline__ void converge() const { __syncwarp(); }
    __device__ __forceinline__ void meet() const { cluster_sync(); }
};

struct Pipeline {
    Waiter waiter;
    int chunk;  // the chunk that is waited for next
    uint32_t full, empty;
    // This warp has read a buffer (or the depthwise filter).  A warp that gave up waiting hands nothing back: its buffer may
    // have a copy in flight, and the copying warp, whose wait then gives up too, must not arm that barrier again.
    __device__ __forceinline__ void hand_back(uint32_t bar) const {
        if ((threadIdx.x & 31) == 0 && !waiter.off) ptx::mbar_arrive(bar);
    }
};

__device__ __forceinline__ void store_pair(int bf16, float* out, int at, float x, float y) {
    if (bf16) *reinterpret_cast<__nv_bfloat162*>(reinterpret_cast<__nv_bfloat16*>(out) + at) = __floats2bfloat162_rn(x, y);
    else *reinterpret_cast<float2*>(out + at) = make_float2(x, y);
}
__device__ __forceinline__ void store2(const ChainOp& o, int bf16, float* out, int at, float x, float y) {
    x = bounded(x, o.lo2, o.hi2);
    y = bounded(y, o.lo2, o.hi2);
    if (o.round2) { x = round_bf16(x); y = round_bf16(y); }
    store_pair(bf16, out, at, x, y);
}
// Where pixel p of a layer's output is: rows of out_row floats, the origin inside the next layer's padding.
__device__ __forceinline__ int out_at(const ChainOp& o, int p) {
    const int oy = div_by(p, o.by_wo);
    return o.out_origin + oy * o.out_row + (p - oy * o.Wo) * o.Co;
}

// Element `at` of a tensor that is read after the run.
__device__ __forceinline__ float* also_at(float* base, int bf16, int64_t at) {
    return bf16 ? reinterpret_cast<float*>(reinterpret_cast<__nv_bfloat16*>(base) + at) : base + at;
}

// What a thread does in a block's units, worked out while the cluster meets.
struct BlockWork {
    bool active;
    int split, m_base, n_base;  // product: share of K, first row and column of the warp's tile
    int q, first;               // depthwise: channel quad, first pixel (strip)
    int src;                    // offset of the first pixel's window in the input
};
__device__ __forceinline__ BlockWork block_work(const ChainOp& o, int rank) {
    BlockWork w;
    const int warp = threadIdx.x >> 5;
    w.split = div_by(warp, o.by_tasks);
    const int task = warp - w.split * o.tasks, task_row = div_by(task, o.by_task_n);
    w.active = w.split < o.k_splits;
    w.m_base = task_row * o.task_rows;
    w.n_base = (task - task_row * o.task_n) * o.task_cols;
    const int lane_px = div_by(threadIdx.x, o.by_quads);
    w.q = threadIdx.x - lane_px * (o.C >> 2);
    w.first = lane_px < o.lanes ? lane_px * o.strip : 1 << 30;
    const int p = div_by(rank, o.by_groups) * o.pixels + lane_px * o.strip, oy = div_by(p, o.by_wo);
    w.src = oy * o.sh * o.in_row + (p - oy * o.Wo) * o.sw * o.C + 4 * w.q;
    return w;
}

// The product of a unit: D [P][C] times this unit's columns of the filter.
template <int MT, int NT, bool KEEP>
__device__ __forceinline__ void block_columns(const ChainOp& o, const BlockWork& work, int u, int p0, int64_t image, float* out, const float* d_sm,
                                              const float* w_sm, float* red, Pipeline& pipe) {
    const int tid = threadIdx.x, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int ldd = o.C + 4, ldw = o.w_stride, splits = o.k_splits, tile_cols = o.tile_cols, Co = o.Co;
    const int split = work.split, m_base = work.m_base, n_base = work.n_base;
    const bool active = work.active;
    const int col0 = (u - div_by(u, o.by_groups) * o.groups) * o.group_cols, col_end = min(Co, col0 + o.group_cols);
    const int M = o.Ho * o.Wo;
    float* also = KEEP && o.also ? also_at(o.also, o.also_bf16, image * M * Co) : nullptr;
    for (int n0 = col0; n0 < col_end; n0 += tile_cols) {
        float acc[MT][NT][4];
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
        const int n_chunks = o.n_chunks;
        for (int kc = 0; kc < n_chunks; ++kc) {
            const int buf = pipe.chunk & 1;
            pipe.waiter.wait(pipe.full + 8 * buf, (pipe.chunk >> 1) & 1);
            ++pipe.chunk;
            if (active) {
                const int k0 = kc * o.chunk_rows, steps = min(o.chunk_rows, o.C - k0) >> 3;
                const float* ap = d_sm + (m_base + g) * ldd + k0 + split * 8 + t;
                const float* bp = w_sm + buf * W_FLOATS + (split * 8 + t) * ldw + n_base + g;
                const int a_step = splits * 8, b_step = splits * 8 * ldw;
#pragma unroll 4
                for (int ks = split; ks < steps; ks += splits) {
                    uint32_t af[MT][4], bf[NT][2];
#pragma unroll
                    for (int i = 0; i < MT; ++i) {
                        af[i][0] = __float_as_uint(ap[(16 * i) * ldd]);
                        af[i][1] = __float_as_uint(ap[(16 * i + 8) * ldd]);
                        af[i][2] = __float_as_uint(ap[(16 * i) * ldd + 4]);
                        af[i][3] = __float_as_uint(ap[(16 * i + 8) * ldd + 4]);
                    }
#pragma unroll
                    for (int j = 0; j < NT; ++j) {
                        bf[j][0] = __float_as_uint(bp[8 * j]);
                        bf[j][1] = __float_as_uint(bp[4 * ldw + 8 * j]);
                    }
#pragma unroll
                    for (int i = 0; i < MT; ++i)
#pragma unroll
                        for (int j = 0; j < NT; ++j) mma_tf32(acc[i][j], af[i], bf[j][0], bf[j][1]);
                    ap += a_step;
                    bp += b_step;
                }
            }
            if (kc + 1 < n_chunks) {
                __syncwarp();
                pipe.hand_back(pipe.empty + 8 * buf);
            }
        }
        const int buf = (pipe.chunk & 1) ^ 1;  // of the last chunk: handed back when its bias has been read
        const float* bias = w_sm + buf * W_FLOATS + o.chunk_floats - 64;
        if (splits == 1) {
            if (active) {
                int at[MT][2];
#pragma unroll
                for (int i = 0; i < MT; ++i)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int p = p0 + m_base + 16 * i + 8 * h + g;
                        at[i][h] = p < M ? out_at(o, p) : -1;
                    }
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const int c = n_base + 8 * j + 2 * t;
                    if (n0 + c >= Co) continue;
                    const float2 b = *reinterpret_cast<const float2*>(bias + c);
#pragma unroll
                    for (int i = 0; i < MT; ++i)
#pragma unroll
                        for (int h = 0; h < 2; ++h)
                            if (at[i][h] >= 0) {
                                store2(o, 0, out, at[i][h] + n0 + c, acc[i][j][2 * h] + b.x, acc[i][j][2 * h + 1] + b.y);
                                if (KEEP && also)
                                    store2(o, o.also_bf16, also, (p0 + m_base + 16 * i + 8 * h + g) * Co + n0 + c, acc[i][j][2 * h] + b.x,
                                           acc[i][j][2 * h + 1] + b.y);
                            }
                }
            }
        } else {
            // the warps' shares of K, added in order
            const int plane = o.pixels * tile_cols;
            if (n0 != col0) block_sync();  // the tile before is done with red (a new unit and a new layer start after a barrier)
            if (active) {
                float* r = red + split * plane;
#pragma unroll
                for (int i = 0; i < MT; ++i)
#pragma unroll
                    for (int j = 0; j < NT; ++j)
#pragma unroll
                        for (int h = 0; h < 2; ++h)
                            *reinterpret_cast<float2*>(r + (m_base + 16 * i + 8 * h + g) * tile_cols + n_base + 8 * j + 2 * t) =
                                make_float2(acc[i][j][2 * h], acc[i][j][2 * h + 1]);
            }
            block_sync();
            for (int j = tid; j < plane / 2; j += THREADS) {
                const int p = div_by(j >> 1, o.by_pieces), c = 2 * j - p * tile_cols;
                float2 s = *reinterpret_cast<const float2*>(bias + c);
                for (int k = 0; k < splits; ++k) {
                    const float2 v = *reinterpret_cast<const float2*>(red + k * plane + 2 * j);
                    s.x += v.x; s.y += v.y;
                }
                if (p0 + p < M && n0 + c < Co) {
                    store2(o, 0, out, out_at(o, p0 + p) + n0 + c, s.x, s.y);
                    if (KEEP && also) store2(o, o.also_bf16, also, (p0 + p) * Co + n0 + c, s.x, s.y);
                }
            }
        }
        __syncwarp();
        pipe.hand_back(pipe.empty + 8 * buf);
    }
}

// Depthwise 3x3 of a unit's pixels, all channels, into shared memory.  The input has its padding around it, so no tap is
// tested.  R > 1 (stride 1, no dilation, Wo a multiple of R): R neighbouring pixels share their 3 (R + 2) loads.
template <int R, bool KEEP>
__device__ __forceinline__ void block_depthwise(const ChainOp& o, const BlockWork& work, bool first_unit, int64_t image, const float* f_sm, const float* in,
                                                int p0, float* d_sm) {
    const int C = o.C, quads = C >> 2, q = work.q, step = o.lanes * R;
    const int M = o.Ho * o.Wo, n = o.pixels, round = o.round1;
    const int in_row = o.in_row, tap_row = o.dh * in_row, tap_col = o.dw * C;
    const float lo = o.lo1, hi = o.hi1;
    const float4* f = reinterpret_cast<const float4*>(f_sm) + q;  // taps `quads` apart, then the bias
    for (int i = work.first; i < n; i += step) {
        float4 v[R];
        if (p0 + i < M) {
            int at = work.src;
            if (!first_unit || i != work.first) {
                const int p = p0 + i, oy = div_by(p, o.by_wo);
                at = oy * o.sh * in_row + (p - oy * o.Wo) * o.sw * C + 4 * q;
            }
            const float* src = in + at;
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = f[9 * quads];
            if (R == 1) {
                float4 x[9];
#pragma unroll
                for (int ky = 0; ky < 3; ++ky)
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx) x[3 * ky + kx] = ld_global4(src + ky * tap_row + kx * tap_col);
#pragma unroll
                for (int k = 0; k < 9; ++k) fma4_packed(v[0], x[k], f[k * quads]);
            } else {
#pragma unroll
                for (int ky = 0; ky < 3; ++ky) {
                    float4 x[R + 2];
#pragma unroll
                    for (int j = 0; j < R + 2; ++j) x[j] = ld_global4(src + ky * in_row + j * C);
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx) {
                        const float4 tap = f[(3 * ky + kx) * quads];
#pragma unroll
                        for (int r = 0; r < R; ++r) fma4_packed(v[r], x[r + kx], tap);
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                v[r].x = bounded(v[r].x, lo, hi); v[r].y = bounded(v[r].y, lo, hi);
                v[r].z = bounded(v[r].z, lo, hi); v[r].w = bounded(v[r].w, lo, hi);
                if (round) {
                    v[r].x = round_bf16(v[r].x); v[r].y = round_bf16(v[r].y);
                    v[r].z = round_bf16(v[r].z); v[r].w = round_bf16(v[r].w);
                }
                if (KEEP && o.also_dw) {  // (by every group of columns: the same values)
                    float* to = also_at(o.also_dw, o.also_dw_bf16, image * M * C);
                    store_pair(o.also_dw_bf16, to, (p0 + i + r) * C + 4 * q, v[r].x, v[r].y);
                    store_pair(o.also_dw_bf16, to, (p0 + i + r) * C + 4 * q + 2, v[r].z, v[r].w);
                }
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) *reinterpret_cast<float4*>(d_sm + (i + r) * (C + 4) + 4 * q) = v[r];
    }
}

// First layer: 3x3 window of a 3-channel image.  The input rows of `pixels` output rows go to shared memory with zeros
// around them; a window row is then 9 neighbouring floats (without dilation), and a lane's fragments of 16 windows are at
// eight fixed offsets from its pixels.
__device__ __forceinline__ void stem(const ChainOp& o, const float* in, float* out, float* x_sm, float* f_sm, int rank, int cs) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int Co = o.Co, ldf = o.w_stride, row = o.in_row;
    int off[8];  // k = t, t + 4, ... ; 27 and above have a zero filter and read nothing
#pragma unroll
    for (int s = 0; s < 8; ++s) {
        const int k = 4 * s + t, ky = k / 9, kx = (k - 9 * ky) / 3;
        off[s] = k < 27 ? ky * o.dh * row + kx * o.dw * 3 + k % 3 : -1;
    }
    const int W3 = o.W * 3;
    for (int u = rank; u < o.units; u += cs) {
        const int oy0 = u * o.pixels, rows = min(o.pixels, o.Ho - oy0), in_rows = (rows - 1) * o.sh + 2 * o.dh + 1;
        const int iy0 = oy0 * o.sh - o.pt, shift = (o.pl * 3 + 3) & ~3;  // the image's rows start on 16 bytes
        if (u != rank) block_sync();
        const uint32_t dst = ptx::smem_u32(x_sm);
        const int H = o.H;
        const unsigned int by_row = o.by_quads;
        if (W3 % 4 == 0) {
#pragma unroll 4
            for (int j = tid; j < in_rows * (row >> 2); j += THREADS) {  // zeros where there is no pixel
                const int r = div_by(j, by_row), c = 4 * (j - r * (row >> 2)) - shift, iy = iy0 + r;
                const bool ok = iy >= 0 && iy < H && c >= 0 && c < W3;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + 16 * j), "l"(ok ? in + iy * W3 + c : in), "r"(ok ? 16 : 0) : "memory");
            }
        } else {
#pragma unroll 4
            for (int j = tid; j < in_rows * row; j += THREADS) {
                const int r = div_by(j >> 2, by_row), c = j - r * row - shift, iy = iy0 + r;
                const bool ok = iy >= 0 && iy < H && c >= 0 && c < W3;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 4 * j), "l"(ok ? in + iy * W3 + c : in), "r"(ok ? 4 : 0) : "memory");
            }
        }
        if (u == rank) {
            for (int j = tid; j < 32 * ldf; j += THREADS) {
                const int k = div_by(j, o.by_pieces), c = j - k * ldf;
                f_sm[j] = k < 27 && c < Co ? load_fixed(o.f1 + k * Co + c) : 0.f;
            }
            if (tid < Co) f_sm[32 * ldf + tid] = o.b1 ? load_fixed(o.b1 + tid) : 0.f;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        block_sync();
        const int pixels = rows * o.Wo;
        for (int m = warp * 16; m < pixels; m += WARPS * 16) {
            uint32_t a[4][4];
            int at[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int p = m + 8 * h + g, oy = div_by(p, o.by_wo), ox = p - oy * o.Wo;
                const bool ok = p < pixels;
                const float* src = x_sm + shift - o.pl * 3 + (ok ? oy * o.sh * row + ox * o.sw * 3 : 0);
                at[h] = ok ? out_at(o, oy0 * o.Wo + p) : -1;
#pragma unroll
                for (int s = 0; s < 8; ++s) {
                    const float x = off[s] >= 0 ? src[off[s]] : 0.f;
                    a[s >> 1][h + 2 * (s & 1)] = __float_as_uint(o.round1 ? round_bf16(x) : x);
                }
            }
            for (int n = 0; n < Co; n += 8) {
                float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    mma_tf32(acc, a[ks], __float_as_uint(f_sm[(8 * ks + t) * ldf + n + g]), __float_as_uint(f_sm[(8 * ks + t + 4) * ldf + n + g]));
                const float2 b = *reinterpret_cast<const float2*>(f_sm + 32 * ldf + n + 2 * t);
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (at[h] >= 0) store2(o, 0, out, at[h] + n + 2 * t, acc[2 * h] + b.x, acc[2 * h + 1] + b.y);
            }
        }
    }
}

// Global average: a warp per 4 channels, its lanes over the pixels.
__device__ __forceinline__ void pool(const ChainOp& o, int64_t image, const float* in, float* out, int rank, int cs) {
    const int lane = threadIdx.x & 31, M = o.H * o.W;
    for (int q = rank * WARPS + (threadIdx.x >> 5); q < (o.C >> 2); q += cs * WARPS) {
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int p = lane; p < M; p += 32) {
            const float4 v = ld_global4(in + p * o.C + 4 * q);
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            s.x += __shfl_xor_sync(0xffffffffu, s.x, d); s.y += __shfl_xor_sync(0xffffffffu, s.y, d);
            s.z += __shfl_xor_sync(0xffffffffu, s.z, d); s.w += __shfl_xor_sync(0xffffffffu, s.w, d);
        }
        if (lane == 0) {
            const float k = 1.f / (float)M;
            store2(o, o.store_bf16, out, 4 * q, s.x * k, s.y * k);
            store2(o, o.store_bf16, out, 4 * q + 2, s.z * k, s.w * k);
            if (o.also) {
                float* row = also_at(o.also, o.also_bf16, image * o.Co);
                store2(o, o.also_bf16, row, 4 * q, s.x * k, s.y * k);
                store2(o, o.also_bf16, row, 4 * q + 2, s.z * k, s.w * k);
            }
        }
    }
}

// Dense layer of one row: 64 columns at a time, shares of K, added in order.  The first filter rows of the block's first
// columns are fetched while the cluster meets.
constexpr int DENSE_SHARES = THREADS / 16, DENSE_AHEAD = 16;
__device__ __forceinline__ void load_dense(const ChainOp& o, float4 (&w)[DENSE_AHEAD], int n0, int k0) {
    // past the end: some other value, multiplied by zero or not stored (a branch around a load would wait for it)
    const float* src = o.f1 + min(n0 + 4 * (int)(threadIdx.x & 15), o.Co - 4);
    const int share = threadIdx.x >> 4, last = o.C - 1, Co = o.Co;
#pragma unroll
    for (int j = 0; j < DENSE_AHEAD; ++j) w[j] = load_fixed(reinterpret_cast<const float4*>(src + (int64_t)min(k0 + share + j * DENSE_SHARES, last) * Co));
}
__device__ __forceinline__ void dense(const ChainOp& o, float4 (&w)[DENSE_AHEAD], int64_t image, const float* in, float* out, float* x_sm, float* red,
                                      int rank, int cs) {
    const int q = threadIdx.x & 15, share = threadIdx.x >> 4, Co = o.Co, C = o.C;
    const int padded = (C + DENSE_AHEAD * DENSE_SHARES - 1) / (DENSE_AHEAD * DENSE_SHARES) * (DENSE_AHEAD * DENSE_SHARES);
    for (int k = 4 * threadIdx.x; k < padded; k += 4 * THREADS)
        *reinterpret_cast<float4*>(x_sm + k) = k < C ? ld_global4(in + k) : make_float4(0.f, 0.f, 0.f, 0.f);
    block_sync();
    for (int n0 = rank * 64; n0 < Co; n0 += cs * 64) {
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k0 = 0; k0 < C; k0 += DENSE_AHEAD * DENSE_SHARES) {
            if (k0 || n0 != rank * 64) load_dense(o, w, n0, k0);
#pragma unroll
            for (int j = 0; j < DENSE_AHEAD; ++j) {
                const int k = k0 + share + j * DENSE_SHARES;
                const float x = x_sm[k];
                fma4_packed(s, make_float4(x, x, x, x), w[j]);
            }
        }
        *reinterpret_cast<float4*>(red + share * 64 + 4 * q) = s;
        block_sync();
        if (threadIdx.x < 64 && n0 + (int)threadIdx.x < Co) {
            float v = o.b1 ? load_fixed(o.b1 + n0 + threadIdx.x) : 0.f;
#pragma unroll
            for (int k = 0; k < DENSE_SHARES; ++k) v += red[k * 64 + threadIdx.x];
            v = bounded(v, o.lo2, o.hi2);
            out[n0 + threadIdx.x] = v;
            if (o.also) o.also[image * Co + n0 + threadIdx.x] = v;
        }
        block_sync();
    }
}

// Softmax of one row by the cluster's first block.
__device__ __forceinline__ void softmax(const ChainOp& o, const float* in, float* out, float* red, int rank) {
    if (rank != 0) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int HELD = 4;  // values a thread keeps; more are read again
    float x[HELD], top = -INFINITY;
#pragma unroll
    for (int k = 0; k < HELD; ++k) {
        const int j = threadIdx.x + k * THREADS;
        x[k] = j < o.Co ? ld_global(in + j) : -INFINITY;
    }
#pragma unroll
    for (int k = 0; k < HELD; ++k) top = fmaxf(top, x[k]);
    for (int j = threadIdx.x + HELD * THREADS; j < o.Co; j += THREADS) top = fmaxf(top, ld_global(in + j));
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, d));
    if (lane == 0) red[warp] = top;
    block_sync();
    top = red[0];
#pragma unroll
    for (int k = 1; k < WARPS; ++k) top = fmaxf(top, red[k]);
    float sum = 0.f;
#pragma unroll
    for (int k = 0; k < HELD; ++k) {
        x[k] = (int)threadIdx.x + k * THREADS < o.Co ? expf(x[k] - top) : 0.f;
        sum += x[k];
    }
    for (int j = threadIdx.x + HELD * THREADS; j < o.Co; j += THREADS) sum += expf(ld_global(in + j) - top);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
    if (lane == 0) red[WARPS + warp] = sum;
    block_sync();
    sum = 0.f;
#pragma unroll
    for (int k = 0; k < WARPS; ++k) sum += red[WARPS + k];
#pragma unroll
    for (int k = 0; k < HELD; ++k) {
        const int j = threadIdx.x + k * THREADS;
        if (j < o.Co) out[j] = x[k] / sum;
    }
    for (int j = threadIdx.x + HELD * THREADS; j < o.Co; j += THREADS) out[j] = expf(ld_global(in + j) - top) / sum;
}

// The end of the layer before.
__device__ __forceinline__ void meet(int cs, bool met) {
    if (met) return;
    __syncwarp();
    if (cs > 1) cluster_wait();
    else block_sync();
}

// KEEP: a block's own outputs are wanted as well (the model ends soon after it).  An instance of its own: every block's code
// would be longer for it, and a step is bound by the fetch of instructions that run once (57.3 us instead of 55.3 for the
// model of width 0.25 on one 128 x 128 image).
template <bool KEEP>
__global__ void __launch_bounds__(THREADS + 32, 1) chain_kernel(const __grid_constant__ ChainArgs a) {
    extern __shared__ __align__(16) float sm[];
    __shared__ __align__(8) unsigned long long bars[CHAIN_BARS];
    float* d_sm = sm;
    float* f_sm = sm + D_FLOATS;
    float* w_sm = f_sm + F_FLOATS;
    float* red = w_sm + 2 * W_FLOATS;
    ChainOp* ops = reinterpret_cast<ChainOp*>(red + RED_FLOATS);  // dynamically indexed constants are slower to reach
    for (int j = threadIdx.x; j < (int)(a.n_ops * sizeof(ChainOp) / 4); j += THREADS + 32)
        reinterpret_cast<uint32_t*>(ops)[j] = reinterpret_cast<const uint32_t*>(a.ops)[j];
    const uint32_t bar0 = ptx::smem_u32(bars), full = bar0 + 8 * CHAIN_FULL0, empty = bar0 + 8 * CHAIN_EMPTY0;
    const uint32_t f_full = bar0 + 8 * CHAIN_F_FULL, f_empty = bar0 + 8 * CHAIN_F_EMPTY;
    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(full + 8 * b, 1);
            ptx::mbar_init(empty + 8 * b, WARPS);
        }
        ptx::mbar_init(f_full, 1);
        ptx::mbar_init(f_empty, WARPS);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int n_ops = a.n_ops;
    const int cs = a.cluster_size, rank = (int)blockIdx.x % cs, cluster = (int)blockIdx.x / cs, clusters = (int)gridDim.x / cs;
    const int images = (int)((a.images - cluster + clusters - 1) / clusters);
    ptx::pdl_launch_dependents();
    if (threadIdx.x >= THREADS) {
        CopyPort port{a.dev_status, bar0, ptx::smem_u32(w_sm), ptx::smem_u32(f_sm), rank};
        chain_copy_filters(ops, n_ops, rank, cs, images, port);
        return;
    }
    Pipeline pipe{Waiter{a.dev_status, false}, 0, full, empty};
    ptx::pdl_wait();
    int blocks = 0;
    bool met = true;  // false after a layer, until the next one's meet()
    float* ws = a.workspace + (int64_t)cluster * a.cluster_elems;
    for (int64_t n = cluster; n < a.images; n += clusters) {
        const float* in = a.input + n * a.in_elems;
        for (int i = 0; i < n_ops; ++i) {
            const ChainOp& o = ops[i];
            float* out = ws + o.out_buffer;
            if (i + 1 == n_ops)
                out = o.store_bf16 ? reinterpret_cast<float*>(reinterpret_cast<__nv_bfloat16*>(a.output) + n * a.out_elems) : a.output + n * a.out_elems;
            // what does not depend on the layer before comes first, then its output is visible to the cluster, and its
            // input and shared memory are free
            if (o.kind == CHAIN_BLOCK) {
                const BlockWork work = block_work(o, rank);
                if (rank < o.units) pipe.waiter.wait(f_full, blocks++ & 1);
                meet(cs, met);
                for (int u = rank; u < o.units; u += cs) {
                    const int p0 = div_by(u, o.by_groups) * o.pixels;
                    if (u != rank) block_sync();  // the unit before is done with D and red
                    if (o.strip == 4) block_depthwise<4, KEEP>(o, work, u == rank, n, f_sm, in, p0, d_sm);
                    else if (o.strip == 2) block_depthwise<2, KEEP>(o, work, u == rank, n, f_sm, in, p0, d_sm);
                    else block_depthwise<1, KEEP>(o, work, u == rank, n, f_sm, in, p0, d_sm);
                    block_sync();
                    if (u + cs >= o.units) pipe.hand_back(f_empty);
                    const int v = o.variant;  // tests, not a jump table in constant memory
                    if (v == 0) block_columns<1, 1, KEEP>(o, work, u, p0, n, out, d_sm, w_sm, red, pipe);
                    else if (v == 1) block_columns<1, 2, KEEP>(o, work, u, p0, n, out, d_sm, w_sm, red, pipe);
                    else if (v == 2) block_columns<1, 4, KEEP>(o, work, u, p0, n, out, d_sm, w_sm, red, pipe);
                    else if (v == 3) block_columns<2, 2, KEEP>(o, work, u, p0, n, out, d_sm, w_sm, red, pipe);
                    else block_columns<2, 4, KEEP>(o, work, u, p0, n, out, d_sm, w_sm, red, pipe);
                }
            } else if (o.kind == CHAIN_STEM) {
                meet(cs, met);
                stem(o, in, out, d_sm, red, rank, cs);
            } else if (o.kind == CHAIN_POOL) {
                meet(cs, met);
                pool(o, n, in, out, rank, cs);
            } else if (o.kind == CHAIN_DENSE) {
                float4 w[DENSE_AHEAD];
                load_dense(o, w, rank * 64, 0);
                meet(cs, met);
                dense(o, w, n, in, out, d_sm, red, rank, cs);
            } else {
                meet(cs, met);
                softmax(o, in, out, red, rank);
            }
            __syncwarp();
            if (cs > 1) cluster_arrive();
            met = false;
            in = out;
        }
    }
    if (cs > 1) cluster_wait();
}

// A block's filters in the order and layout in which the copying warp wants them: the depthwise filter and its bias
// [10][C], then for every group, column tile and chunk the chunk's rows [chunk_rows][w_stride] and the tile's bias [64].
__global__ void pack_chain_kernel(const ChainOp o, float* __restrict__ dst) {
    const int64_t first = 10 * (int64_t)o.C, total = first + (int64_t)o.groups * o.group_tiles * o.n_chunks * o.chunk_floats;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < total; j += (int64_t)gridDim.x * blockDim.x) {
        float v = 0.f;
        if (j < first) {
            if (j < 9 * (int64_t)o.C) v = o.f1[j];
            else if (o.b1) v = o.b1[j - 9 * (int64_t)o.C];
        } else {
            const int64_t chunk = (j - first) / o.chunk_floats;
            const int at = (int)((j - first) - chunk * o.chunk_floats);
            const int kc = (int)(chunk % o.n_chunks);
            const int64_t tile = chunk / o.n_chunks;  // group * group_tiles + column tile
            const int64_t col0 = (tile / o.group_tiles) * o.group_cols + (tile % o.group_tiles) * o.tile_cols;
            const int r = at / o.w_stride, body = o.chunk_rows * o.w_stride;
            const int c = at < body ? at - r * o.w_stride : at - body, k = kc * o.chunk_rows + r;
            if (c < o.tile_cols && col0 + c < o.Co) {
                if (at < body) v = r < o.chunk_rows && k < o.C ? o.f2[(int64_t)k * o.Co + col0 + c] : 0.f;
                else v = o.b2 ? o.b2[col0 + c] : 0.f;
            }
        }
        dst[j] = v;
    }
}

constexpr int kVariantM[5] = {1, 1, 1, 2, 2}, kVariantN[5] = {1, 2, 4, 2, 4};

int ceil_div(int a, int b) { return (a + b - 1) / b; }
unsigned int magic(int d) { return d <= 1 ? 0u : (unsigned int)((0x100000000ull + d - 1) / d); }
int padded_stride(int cols) { return cols % 16 == 0 ? cols + 8 : cols; }  // 8 or 24 modulo 32 words (tile_cols is a multiple of 8, not 32 k + 0)

// Clocks of a step on `cs` blocks, and the tile parameters that give them.
double tune_block(ChainOp& o, int cs) {
    const int M = o.Ho * o.Wo, K = o.C, N = o.Co, quads = K / 4, lanes = THREADS / quads;
    double best = 1e30;
    ChainOp pick = o;
    for (int P = 16; P <= 256; P *= 2) {
        if (P > 16 && P / 2 >= M) break;
        if (P * (K + 4) > D_FLOATS) break;
        const int row_tiles = ceil_div(M, P);
        for (int G = 1; G <= 16; G *= 2) {
            if (G > 1 && row_tiles * (G / 2) >= cs) break;
            for (int v = 0; v < 5; ++v) {
                const int MT = kVariantM[v], NT = kVariantN[v];
                if (P % (16 * MT)) continue;
                const int share = ceil_div(ceil_div(N, G), 8 * NT) * 8 * NT;  // columns of a group
                for (int cols = 8 * NT; cols <= 64; cols += 8 * NT) {
                    if (cols > share) break;
                    const int task_n = cols / (8 * NT), tasks = (P / (16 * MT)) * task_n;
                    if (tasks > WARPS) break;
                    const int group_cols = ceil_div(share, cols) * cols, groups = ceil_div(N, group_cols);
                    const int stride = padded_stride(cols);
                    int chunk = std::min(K, (W_FLOATS - 64) / stride / 8 * 8);
                    const int chunks = ceil_div(K, chunk);
                    chunk = ceil_div(ceil_div(K, chunks), 8) * 8;
                    for (int S = 1; S * tasks <= WARPS; S *= 2) {
                        if (S > 1 && (S * P * cols > RED_FLOATS || S > chunk / 8)) break;
                        const int units = row_tiles * groups, rounds = ceil_div(units, cs), tiles = ceil_div(std::min(group_cols, N), cols);
                        const double steps = K / 8.0;
                        const double lds = tasks * steps * (4 * MT + 2 * NT), mma = tasks * steps * MT * NT * 2.0;
                        const double chain = steps / S * (80 + 4.0 * MT * NT);
                        const double copy = (double)K * cols * 4 / 40;
                        double tile = std::max(std::max(lds, mma), std::max(chain, copy)) + 100 + chunks * 60 + P * cols / 64.0;
                        if (S > 1) tile += 120 + 2.5 * S * P * cols / 64;
                        const double unit = 900 + ceil_div(P, lanes) * 650.0 + tiles * tile;
                        const double total = rounds * unit;
                        if (total < best) {
                            best = total;
                            pick.pixels = P; pick.groups = groups; pick.group_cols = group_cols; pick.tile_cols = cols;
                            pick.units = units; pick.variant = v; pick.k_splits = S; pick.w_stride = stride;
                            pick.chunk_rows = chunk; pick.n_chunks = chunks; pick.tasks = tasks; pick.task_n = task_n; pick.task_rows = 16 * MT; pick.task_cols = 8 * NT;
                        }
                    }
                }
            }
        }
    }
    o = pick;
    o.lanes = lanes;
    o.strip = 1;
    if (o.sh == 1 && o.sw == 1 && o.dh == 1 && o.dw == 1)
        for (int r = 2; r <= 4; r *= 2)
            if (o.Wo % r == 0 && o.pixels * quads / r >= THREADS) o.strip = r;
    o.group_tiles = o.group_cols / o.tile_cols;
    o.chunk_floats = o.chunk_rows * o.w_stride + 64;
    o.by_groups = magic(o.groups);
    o.by_pieces = magic(o.tile_cols / 4);
    o.by_tasks = magic(o.tasks);
    o.by_task_n = magic(o.task_n);
    return best;
}

bool tune_stem(ChainOp& o, int cs) {
    // whole output rows whose input rows fit, no more than an even share of the cluster
    o.in_row = (std::max(((o.Wo - 1) * o.sw + 2 * o.dw + 1) * 3 + 3, (o.pl + o.W) * 3 + 3) + 3) / 4 * 4;
    int rows = 0;
    while (rows < ceil_div(o.Ho, cs) && ((int64_t)rows * o.sh + 2 * o.dh + 1) * o.in_row <= D_FLOATS) ++rows;
    if (!rows) return false;
    o.pixels = rows;
    o.units = ceil_div(o.Ho, rows);
    o.w_stride = padded_stride(o.Co);
    o.by_pieces = magic(o.w_stride);
    o.by_quads = magic(o.in_row / 4);
    return true;
}

double tune_op(ChainOp& o, int cs) {
    o.by_wo = magic(o.Wo);
    if (o.kind != CHAIN_STEM) o.by_quads = magic(o.C / 4);
    const double inf = INFINITY;
    o.lo1 = o.act1 == TFJSB_ACT_NONE ? -inf : 0; o.hi1 = o.act1 == TFJSB_ACT_RELU6 ? 6 : inf;
    o.lo2 = o.act2 == TFJSB_ACT_NONE ? -inf : 0; o.hi2 = o.act2 == TFJSB_ACT_RELU6 ? 6 : inf;
    switch (o.kind) {
        case CHAIN_STEM:
            if (!tune_stem(o, cs)) return 1e30;
            return ceil_div(o.units, cs) * (1500 + (o.pixels * o.sh + 2.0) * o.in_row / THREADS * 60 + o.pixels * o.Wo / 256.0 * (100 + o.Co / 8 * 80));
        case CHAIN_BLOCK: return tune_block(o, cs);
        case CHAIN_POOL: return 900 + std::ceil(o.C / 4.0 / (cs * WARPS)) * std::ceil(o.H * o.W / 32.0) * 500;
        case CHAIN_DENSE: return ceil_div(ceil_div(o.Co, 64), cs) * (400 + ceil_div(o.C, 256) * 900.0);
        default: return 1000;
    }
}

template <bool KEEP>
bool prepare_kernel() {
    return smem_attr_once(reinterpret_cast<const void*>(chain_kernel<KEEP>), SMEM_BYTES) == cudaSuccess &&
           cudaFuncSetAttribute(chain_kernel<KEEP>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
}

// How many clusters of `cs` blocks run at once; 0 where none can.
int max_clusters(int cs) {
    if (!prepare_kernel<false>() || !prepare_kernel<true>()) {
        (void)cudaGetLastError();
        return 0;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cs);
    cfg.blockDim = dim3(THREADS + 32);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, chain_kernel<false>, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return n;
}

}  // namespace

bool chain_stem_supported(const ConvGeom& g) {
    return g.fh == 3 && g.fw == 3 && g.C == 3 && g.Co % 8 == 0 && g.Co <= 128 && (int64_t)g.Ho * g.Wo * g.Wo <= 0x7fffffff &&
           (int64_t)(g.H + 2) * (g.W + 2) * 3 <= 0x7fffffff;
}
bool chain_block_supported(const ConvGeom& g, int64_t N) {
    return g.fh == 3 && g.fw == 3 && g.mult == 1 && g.C % 8 == 0 && g.C <= 4 * THREADS && N % 8 == 0 && N <= 4096 && (int64_t)g.Ho * g.Wo * g.Wo <= 0x7fffffff &&
           (int64_t)g.H * g.W * g.C <= 0x3fffffff && (int64_t)g.Ho * g.Wo * N <= 0x3fffffff;
}

int chain_plan(const ChainOp* ops, int n_ops, int64_t images, const double* rest, double separate, ChainPlan* plan) {
    if (n_ops < 1 || n_ops > CHAIN_MAX_OPS || images < 1) return 0;
    // every layer's output has a buffer of its own, with the zeros around it that the next layer's windows reach into
    ChainOp laid[CHAIN_MAX_OPS];
    int64_t elems = 0;
    for (int i = 0; i < n_ops; ++i) {
        ChainOp& o = laid[i] = ops[i];
        o.out_buffer = elems;
        o.out_origin = 0;
        o.out_row = o.Wo * o.Co;
        int64_t size = (int64_t)o.Ho * o.out_row;
        if (i + 1 < n_ops && ops[i + 1].kind == CHAIN_BLOCK) {
            const ChainOp& next = ops[i + 1];
            const int rows = std::max((next.Ho - 1) * next.sh + 2 * next.dh + 1, next.pt + o.Ho);
            const int cols = std::max((next.Wo - 1) * next.sw + 2 * next.dw + 1, next.pl + o.Wo);
            o.out_row = cols * o.Co;
            o.out_origin = next.pt * o.out_row + next.pl * o.Co;
            size = (int64_t)rows * o.out_row;
            if (size > 0x7fffffff) return 0;
        }
        if (i && o.kind == CHAIN_BLOCK) o.in_row = laid[i - 1].out_row;
        if (i + 1 < n_ops) elems += (size + 63) / 64 * 64;
    }
    double best = separate;
    int used = 0;
    for (int cs = 16; cs >= 1; cs /= 2) {
        // the clocks above are those of the arithmetic and the copies; measured, a step takes about twice as long (its
        // instructions are fetched and run once: 1.9 to 2.1 for clusters of 16 and 8, up to 2.4 for smaller ones)
        const double slower = cs >= 8 ? 2.1 : 2.4;
        ChainOp tuned[CHAIN_MAX_OPS];
        // first as if every SM were in a cluster, then, if that would win, with the clusters that there is room for
        int fit = current_sm_count() / cs;
        for (int pass = 0; pass < 2; ++pass) {
            if (pass && (fit = max_clusters(cs)) < 1) break;
            const int64_t clusters = std::min<int64_t>(fit, images), rounds = (images + clusters - 1) / clusters;
            double ns = 0, least = best;
            int ends = 0;
            for (int i = 0; i < n_ops && ns < least; ++i) {
                tuned[i] = laid[i];
                ns += (tune_op(tuned[i], cs) + (cs > 1 ? 700 : 100)) * rounds * slower / 1.9;
                if (rest[i] < 0 || ns + rest[i] >= least) continue;
                least = ns + rest[i];
                ends = i + 1;
            }
            if (!ends) break;
            if (!pass) continue;
            best = least;
            used = ends;
            ChainArgs& args = plan->args;
            std::copy(tuned, tuned + ends, args.ops);
            args.n_ops = ends;
            args.cluster_size = cs;
            args.images = images;
            args.cluster_elems = elems;  // the same for every length: the borders of zeros stay where they are
            plan->blocks = (int)clusters * cs;
        }
    }
    return used;
}

static int64_t packed_floats(const ChainOp& o) {
    if (o.kind != CHAIN_BLOCK) return 0;
    const int64_t n = 10 * (int64_t)o.C + (int64_t)o.groups * o.group_tiles * o.n_chunks * o.chunk_floats;
    return (n + 63) / 64 * 64;
}
int64_t chain_packed_floats(const ChainPlan& plan) {
    int64_t n = 0;
    for (int i = 0; i < plan.args.n_ops; ++i) n += packed_floats(plan.args.ops[i]);
    return n;
}
cudaError_t chain_pack(ChainPlan* plan, float* dst, cudaStream_t s, int64_t* launches) {
    for (int i = 0; i < plan->args.n_ops; ++i) {
        ChainOp& o = plan->args.ops[i];
        const int64_t n = packed_floats(o);
        if (!n) continue;
        pack_chain_kernel<<<(unsigned)std::min<int64_t>((n + 255) / 256, 1024), 256, 0, s>>>(o, dst);
        ++*launches;
        o.f1 = dst;
        o.f2 = dst + 10 * (int64_t)o.C;
        dst += n;
    }
    return cudaGetLastError();
}

cudaError_t launch_chain(const ChainPlan& plan, const float* input, float* output, unsigned int* dev_status, cudaStream_t s,
                         int64_t* launches) {
    ChainArgs args = plan.args;
    args.input = input;
    args.output = output;
    args.dev_status = dev_status;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)plan.blocks);
    cfg.blockDim = dim3(THREADS + 32);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)args.cluster_size;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g_launch_pdl ? 2 : 1;
    ++*launches;
    bool keep = false;
    for (int i = 0; i < args.n_ops; ++i) keep = keep || (args.ops[i].kind == CHAIN_BLOCK && (args.ops[i].also || args.ops[i].also_dw));
    return cudaLaunchKernelEx(&cfg, keep ? chain_kernel<true> : chain_kernel<false>, args);
}

}  // namespace tfjsb
