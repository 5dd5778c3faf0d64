// Gradients of conv2d on the tensor cores (tcgen05), for any window, stride and dilation with channel counts that are
// multiples of 4.
//
// Precision.  These gradients are fp32 results: every fp32 operand is used as two TF32 values and the large products are
// summed in segments (umma_tile.cuh).  Against 64 bits, and fp32 multiply-adds on the same data: input gradient 1.5e-7 and
// 1.4e-7 at K = 72, 2.4e-7 and 6.0e-7 at 1152, 3.9e-7 and 1.2e-6 at 4608; filter gradient of 12544 pixels 2.1e-7 and 5.6e-7.
// (The filter gradient of a pointwise convolution whose operands are read as plain TF32 runs on the same kernel
// without the lo half.)
//
// Input gradient, conv2d_grad_input_kernel.  In padded coordinates u = iy + pt an input sample of residue a = u mod s
// receives the taps ky = a + s j from the output rows oy = (u - a) / s - j: for each of the sh * sw residue classes a
// stride-1 convolution of dy with the class's taps.  It is the implicit GEMM  dx[pixels, Cin] = dy_im2col . f^T  with
// K = (tap, Cout): both operands have Cout contiguous in memory already, so neither is packed or transposed.
//   warp 0      producer: A tile = im2col copy of 128 pixels x 32 channels of dy for one tap, B tile = block_n x 32
//               box of f[tap]; both swizzled K-major operand tiles as they land.
//   warp 1      MMA issuer: three products per 8 of K.
//   warps 2-5   epilogue: segments added up, the sum staged and stored row by row to the class's pixels.
//   warps 6-13  split: lo tile = elementwise function of the landed tile in the same layout (no index arithmetic).
// All classes are tiles of one launch; with too few tiles for the SMs the K loop is cut and the parts are added
// by a column sum.  Bound by shared memory: per k-block at block_n 128, 32 KB landed, 64 KB split and 96 KB read by the
// MMAs are 1500 cycles (768 of MMAs, about 600 of im2col copy); measured 1900.
// [16,28,28,128], 3x3, 128 channels: 6600 us with one CUDA-core thread per sample, 39 us here (35.6 with one accumulator for
// the whole sum, which 2.7e-6 of it is then missing); [4,14,14,512], 512 channels: 92 us (104 with one accumulator, when one
// lane and not an elected thread of a converged warp issued the MMAs).
//
// Filter gradient, conv2d_grad_filter_kernel.  df[(tap, ci), co] = sum over pixels: the summed index is the row of
// both x and dy, so a landed group ([32 pixels][32 channels]: an im2col or matrix box, with the swizzle of 32-byte pieces) is
// an MN-major operand as it is, and its halves are elementwise functions of it.  hi is rounded here, in place: left as copied,
// cut, it is 2.7e-7 off where rounded it is 2.2e-7 ([16,28,28,128], 3x3; 33.6 us).  M = four (tap, 32-channel)
// groups, N = 32..128 channels of dy, one (M tile, N tile, slice of the pixels) per CTA, partial sums added in slice
// order.  Per k-block at block_n 128, 32 KB landed and read, 64 KB of halves written and 96 KB read by the MMAs are 1750 cycles
// of shared memory (768 of MMAs); without the lo half the copy and 256 cycles of MMAs.  Against tiles transposed by the
// converter warps: [16,28,28,128], 3x3, 38.5 -> 36 us, [4,14,14,512] of 512 34 -> 32; pointwise, plain TF32, [32,56,56]
// 128 x 128 31 -> 26.5 with the sum of the parts, [64,14,14] 512 x 512 53 -> 46.
#include <algorithm>
#include <cstdlib>

#include "common.cuh"
#include "ptx_sm100.cuh"
#include "umma_tile.cuh"

namespace tfjsb {

using namespace ptx;
using namespace tile;

namespace {

constexpr int EPI_WARPS = 4, CVT_WARPS = 8;
constexpr int CG_THREADS = (2 + EPI_WARPS + CVT_WARPS) * 32;
constexpr int CG_MAX_STAGES = 4;
constexpr int GROUP_BYTES = 4096;  // 32 pixels x 32 channels

__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t base, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols) : "memory");
}

// A row of 32 results, and where it lies in the slab: the ones that are not finite among the first `live` are asked for again.
__device__ __forceinline__ bool row_not_finite(const uint32_t (&u)[32]) {
    bool odd = false;
#pragma unroll
    for (int e = 0; e < 32; ++e) odd = odd || not_finite(u[e]);
    return odd;
}
template <typename F>
__device__ __forceinline__ void mend_row(uint32_t slab, int lane, int live, F again) {
    for (int e = 0; e < min(32, live); ++e) {
        const uint32_t at = slab + (uint32_t)lane * 128u + (uint32_t)((((e >> 2) ^ (lane & 7)) << 4) + (e & 3) * 4);
        uint32_t bits;
        asm volatile("ld.shared.b32 %0, [%1];" : "=r"(bits) : "r"(at) : "memory");
        if (!not_finite(bits)) continue;
        const float v = again(e);
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(at), "f"(v) : "memory");
    }
}

// ---- input gradient --------------------------------------------------------------------------------------
struct GradInputArgs {
    int H, W, Cin, Cout, fh, fw, sh, sw, dh, dw, pt, pl;  // the forward convolution's
    int q0h, q0w, Qh, Qw;    // u / s of the first row / column, and how many
    int reach_h, reach_w;    // (taps of the largest class - 1) * dilation
    long long M;             // N * Qh * Qw
    int m_tiles, n_tiles, block_n, stages, splits, num_tiles;
    int segment;             // k-blocks per accumulator of the large products
    int Ho, Wo;
    const float *dy, *f;     // for results that are not finite
    float* out;              // dx, or `splits` of them one after the other
    long long out_elems;
    unsigned int* dev_status;
};

struct GradInputTile {
    int a, b, m0, n0, kb_begin, kb_end, c_blocks, taps_x, split;
};
__device__ __forceinline__ GradInputTile grad_input_tile(const GradInputArgs& g, int t) {
    GradInputTile r;
    r.split = t % g.splits;
    t /= g.splits;
    r.n0 = (t % g.n_tiles) * g.block_n;
    t /= g.n_tiles;
    r.m0 = (t % g.m_tiles) * BLOCK_M;
    const int cls = t / g.m_tiles;
    r.a = cls / g.sw;
    r.b = cls - r.a * g.sw;
    const int ny = r.a < g.fh ? (g.fh - r.a + g.sh - 1) / g.sh : 0;
    r.taps_x = r.b < g.fw ? (g.fw - r.b + g.sw - 1) / g.sw : 0;
    r.c_blocks = (g.Cout + BLOCK_K - 1) / BLOCK_K;
    const int kbs = ny * r.taps_x * r.c_blocks;
    r.kb_begin = (int)((long long)kbs * r.split / g.splits);
    r.kb_end = (int)((long long)kbs * (r.split + 1) / g.splits);
    return r;
}

// A result that is not finite once more: the tile's k-blocks of sample (n, qy, qx) of its class, channel ci, by fp32
// multiply-adds.  Taps whose output pixel does not exist take no part (in the copied tiles they are zeros, which an
// infinite filter value turns into NaN).
__device__ __noinline__ float grad_input_in_fp32(const GradInputArgs& g, const GradInputTile& r, long long n, int qy, int qx, int ci) {
    float acc = 0.f;
    for (int kb = r.kb_begin; kb < r.kb_end; ++kb) {
        const int tap = kb / r.c_blocks, co0 = (kb - tap * r.c_blocks) * BLOCK_K, jy = tap / r.taps_x, jx = tap - jy * r.taps_x;
        const int oy = g.q0h + qy - jy * g.dh, ox = g.q0w + qx - jx * g.dw;
        if (oy < 0 || oy >= g.Ho || ox < 0 || ox >= g.Wo) continue;
        const float* dy = g.dy + ((n * g.Ho + oy) * (long long)g.Wo + ox) * g.Cout;
        const float* f = g.f + ((long long)((r.a + jy * g.sh) * g.fw + r.b + jx * g.sw) * g.Cin + ci) * g.Cout;
        for (int co = co0; co < min(co0 + BLOCK_K, g.Cout); ++co) acc = fmaf(load_global(dy + co), load_global(f + co), acc);
        if (acc != acc) break;
    }
    return acc;
}

__global__ void __launch_bounds__(CG_THREADS, 1)
conv2d_grad_input_kernel(const __grid_constant__ CUtensorMap map_dy, const __grid_constant__ CUtensorMap map_f,
                         const __grid_constant__ GradInputArgs g) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[CG_MAX_STAGES], bar_split[CG_MAX_STAGES], bar_empty[CG_MAX_STAGES];
    __shared__ __align__(8) uint64_t bar_acc_full[2], bar_acc_empty[2], bar_small_empty, bar_drain;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag_s;
    volatile int* abort_flag = &abort_flag_s;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int raw_bytes = A_STAGE_BYTES + g.block_n * 128;
    const uint32_t epi_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t stage_base = epi_base + EPI_WARPS * EPI_SLAB_BYTES;
    auto stage_addr = [&](int s) { return stage_base + (uint32_t)s * (uint32_t)(2 * raw_bytes); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < g.stages; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_split[s]), CVT_WARPS);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&bar_acc_full[s]), 1);
            mbar_init(smem_u32(&bar_acc_empty[s]), EPI_WARPS);
        }
        mbar_init(smem_u32(&bar_small_empty), EPI_WARPS);
        mbar_init(smem_u32(&bar_drain), 1);
        abort_flag_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const uint32_t tmem_cols = (uint32_t)(4 * g.block_n);  // [large 0 | large 1 | small | sum]; block_n 32, 64, 128
    if (warp == 1) tmem_alloc(smem_u32(&tmem_slot), tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    pdl_launch_dependents();
    pdl_wait();

    if (warp == 0) {
        if (lane == 0) {
            int stage = 0, filled = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int t = blockIdx.x; ok && t < g.num_tiles; t += gridDim.x) {
                const GradInputTile r = grad_input_tile(g, t);
                const int row = r.m0 / g.Qw, img = row / g.Qh;
                const int h0 = g.q0h + row - img * g.Qh - g.reach_h, w0 = g.q0w + r.m0 - row * g.Qw - g.reach_w;
                int tap = r.kb_begin / r.c_blocks, cb = r.kb_begin - tap * r.c_blocks;
                for (int kb = r.kb_begin; kb < r.kb_end; ++kb) {
                    if (!bounded_wait(smem_u32(&bar_empty[stage]), phase ^ 1u, abort_flag)) { ok = false; break; }
                    const int jy = tap / r.taps_x, jx = tap - jy * r.taps_x;
                    const uint32_t full = smem_u32(&bar_full[stage]), dst = stage_addr(stage);
                    mbar_arrive_expect_tx(full, (uint32_t)raw_bytes);
                    tma_load_im2col(dst, &map_dy, full, cb * BLOCK_K, w0, h0, img, g.reach_w - jx * g.dw, g.reach_h - jy * g.dh);
                    tma_load_3d(dst + A_STAGE_BYTES, &map_f, full, cb * BLOCK_K, r.n0, (r.a + jy * g.sh) * g.fw + r.b + jx * g.sw);
                    if (++cb == r.c_blocks) { cb = 0; ++tap; }
                    ++filled;
                    if (++stage == g.stages) { stage = 0; phase ^= 1u; }
                }
            }
            if (!ok) {
                give_up(abort_flag, g.dev_status, DEV_STATUS_TIMEOUT_PRODUCER);
                for (int k = filled > g.stages ? filled - g.stages : 0; k < filled; ++k)
                    drain(smem_u32(&bar_full[k % g.stages]), (uint32_t)((k / g.stages) & 1), g.dev_status);
            }
        }
    } else if (warp == 1) {
        const uint32_t idesc = make_idesc_tf32(BLOCK_M, g.block_n);
        const uint32_t small = tmem + (uint32_t)(2 * g.block_n);
        int stage = 0, acc = 0;
        uint32_t phase = 0, acc_phase = 0, small_phase = 0;
        const bool leader = elect_one();
        bool ok = true, issued = false;  // the leader's
        for (int t = blockIdx.x; t < g.num_tiles; t += gridDim.x) {
            const GradInputTile r = grad_input_tile(g, t);
            if (r.kb_begin == r.kb_end) continue;  // no tap reaches these samples
            // the tile before has been added up
            if (leader && ok) ok = bounded_wait(smem_u32(&bar_small_empty), small_phase ^ 1u, abort_flag);
            small_phase ^= 1u;
            int in_seg = 0;
            for (int kb = r.kb_begin; kb < r.kb_end; ++kb) {
                if (in_seg == 0 && leader && ok) ok = bounded_wait(smem_u32(&bar_acc_empty[acc]), acc_phase ^ 1u, abort_flag);
                const uint32_t large = tmem + (uint32_t)(acc * g.block_n);
                const uint32_t hi = stage_addr(stage), lo = hi + (uint32_t)raw_bytes;
                const uint64_t ah = make_kmajor_sw128_desc(hi), bh = make_kmajor_sw128_desc(hi + A_STAGE_BYTES);
                const uint64_t al = make_kmajor_sw128_desc(lo), bl = make_kmajor_sw128_desc(lo + A_STAGE_BYTES);
                if (leader && ok && (ok = bounded_wait(smem_u32(&bar_full[stage]), phase, abort_flag) &&
                                          bounded_wait(smem_u32(&bar_split[stage]), phase, abort_flag))) {
                    tc_fence_after();
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint64_t o = (uint64_t)(2 * k);
                        tc_mma_tf32(large, ah + o, bh + o, idesc, (in_seg | k) != 0 ? 1u : 0u);
                        tc_mma_tf32(small, ah + o, bl + o, idesc, (kb != r.kb_begin || k != 0) ? 1u : 0u);
                        tc_mma_tf32(small, al + o, bh + o, idesc, 1u);
                    }
                    issued = true;
                    tc_commit(smem_u32(&bar_empty[stage]));
                }
                if (++stage == g.stages) { stage = 0; phase ^= 1u; }
                if (++in_seg == g.segment || kb + 1 == r.kb_end) {
                    if (leader && ok) tc_commit(smem_u32(&bar_acc_full[acc]));
                    in_seg = 0;
                    if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
                }
            }
        }
        if (!ok) {
            give_up(abort_flag, g.dev_status, DEV_STATUS_TIMEOUT_MMA);
            if (issued) {
                tc_commit(smem_u32(&bar_drain));
                drain(smem_u32(&bar_drain), 0u, g.dev_status);
            }
        }
        __syncwarp();
    } else if (warp < 2 + EPI_WARPS) {
        const int quad = warp & 3;
        const uint32_t slab = epi_base + (uint32_t)(warp - 2) * EPI_SLAB_BYTES;
        const uint32_t lanes = tmem + ((uint32_t)(quad * 32) << 16);
        const bool vec = (g.Cin & 3) == 0;
        int acc = 0;
        uint32_t acc_phase = 0;
        for (int t = blockIdx.x; t < g.num_tiles; t += gridDim.x) {
            const GradInputTile r = grad_input_tile(g, t);
            const bool any = r.kb_begin != r.kb_end;
            // lane = one sample of dx: where its row of channels goes, or -1
            long long at = -1, n = 0;
            int qx = 0, qy = 0;
            const long long p = (long long)r.m0 + quad * 32 + lane;
            if (p < g.M) {
                const long long row = p / g.Qw;
                qx = (int)(p - row * g.Qw);
                n = row / g.Qh;
                qy = (int)(row - n * g.Qh);
                const int iy = (g.q0h + qy) * g.sh + r.a - g.pt, ix = (g.q0w + qx) * g.sw + r.b - g.pl;
                if (iy >= 0 && iy < g.H && ix >= 0 && ix < g.W) at = ((n * g.H + iy) * (long long)g.W + ix) * g.Cin;
            }
            float* out = g.out + (long long)r.split * g.out_elems;
            const int live = min(g.block_n, g.Cin - r.n0);
            bool ok = true;
            for (int kb = r.kb_begin; kb < r.kb_end; kb += g.segment) {
                const bool got = bounded_wait(smem_u32(&bar_acc_full[acc]), acc_phase, abort_flag), last = kb + g.segment >= r.kb_end;
                if (!(ok = __all_sync(0xffffffffu, got))) break;
                tc_fence_after();
                add_segment<16>(lanes + (uint32_t)(acc * g.block_n), lanes + (uint32_t)(2 * g.block_n), lanes + (uint32_t)(3 * g.block_n), (live + 15) & ~15,
                            kb == r.kb_begin, last);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(smem_u32(&bar_acc_empty[acc]));
                    if (last) mbar_arrive(smem_u32(&bar_small_empty));
                }
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
            if (!ok) {
                if (lane == 0) give_up(abort_flag, g.dev_status, DEV_STATUS_TIMEOUT_EPILOGUE);
                break;
            }
            for (int c0 = 0; c0 < live; c0 += 32) {
                uint32_t u[32];
                if (any) {
                    tc_ld_32x32(lanes + (uint32_t)(3 * g.block_n + c0), u);
                    tc_ld_wait();
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) u[e] = 0u;
                }
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    sts4(slab + (uint32_t)lane * 128u + (uint32_t)((j ^ (lane & 7)) << 4), __uint_as_float(u[4 * j]), __uint_as_float(u[4 * j + 1]),
                         __uint_as_float(u[4 * j + 2]), __uint_as_float(u[4 * j + 3]));
                const int col0 = r.n0 + c0;
                if (any && at >= 0 && row_not_finite(u))
                    mend_row(slab, lane, g.Cin - col0, [&](int e) { return grad_input_in_fp32(g, r, n, qy, qx, col0 + e); });
                __syncwarp();
                if (vec) {
                    // four rows per step, eight lanes to a row's 128 bytes
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int rr = 4 * i + (lane >> 3), j = lane & 7;
                        const long long o = __shfl_sync(0xffffffffu, at, rr);
                        const float4 w = lds4(slab + (uint32_t)rr * 128u + (uint32_t)((j ^ (rr & 7)) << 4));
                        if (o >= 0 && col0 + 4 * j < g.Cin) *reinterpret_cast<float4*>(out + o + col0 + 4 * j) = w;
                    }
                } else {
                    for (int rr = 0; rr < 32; ++rr) {
                        const long long o = __shfl_sync(0xffffffffu, at, rr);
                        float w;
                        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(w) : "r"(slab + (uint32_t)rr * 128u + (uint32_t)((((lane >> 2) ^ (rr & 7)) << 4) + (lane & 3) * 4)) : "memory");
                        if (o >= 0 && col0 + lane < g.Cin) out[o + col0 + lane] = w;
                    }
                }
                __syncwarp();
            }
        }
    } else {
        const uint32_t mine = (uint32_t)(threadIdx.x - (2 + EPI_WARPS) * 32) * 16u;
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int t = blockIdx.x; ok && t < g.num_tiles; t += gridDim.x) {
            const GradInputTile r = grad_input_tile(g, t);
            for (int kb = r.kb_begin; kb < r.kb_end; ++kb) {
                const bool got = bounded_wait(smem_u32(&bar_full[stage]), phase, abort_flag);
                if (!__all_sync(0xffffffffu, got)) {
                    if (lane == 0) give_up(abort_flag, g.dev_status, DEV_STATUS_TIMEOUT_PRODUCER);
                    ok = false;
                    break;
                }
                const uint32_t src = stage_addr(stage) + mine, dst = src + (uint32_t)raw_bytes;
                // 256 threads x 16 bytes = 4 KB per step; raw_bytes is a multiple of 4 KB
#pragma unroll 4
                for (int o = 0; o < raw_bytes; o += CVT_WARPS * 512) {
                    const float4 v = lds4(src + (uint32_t)o);
                    const uint32_t round = o < A_STAGE_BYTES ? SPLIT_UP : SPLIT_NEAREST;
                    sts4(dst + (uint32_t)o, tf32_rest(v.x, round), tf32_rest(v.y, round), tf32_rest(v.z, round), tf32_rest(v.w, round));
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bar_split[stage]));
                if (++stage == g.stages) { stage = 0; phase ^= 1u; }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_free(tmem, tmem_cols);
    }
}

// ---- filter gradient ---------------------------------------------------------------------------------------
struct GradFilterArgs {
    int taps, fw, sh, sw, dh, dw, pt, pl, Ho, Wo;
    int c_blocks;   // 32-channel blocks of x
    int groups;     // taps * c_blocks
    int n_tiles, block_n, stages;
    int pixel_blocks, blocks_per_slice;  // blocks of 32 pixels
    int m_tiles;
    int segment;    // k-blocks per accumulator of the large products
    int tiled;      // x as a matrix [pixels, Cin] (1x1, stride 1) instead of im2col copies
    int H, W, Cin, Cout;
    long long pixels;
    const float *x, *dy;  // for results that are not finite
    unsigned int* dev_status;
};

// A result that is not finite once more: output pixels p0 .. p1 by fp32 multiply-adds, samples outside the image as zeros.
__device__ __noinline__ float grad_filter_in_fp32(const GradFilterArgs& g, long long p0, long long p1, int tap, int ci, int co) {
    const int ky = tap / g.fw, off_h = ky * g.dh - g.pt, off_w = (tap - ky * g.fw) * g.dw - g.pl;
    float acc = 0.f;
    for (long long p = p0; p < p1 && acc == acc; ++p) {
        const long long row = p / g.Wo, n = row / g.Ho;
        const int iy = (int)(row - n * g.Ho) * g.sh + off_h, ix = (int)(p - row * g.Wo) * g.sw + off_w;
        const bool inside = iy >= 0 && iy < g.H && ix >= 0 && ix < g.W;
        acc = fmaf(inside ? load_global(g.x + ((n * g.H + iy) * (long long)g.W + ix) * g.Cin + ci) : 0.f, load_global(g.dy + p * g.Cout + co), acc);
    }
    return acc;
}

template <bool SPLIT>
__global__ void __launch_bounds__(CG_THREADS, 1)
conv2d_grad_filter_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_dy,
                          const __grid_constant__ CUtensorMap map_out, const __grid_constant__ GradFilterArgs g) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[CG_MAX_STAGES], bar_split[CG_MAX_STAGES], bar_empty[CG_MAX_STAGES];
    __shared__ __align__(8) uint64_t bar_acc_full[2], bar_acc_empty[2], bar_drain;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag_s;
    volatile int* abort_flag = &abort_flag_s;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b_groups = g.block_n >> 5;
    const int raw_bytes = (4 + b_groups) * GROUP_BYTES;  // A groups, then B groups; SPLIT: their lo halves behind them
    constexpr int HALVES = SPLIT ? 2 : 1;
    const uint32_t epi_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t stage_base = epi_base + EPI_WARPS * EPI_SLAB_BYTES;
    auto stage_addr = [&](int s) { return stage_base + (uint32_t)(s * HALVES * raw_bytes); };

    int unit = blockIdx.x;
    const int nt = unit % g.n_tiles;
    unit /= g.n_tiles;
    const int mt = unit % g.m_tiles, slice = unit / g.m_tiles;
    const int g0 = mt * 4, live_groups = min(4, g.groups - g0), n0 = nt * g.block_n;
    const int pb0 = slice * g.blocks_per_slice;
    const int kbs = max(0, min(g.blocks_per_slice, g.pixel_blocks - pb0));  // never zero: the host makes no empty slice

    if (threadIdx.x == 0) {
        for (int s = 0; s < g.stages; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_split[s]), CVT_WARPS);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&bar_acc_full[s]), 1);
            mbar_init(smem_u32(&bar_acc_empty[s]), EPI_WARPS);
        }
        mbar_init(smem_u32(&bar_drain), 1);
        abort_flag_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const uint32_t tmem_cols = (uint32_t)((SPLIT ? 4 : 1) * g.block_n);  // [large 0 | large 1 | small | sum], or one accumulator
    if (warp == 1) tmem_alloc(smem_u32(&tmem_slot), tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    pdl_launch_dependents();
    pdl_wait();

    if (warp == 0) {
        if (lane == 0) {
            int tap_h[4], tap_w[4], ch[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int gi = g0 + i, tap = gi / g.c_blocks;
                ch[i] = (gi - tap * g.c_blocks) * 32;
                const int ky = tap / g.fw;
                tap_h[i] = ky * g.dh;
                tap_w[i] = (tap - ky * g.fw) * g.dw;
            }
            int stage = 0, filled = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int kb = 0; kb < kbs; ++kb) {
                if (!bounded_wait(smem_u32(&bar_empty[stage]), phase ^ 1u, abort_flag)) { ok = false; break; }
                const uint32_t full = smem_u32(&bar_full[stage]), dst = stage_addr(stage);
                const int p0 = (pb0 + kb) * 32;
                mbar_arrive_expect_tx(full, (uint32_t)((live_groups + b_groups) * GROUP_BYTES));
                const int row = p0 / g.Wo, img = row / g.Ho;
                const int h0 = (row - img * g.Ho) * g.sh - g.pt, w0 = (p0 - row * g.Wo) * g.sw - g.pl;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (i >= live_groups) break;
                    if (g.tiled) tma_load_2d(dst + i * GROUP_BYTES, &map_x, full, ch[i], p0);
                    else tma_load_im2col(dst + i * GROUP_BYTES, &map_x, full, ch[i], w0, h0, img, tap_w[i], tap_h[i]);
                }
                for (int i = 0; i < b_groups; ++i) tma_load_2d(dst + (4 + i) * GROUP_BYTES, &map_dy, full, n0 + i * 32, p0);
                ++filled;
                if (++stage == g.stages) { stage = 0; phase ^= 1u; }
            }
            if (!ok) {
                give_up(abort_flag, g.dev_status, DEV_STATUS_TIMEOUT_PRODUCER);
                for (int k = filled > g.stages ? filled - g.stages : 0; k < filled; ++k)
                    drain(smem_u32(&bar_full[k % g.stages]), (uint32_t)((k / g.stages) & 1), g.dev_status);
            }
        }
    } else if (warp == 1) {
        const uint32_t idesc = make_idesc_tf32(BLOCK_M, g.block_n) | IDESC_A_MN | IDESC_B_MN;
        const uint32_t small = tmem + (uint32_t)(2 * g.block_n);
        int stage = 0, acc = 0, in_seg = 0;
        uint32_t phase = 0, acc_phase = 0;
        const bool leader = elect_one();
        bool ok = true, issued = false;  // the leader's
        for (int kb = 0; kb < kbs; ++kb) {
            if (SPLIT && in_seg == 0 && leader && ok) ok = bounded_wait(smem_u32(&bar_acc_empty[acc]), acc_phase ^ 1u, abort_flag);
            const uint32_t large = tmem + (uint32_t)(acc * g.block_n);
            const uint32_t hi = stage_addr(stage), lo = hi + (uint32_t)raw_bytes;
            uint64_t ah[4], bh[4], al[4], bl[4];  // eight pixels per MMA
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                ah[k] = make_mnmajor_desc(hi) + (uint64_t)(64 * k);
                bh[k] = make_mnmajor_desc(hi + A_STAGE_BYTES) + (uint64_t)(64 * k);
                al[k] = make_mnmajor_desc(lo) + (uint64_t)(64 * k);
                bl[k] = make_mnmajor_desc(lo + A_STAGE_BYTES) + (uint64_t)(64 * k);
            }
            if (leader && ok && (ok = bounded_wait(smem_u32(&bar_full[stage]), phase, abort_flag) &&
                                      (!SPLIT || bounded_wait(smem_u32(&bar_split[stage]), phase, abort_flag)))) {
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    tc_mma_tf32(large, ah[k], bh[k], idesc, ((SPLIT ? in_seg : kb) | k) != 0 ? 1u : 0u);
                    if (SPLIT) {
                        tc_mma_tf32(small, ah[k], bl[k], idesc, (kb | k) != 0 ? 1u : 0u);
                        tc_mma_tf32(small, al[k], bh[k], idesc, 1u);
                    }
                }
                issued = true;
                tc_commit(smem_u32(&bar_empty[stage]));
            }
            if (++stage == g.stages) { stage = 0; phase ^= 1u; }
            if (kb + 1 == kbs || (SPLIT && ++in_seg == g.segment)) {
                if (leader && ok) tc_commit(smem_u32(&bar_acc_full[acc]));
                in_seg = 0;
                if (SPLIT && ++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
        }
        if (!ok) {
            give_up(abort_flag, g.dev_status, DEV_STATUS_TIMEOUT_MMA);
            if (issued) {
                tc_commit(smem_u32(&bar_drain));
                drain(smem_u32(&bar_drain), 0u, g.dev_status);
            }
        }
        __syncwarp();
    } else if (warp < 2 + EPI_WARPS) {
        const int quad = warp & 3;  // the M tile's group whose 32 rows this warp may read
        const uint32_t slab = epi_base + (uint32_t)(warp - 2) * EPI_SLAB_BYTES;
        const uint32_t lanes = tmem + ((uint32_t)(quad * 32) << 16);
        bool ok = true;
        int acc = 0;
        uint32_t acc_phase = 0;
        for (int kb = 0; kb < kbs; kb += SPLIT ? g.segment : kbs) {
            const bool got = bounded_wait(smem_u32(&bar_acc_full[acc]), acc_phase, abort_flag);
            if (!(ok = __all_sync(0xffffffffu, got))) break;
            tc_fence_after();
            if (SPLIT) {
                add_segment<16>(lanes + (uint32_t)(acc * g.block_n), lanes + (uint32_t)(2 * g.block_n), lanes + (uint32_t)(3 * g.block_n), g.block_n, kb == 0,
                            kb + g.segment >= kbs);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bar_acc_empty[acc]));
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
        }
        if (!ok) {
            if (lane == 0) give_up(abort_flag, g.dev_status, DEV_STATUS_TIMEOUT_EPILOGUE);
        } else if (quad < live_groups) {
            const int gi = g0 + quad, tap = gi / g.c_blocks, ci0 = (gi - tap * g.c_blocks) * 32;
            for (int c0 = 0; c0 < g.block_n; c0 += 32) {
                uint32_t u[32];
                tc_ld_32x32(lanes + (uint32_t)((SPLIT ? 3 * g.block_n : 0) + c0), u);
                tc_ld_wait();
                if (lane == 0) tma_store_wait_read<0>();
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    sts4(slab + (uint32_t)lane * 128u + (uint32_t)((j ^ (lane & 7)) << 4), __uint_as_float(u[4 * j]), __uint_as_float(u[4 * j + 1]),
                         __uint_as_float(u[4 * j + 2]), __uint_as_float(u[4 * j + 3]));
                if (SPLIT && ci0 + lane < g.Cin && row_not_finite(u)) {
                    const long long p0 = (long long)pb0 * 32, p1 = min(g.pixels, p0 + kbs * 32LL);
                    mend_row(slab, lane, g.Cout - n0 - c0, [&](int e) { return grad_filter_in_fp32(g, p0, p1, tap, ci0 + lane, n0 + c0 + e); });
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    tma_store_3d(&map_out, slab, n0 + c0, ci0, slice * g.taps + tap);  // clipped at Cout and Cin
                    tma_store_commit();
                }
            }
            if (lane == 0) tma_store_wait_all();
            __syncwarp();
        }
    } else if (SPLIT) {
        const uint32_t mine = (uint32_t)(threadIdx.x - (2 + EPI_WARPS) * 32) * 16u;
        int stage = 0;
        uint32_t phase = 0;
        for (int kb = 0; kb < kbs; ++kb) {
            const bool got = bounded_wait(smem_u32(&bar_full[stage]), phase, abort_flag);
            if (!__all_sync(0xffffffffu, got)) {
                if (lane == 0) give_up(abort_flag, g.dev_status, DEV_STATUS_TIMEOUT_PRODUCER);
                break;
            }
            const uint32_t src = stage_addr(stage) + mine, dst = src + (uint32_t)raw_bytes;
            // 256 threads x 16 bytes: a group of 32 pixels x 32 channels per step
#pragma unroll 4
            for (int o = 0; o < raw_bytes; o += CVT_WARPS * 512) {
                const float4 v = lds4(src + (uint32_t)o);
                float hi[4], lo[4];
                tf32_split(v.x, hi[0], lo[0]);
                tf32_split(v.y, hi[1], lo[1]);
                tf32_split(v.z, hi[2], lo[2]);
                tf32_split(v.w, hi[3], lo[3]);
                sts4(src + (uint32_t)o, hi[0], hi[1], hi[2], hi[3]);
                sts4(dst + (uint32_t)o, lo[0], lo[1], lo[2], lo[3]);
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bar_split[stage]));
            if (++stage == g.stages) { stage = 0; phase ^= 1u; }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_free(tmem, tmem_cols);
    }
}

constexpr int CG_SMEM = SMEM_LIMIT - 1024;  // beside the barriers

tfjsb_status encode_im2col(tfjsb_ctx* ctx, CUtensorMap* map, const float* base, int64_t n, int h, int w, int c, const int lower[2],
                           const int upper[2], int sw, int sh, int pixels, const char* what, CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B) {
    cuuint64_t d[4] = {(cuuint64_t)c, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)n};
    cuuint64_t st[3] = {(cuuint64_t)c * 4, (cuuint64_t)w * c * 4, (cuuint64_t)h * w * c * 4};
    cuuint32_t elem[4] = {1u, (cuuint32_t)sw, (cuuint32_t)sh, 1u};
    CUresult r = ctx->encode_im2col(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float*>(base), d, st, lower, upper, 32,
                                    (cuuint32_t)pixels, elem, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(ctx, TFJSB_ERR_CUDA, std::string("cuTensorMapEncodeIm2col failed for ") + what + " (CUresult " + std::to_string((int)r) + ")");
    return TFJSB_OK;
}

bool corner_ok(int64_t v) { return v >= -128 && v <= 127; }

}  // namespace

tfjsb_status encode_tile_map(tfjsb_ctx* ctx, CUtensorMap* map, const float* base, int rank, const int64_t* dims, const uint32_t* box, const char* what,
                             CUtensorMapSwizzle swizzle) {
    cuuint64_t d[4], st[3];
    cuuint32_t b[4], elem[4] = {1u, 1u, 1u, 1u};
    cuuint64_t pitch = 4;
    for (int i = 0; i < rank; ++i) {
        d[i] = (cuuint64_t)dims[i];
        b[i] = box[i];
        pitch *= d[i];
        if (i + 1 < rank) st[i] = pitch;
    }
    CUresult r = ctx->encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, (cuuint32_t)rank, const_cast<float*>(base), d, st, b, elem,
                                   CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(ctx, TFJSB_ERR_CUDA, std::string("cuTensorMapEncodeTiled failed for ") + what + " (CUresult " + std::to_string((int)r) + ")");
    return TFJSB_OK;
}

// u / s of the first sample along one dimension, and how many values it takes
static void grad_rows(int size, int pad, int s, int* q0, int* count) {
    *q0 = pad / s;
    *count = (size - 1 + pad) / s - *q0 + 1;
}

struct GradInputTiling {
    int block_n = 32, kbs = 0, splits = 1;  // kbs: k-blocks of the largest class
    int64_t tiles = 0;
};
static GradInputTiling grad_input_tiling(const ConvGeom& g, int64_t m_tiles, int sms) {
    GradInputTiling t;
    // Tile width: the fewest rounds, each as long as the slower of the MMAs (6 cycles per column and k-block) and the
    // im2col copy (about 600 cycles per k-block).
    int64_t best = INT64_MAX;
    for (int bn = 32; bn <= 128; bn <<= 1) {
        const int64_t tiles = m_tiles * ((g.C + bn - 1) / bn) * g.sh * g.sw;
        const int64_t cost = (tiles + sms - 1) / sms * (6 * bn > 600 ? 6 * bn : 600);
        if (cost < best) { best = cost; t.block_n = bn; t.tiles = tiles; }
        if (bn >= g.C) break;
    }
    t.kbs = ((g.fh + g.sh - 1) / g.sh) * ((g.fw + g.sw - 1) / g.sw) * ((g.Co + 31) / 32);
    // fewer tiles than half the SMs: the K loop in parts of at least eight k-blocks
    if (2 * t.tiles <= sms) {
        t.splits = (int)(sms / t.tiles);
        if (t.splits > t.kbs / 8) t.splits = t.kbs / 8;
        if (t.splits > 16) t.splits = 16;
        if (t.splits < 1) t.splits = 1;
    }
    return t;
}

// The kernel below at stride 1 with 3x3 windows of 16 channels or more, fitted like the patch kernel's estimate and to the same
// shapes (conv_patch_tcgen05.cu; nine in ten within 10 %): per round an epilogue and k-blocks.
double conv2d_grad_input_us(const ConvGeom& g, int sm_count) {
    const GradInputTiling t = grad_input_tiling(g, (g.N * g.H * g.W + BLOCK_M - 1) / BLOCK_M, sm_count);
    const double round = t.block_n == 32 ? 2.6 : t.block_n == 64 ? 3.8 : 5.8, kb = t.block_n == 32 ? 0.62 : t.block_n == 64 ? 0.65 : 0.77;
    const double rounds = (double)((t.tiles * t.splits + sm_count - 1) / sm_count), out_mb = (double)g.N * g.H * g.W * g.C * 4e-6;
    return 4.5 + rounds * (round + kb * ((t.kbs + t.splits - 1) / t.splits)) + (t.splits > 1 ? 1.0 + t.splits * out_mb : 0.0);
}

// Where a sample's sum is short, one CUDA-core thread per sample is the faster kernel.  In microseconds, fitted to both on
// 145 shapes (4 to 64 output channels, windows up to 7 x 7, strides 1 to 3; 4 % of them still go to the slower one):
//   here         3, and for each round of tiles 1.4 and 0.72 per k-block, of which a tap makes at least one however few its
//                channels; parts of the K loop 2.5 more, several residue classes 1
//   CUDA cores   2.5 and 0.42 per tap of a class, the chain of one thread; its samples x products at 0.2 to 1.7 per ps, the
//                fewer the longer the filter rows that threads read apart; strided, 2 ps a sample, also of those without a
//                product; a strided 1x1, most of whose samples have none, 6.2 ps a sample and 0.6 per product
// [15,8,8,20], 3x3, 8 channels: 11.3 us here and 7.6; [5,27,27,256]: 13.6 and 70; [35,108,108,4]: 174 and 75;
// [4,224,224,64], 1x1 / 3, 4 channels: 28 and 85.
bool conv2d_grad_input_preferred(const ConvGeom& g, int sm_count) {
    if (const char* env = getenv("TFJSB_GRAD_INPUT")) return atoi(env) != 0;  // for tests: 1 = this kernel wherever it can
    int q0h, q0w, Qh, Qw;
    grad_rows(g.H, g.pt, g.sh, &q0h, &Qh);
    grad_rows(g.W, g.pl, g.sw, &q0w, &Qw);
    const GradInputTiling t = grad_input_tiling(g, (g.N * Qh * Qw + BLOCK_M - 1) / BLOCK_M, sm_count);
    const bool strided = g.sh * g.sw > 1;
    const double rounds = (double)((t.tiles * t.splits + sm_count - 1) / sm_count), taps = (double)g.fh * g.fw;
    const double here = 3 + rounds * (0.72 * t.kbs / t.splits + 1.4) + (t.splits > 1 ? 2.5 : 0) + (strided ? 1 : 0);
    const double samples = (double)g.N * g.H * g.W * g.C, products = taps * g.Co / (g.sh * g.sw);
    const double per_us = g.C <= 8 && g.Co <= 16 ? 1.7e6 : g.Co <= 12 ? 1.0e6 : g.Co <= 16 || g.C <= 8 ? 0.52e6 : 0.22e6;
    const double class_taps = (double)((g.fh + g.sh - 1) / g.sh) * ((g.fw + g.sw - 1) / g.sw);
    // the threads of a warp are neighbouring channels: fewer than 32 of them and a strided window's taps diverge
    const double chain = !strided ? 0.02 * products : (taps > 1 ? 0.08 * g.Co : 0.07 * std::max<int64_t>(0, g.Co - 24)) + (g.C < 32 ? 0.2 : 0.02) * taps;
    const double each = !strided ? products / per_us : taps > 1 ? 2 * products / per_us + 2e-6 : 0.6e-6 * products + 6.2e-6;
    return here <= 2.5 + 0.42 * class_taps + chain + samples * each;
}

bool conv2d_grad_input_supported(const ConvGeom& g) {
    int q0h, q0w, Qh, Qw;
    grad_rows(g.H, g.pt, g.sh, &q0h, &Qh);
    grad_rows(g.W, g.pl, g.sw, &q0w, &Qw);
    const int64_t reach_h = (int64_t)((g.fh - 1) / g.sh) * g.dh, reach_w = (int64_t)((g.fw - 1) / g.sw) * g.dw;
    const int64_t m_tiles = (g.N * Qh * Qw + BLOCK_M - 1) / BLOCK_M;
    return g.Co % 4 == 0 && reach_h <= 127 && reach_w <= 127 && corner_ok(q0h - reach_h) && corner_ok(q0w - reach_w) &&
           corner_ok(q0h - reach_h + Qh - g.Ho) && corner_ok(q0w - reach_w + Qw - g.Wo) && g.Ho > 0 && g.Wo > 0 &&
           g.N * Qh * Qw < (1LL << 31) - 256 && m_tiles * g.sh * g.sw * ((g.C + 31) / 32) * 16 < (1LL << 31) &&
           (int64_t)g.fh * g.fw * ((g.Co + 31) / 32) * 32 <= SPLIT_MAX_K;
}

tfjsb_status run_conv2d_grad_input(tfjsb_ctx* ctx, const float* dy, const float* f, float* dx, const ConvGeom& g, cudaStream_t s) {
    GradInputArgs a{};
    a.H = g.H; a.W = g.W; a.Cin = g.C; a.Cout = g.Co; a.fh = g.fh; a.fw = g.fw;
    a.sh = g.sh; a.sw = g.sw; a.dh = g.dh; a.dw = g.dw; a.pt = g.pt; a.pl = g.pl;
    grad_rows(g.H, g.pt, g.sh, &a.q0h, &a.Qh);
    grad_rows(g.W, g.pl, g.sw, &a.q0w, &a.Qw);
    a.reach_h = (g.fh - 1) / g.sh * g.dh;
    a.reach_w = (g.fw - 1) / g.sw * g.dw;
    a.M = g.N * a.Qh * a.Qw;
    a.m_tiles = (int)((a.M + BLOCK_M - 1) / BLOCK_M);
    const int sms = ctx->sm_count;
    const GradInputTiling tl = grad_input_tiling(g, a.m_tiles, sms);
    a.block_n = tl.block_n;
    a.n_tiles = (g.C + a.block_n - 1) / a.block_n;
    const int64_t tiles = tl.tiles;
    const int kbs = tl.kbs;
    a.splits = (int)scratch_parts(ctx->scratch_c, tl.splits, (size_t)g.N * g.H * g.W * g.C * 4, s);
    a.num_tiles = (int)(tiles * a.splits);
    a.segment = split_segment((int64_t)kbs * BLOCK_K);
    const int stage_bytes = 2 * (A_STAGE_BYTES + a.block_n * 128);
    a.stages = (CG_SMEM - 1024 - EPI_WARPS * EPI_SLAB_BYTES) / stage_bytes;
    if (a.stages > CG_MAX_STAGES) a.stages = CG_MAX_STAGES;
    a.out_elems = (long long)g.N * g.H * g.W * g.C;
    a.Ho = g.Ho; a.Wo = g.Wo;
    a.dy = dy; a.f = f;
    a.dev_status = ctx->dev_status;
    tfjsb_status st;
    a.out = dx;
    if (a.splits > 1) {
        if ((st = ensure_scratch(ctx, &ctx->scratch_c, (size_t)a.splits * a.out_elems * 4)) != TFJSB_OK) return st;
        a.out = ctx->scratch_c.ptr;
    }
    CUtensorMap map_dy, map_f;
    const int lower[2] = {a.q0w - a.reach_w, a.q0h - a.reach_h};
    const int upper[2] = {lower[0] + a.Qw - g.Wo, lower[1] + a.Qh - g.Ho};
    if ((st = encode_im2col(ctx, &map_dy, dy, g.N, g.Ho, g.Wo, g.Co, lower, upper, 1, 1, BLOCK_M, "dy")) != TFJSB_OK) return st;
    const int64_t fd[3] = {g.Co, g.C, (int64_t)g.fh * g.fw};
    const uint32_t fb[3] = {32u, (uint32_t)a.block_n, 1u};
    if ((st = encode_tile_map(ctx, &map_f, f, 3, fd, fb, "the filter")) != TFJSB_OK) return st;
    cudaError_t e = smem_attr_once(reinterpret_cast<const void*>(&conv2d_grad_input_kernel), CG_SMEM);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "shared-memory limit");
    const size_t smem = 1024 + (size_t)EPI_WARPS * EPI_SLAB_BYTES + (size_t)a.stages * stage_bytes;
    const int grid = a.num_tiles < sms ? a.num_tiles : sms;
    if ((e = launch_k(conv2d_grad_input_kernel, dim3(grid), dim3(CG_THREADS), smem, s, map_dy, map_f, a)) != cudaSuccess)
        return cuda_fail(ctx, e, "conv2d_grad_input launch");
    ++ctx->launches;
    if (a.splits > 1 && (e = launch_sum_rows(a.out, dx, nullptr, a.splits, a.out_elems, 1, s, &ctx->launches)) != cudaSuccess)
        return cuda_fail(ctx, e, "partial-sum launch");
    return TFJSB_OK;
}

bool conv2d_grad_filter_supported(const ConvGeom& g) {
    const int64_t upper_w = (int64_t)(g.Wo - 1) * g.sw - g.pl - (g.W - 1), upper_h = (int64_t)(g.Ho - 1) * g.sh - g.pt - (g.H - 1);
    const int64_t pixels = g.N * g.Ho * g.Wo, taps = (int64_t)g.fh * g.fw;
    const bool tiled = taps == 1 && g.sh == 1 && g.sw == 1;
    return g.C % 4 == 0 && g.Co % 4 == 0 && g.C > 0 && g.Co > 0 && pixels > 0 && pixels < (1LL << 31) - 256 &&
           (tiled || (g.sh <= 8 && g.sw <= 8 && (int64_t)(g.fh - 1) * g.dh <= 127 && (int64_t)(g.fw - 1) * g.dw <= 127 && g.pl <= 127 &&
                      g.pt <= 127 && corner_ok(upper_w) && corner_ok(upper_h))) &&
           taps * ((g.C + 31) / 32) * ((g.Co + 31) / 32) < (1LL << 20);
}

tfjsb_status run_conv2d_grad_filter(tfjsb_ctx* ctx, const float* x, const float* dy, float* df, const ConvGeom& g, bool split, cudaStream_t s) {
    GradFilterArgs a{};
    const int64_t pixels = g.N * g.Ho * g.Wo;
    a.taps = g.fh * g.fw; a.fw = g.fw; a.sh = g.sh; a.sw = g.sw; a.dh = g.dh; a.dw = g.dw; a.pt = g.pt; a.pl = g.pl;
    a.Ho = g.Ho; a.Wo = g.Wo;
    a.H = g.H; a.W = g.W; a.Cin = g.C; a.Cout = g.Co;
    a.pixels = pixels;
    a.x = x; a.dy = dy;
    a.c_blocks = (g.C + 31) / 32;
    a.groups = a.taps * a.c_blocks;
    a.m_tiles = (a.groups + 3) / 4;
    a.block_n = g.Co > 64 ? 128 : (g.Co > 32 ? 64 : 32);
    a.n_tiles = (g.Co + a.block_n - 1) / a.block_n;
    a.tiled = a.taps == 1 && g.sh == 1 && g.sw == 1;
    a.pixel_blocks = (int)((pixels + 31) / 32);
    a.dev_status = ctx->dev_status;
    // One wave of CTAs; a slice has at least 4 blocks of 32 pixels, and at most 32 (1024 additions per 8 products keep
    // the rounding of the accumulator below 1e-6), the latter while the partial sums stay smaller than the operands.
    const int64_t units = (int64_t)a.m_tiles * a.n_tiles, elems = (int64_t)a.taps * g.C * g.Co;
    int64_t slices = ctx->sm_count / units;
    if (slices < (a.pixel_blocks + 31) / 32) {
        int64_t more = (a.pixel_blocks + 31) / 32;
        const int64_t most = pixels * (g.C + g.Co) / elems + 1;
        if (more > most) more = most;
        if (slices < more) slices = (more * units + ctx->sm_count - 1) / ctx->sm_count * ctx->sm_count / units;
    }
    if (slices > (a.pixel_blocks + 3) / 4) slices = (a.pixel_blocks + 3) / 4;
    if (slices < 1) slices = 1;
    slices = scratch_parts(ctx->scratch_c, slices, (size_t)elems * 4, s);
    a.blocks_per_slice = (int)((a.pixel_blocks + slices - 1) / slices);
    slices = (a.pixel_blocks + a.blocks_per_slice - 1) / a.blocks_per_slice;
    a.segment = split_segment((int64_t)a.blocks_per_slice * 32);
    const int raw_bytes = (4 + a.block_n / 32) * GROUP_BYTES, halves = split ? 2 : 1;
    a.stages = (CG_SMEM - 1024 - EPI_WARPS * EPI_SLAB_BYTES) / (halves * raw_bytes);
    if (a.stages > CG_MAX_STAGES) a.stages = CG_MAX_STAGES;
    tfjsb_status st;
    float* out = df;
    if (slices > 1) {
        if ((st = ensure_scratch(ctx, &ctx->scratch_c, (size_t)slices * elems * 4)) != TFJSB_OK) return st;
        out = ctx->scratch_c.ptr;
    }
    CUtensorMap map_x, map_dy, map_out;
    const uint32_t box[3] = {32u, 32u, 1u};
    if (a.tiled) {
        const int64_t d[2] = {g.C, pixels};
        if ((st = encode_tile_map(ctx, &map_x, x, 2, d, box, "x", CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B)) != TFJSB_OK) return st;
    } else {
        const int lower[2] = {-g.pl, -g.pt};
        const int upper[2] = {(g.Wo - 1) * g.sw - g.pl - (g.W - 1), (g.Ho - 1) * g.sh - g.pt - (g.H - 1)};
        if ((st = encode_im2col(ctx, &map_x, x, g.N, g.H, g.W, g.C, lower, upper, g.sw, g.sh, 32, "x", CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B)) != TFJSB_OK) return st;
    }
    const int64_t dd[2] = {g.Co, pixels}, od[3] = {g.Co, g.C, slices * a.taps};
    if ((st = encode_tile_map(ctx, &map_dy, dy, 2, dd, box, "dy", CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B)) != TFJSB_OK) return st;
    if ((st = encode_tile_map(ctx, &map_out, out, 3, od, box, "the filter gradient")) != TFJSB_OK) return st;
    auto kernel = split ? conv2d_grad_filter_kernel<true> : conv2d_grad_filter_kernel<false>;
    cudaError_t e = smem_attr_once(reinterpret_cast<const void*>(kernel), CG_SMEM);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "shared-memory limit");
    const size_t smem = 1024 + (size_t)EPI_WARPS * EPI_SLAB_BYTES + (size_t)a.stages * halves * raw_bytes;
    if ((e = launch_k(kernel, dim3((unsigned)(units * slices)), dim3(split ? CG_THREADS : CG_THREADS - CVT_WARPS * 32), smem, s, map_x, map_dy, map_out, a)) != cudaSuccess)
        return cuda_fail(ctx, e, "conv2d_grad_filter launch");
    ++ctx->launches;
    if (slices > 1 && (e = launch_sum_rows(out, df, nullptr, slices, elems, 1, s, &ctx->launches)) != cudaSuccess)
        return cuda_fail(ctx, e, "partial-sum launch");
    return TFJSB_OK;
}

}  // namespace tfjsb
