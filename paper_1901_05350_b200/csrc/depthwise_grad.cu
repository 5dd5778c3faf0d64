// Filter gradient of the 3x3 depthwise convolution (multiplier 1, stride 1 or 2, C % 4 == 0):
//   df[ky,kx,c] = sum over n,oy,ox of x[n, oy*S - pt + ky, ox*S - pl + kx, c] * dy[n,oy,ox,c].
//
// Bound by memory: x and dy are read once, the result is 9 C values.  The structure is that of the pipelined forward
// kernel (depthwise.cu): persistent CTAs, two per SM, walk tiles of TH x TW output pixels x 32 channels; one thread
// issues two bulk tensor copies per tile (the input patch and the dy tile, both zero-filled outside the image, so no
// bounds are checked in the arithmetic) into a ring of stages; eight compute warps (thread = 4 channels x one output
// column x R rows) slide down the patch rows, each row feeding up to three filter rows.  The grid is a multiple of
// the channel blocks, so a CTA stays on one of them and keeps its nine sums per channel in registers for its whole
// life; it writes them once, and column sums over the CTAs finish.  One block per (tap, slice), re-reading x and dy
// for every tap with 4-byte loads, took 535 + 30 us for [32,56,56,128] (103 MB of input).
#include "common.cuh"
#include "ptx_sm100.cuh"

namespace tfjsb {

namespace {

constexpr int DG_THREADS = 256;           // compute threads
constexpr int DG_ALL_THREADS = DG_THREADS + 32;
constexpr int DG_CB = 32;                 // channels per tile: one 128-byte line per pixel
constexpr int DG_QUADS = DG_CB / 4;
constexpr int DG_MAX_STAGES = 4;
constexpr int DG_SMEM_BUDGET = 100 * 1024;  // two CTAs per SM, beside 10 KB each of static shared memory

template <int S, int TW, int R>
struct DgTile {
    static constexpr int RG = DG_THREADS / DG_QUADS / TW;
    static constexpr int TH = RG * R;
    static constexpr int TWIN = (TW - 1) * S + 3, THIN = (TH - 1) * S + 3;
    static constexpr int X_BYTES = THIN * TWIN * DG_CB * 4;
    static constexpr int DY_BYTES = TH * TW * DG_CB * 4;
    static constexpr int STAGE_BYTES = X_BYTES + DY_BYTES;
};

struct DgTiling {
    int tiles_x, tiles_y, c_blocks, stages, num_tiles;
};

// The tensors themselves, for sums that are not finite.
struct DgTensors {
    const float *x, *dy;
    int H, W, Ho, Wo;
};

// A sum that is not finite once more, over the CTA's tiles: products with samples that do not exist take no part, where
// the zeros that were copied for them make NaNs of infinite values of dy.
__device__ __noinline__ float sum_of_existing(const DgTensors& d, const DgTiling& t, int S, int TH, int TW, int C, int pt, int pl, int c, int tap,
                                              int first, int step) {
    const int off_y = tap / 3 - pt, off_x = tap % 3 - pl;
    float acc = 0.f;
    for (int tile = first; tile < t.num_tiles; tile += step) {
        int q = tile / t.c_blocks;
        const int tx = q % t.tiles_x; q /= t.tiles_x;
        const int ty = q % t.tiles_y;
        const int64_t n = q / t.tiles_y;
        for (int oy = ty * TH; oy < min(d.Ho, (ty + 1) * TH); ++oy)
            for (int ox = tx * TW; ox < min(d.Wo, (tx + 1) * TW); ++ox) {
                const int iy = oy * S + off_y, ix = ox * S + off_x;
                if (iy < 0 || iy >= d.H || ix < 0 || ix >= d.W) continue;
                acc = fmaf(load_global(d.x + ((n * d.H + iy) * d.W + ix) * C + c), load_global(d.dy + ((n * d.Ho + oy) * d.Wo + ox) * C + c), acc);
            }
        if (acc != acc) break;
    }
    return acc;
}

template <int S, int TW, int R>
__global__ void __launch_bounds__(DG_ALL_THREADS, 2)
depthwise3x3_backprop_filter_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_dy,
                                    float* __restrict__ partial, int C, int pt, int pl, const __grid_constant__ DgTiling t,
                                    const __grid_constant__ DgTensors d, unsigned int* dev_status) {
    using T = DgTile<S, TW, R>;
    extern __shared__ uint8_t dg_smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[DG_MAX_STAGES], bar_empty[DG_MAX_STAGES];
    __shared__ float4 red[DG_THREADS / 32][9][DG_QUADS];
    __shared__ int abort_flag_s;
    volatile int* abort_flag = &abort_flag_s;
    const uint32_t smem_base = (ptx::smem_u32(dg_smem_raw) + 127u) & ~127u;
    const uint8_t* smem_p = dg_smem_raw + (smem_base - ptx::smem_u32(dg_smem_raw));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < t.stages; ++s) {
            ptx::mbar_init(ptx::smem_u32(&bar_full[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&bar_empty[s]), DG_THREADS / 32);
        }
        abort_flag_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    ptx::pdl_wait();  // (the next kernel starts as this one ends: two CTAs fit an SM, see DepthwisePlan)
    const int first = blockIdx.x, step = gridDim.x;  // step is a multiple of the channel blocks
    const int my_tiles = first < t.num_tiles ? (t.num_tiles - first + step - 1) / step : 0;
    const int cb = first % t.c_blocks;

    if (warp == DG_THREADS / 32) {
        if (lane == 0) {
            int slot = 0, i = 0;
            uint32_t parity = 0;
            bool ok = true;
            for (; i < my_tiles; ++i) {
                if (!ptx::bounded_wait(ptx::smem_u32(&bar_empty[slot]), parity ^ 1u, abort_flag)) { ok = false; break; }
                int q = (first + i * step) / t.c_blocks;
                const int tx = q % t.tiles_x; q /= t.tiles_x;
                const int ty = q % t.tiles_y;
                const int n = q / t.tiles_y;
                const uint32_t bar = ptx::smem_u32(&bar_full[slot]);
                const uint32_t dst = smem_base + (uint32_t)slot * (uint32_t)T::STAGE_BYTES;
                ptx::mbar_arrive_expect_tx(bar, (uint32_t)T::STAGE_BYTES);
                ptx::tma_load_4d(dst, &map_x, bar, cb * DG_CB, tx * TW * S - pl, ty * T::TH * S - pt, n);
                ptx::tma_load_4d(dst + T::X_BYTES, &map_dy, bar, cb * DG_CB, tx * TW, ty * T::TH, n);
                if (++slot == t.stages) { slot = 0; parity ^= 1u; }
            }
            if (!ok || *abort_flag) {
                if (!*abort_flag) *abort_flag = 1;
                atomicOr(dev_status, DEV_STATUS_TIMEOUT_DEPTHWISE);
                // wait (bounded) for the copies still in flight so nothing lands after the CTA has gone
                for (int k = i - t.stages > 0 ? i - t.stages : 0; k < i; ++k) {
                    const unsigned long long t0 = ptx::global_ns();
                    while (!ptx::mbar_try_wait(ptx::smem_u32(&bar_full[k % t.stages]), (uint32_t)((k / t.stages) & 1))) {
                        if (ptx::global_ns() - t0 > ptx::WAIT_LIMIT_NS) {
                            atomicOr(dev_status, DEV_STATUS_TIMEOUT_DRAIN);
                            break;
                        }
                    }
                }
            }
        }
        return;
    }

    const int c4 = tid % DG_QUADS, col = (tid / DG_QUADS) % TW, rg = tid / (DG_QUADS * TW);
    float4 acc[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    int slot = 0;
    uint32_t parity = 0;
    for (int i = 0; i < my_tiles; ++i) {
        const bool got = ptx::bounded_wait(ptx::smem_u32(&bar_full[slot]), parity, abort_flag);
        if (!__all_sync(0xffffffffu, got)) {
            if (lane == 0) *abort_flag = 1;
            break;
        }
        const float4* xp = reinterpret_cast<const float4*>(smem_p + (size_t)slot * T::STAGE_BYTES) +
                           ((rg * R * S) * T::TWIN + col * S) * DG_QUADS + c4;
        const float4* gp = reinterpret_cast<const float4*>(smem_p + (size_t)slot * T::STAGE_BYTES + T::X_BYTES) +
                           (rg * R * TW + col) * DG_QUADS + c4;
        float4 gy[R];
#pragma unroll
        for (int r = 0; r < R; ++r) gy[r] = gp[r * TW * DG_QUADS];
        constexpr int IN_ROWS = (R - 1) * S + 3;
#pragma unroll
        for (int j = 0; j < IN_ROWS; ++j) {
            const float4* row = xp + j * T::TWIN * DG_QUADS;
            const float4 v0 = row[0], v1 = row[DG_QUADS], v2 = row[2 * DG_QUADS];
#pragma unroll
            for (int ky = 0; ky < 3; ++ky) {
                const int d = j - ky;
                if (d >= 0 && d % S == 0 && d / S < R) {
                    fma4_packed(acc[ky * 3 + 0], v0, gy[d / S]);
                    fma4_packed(acc[ky * 3 + 1], v1, gy[d / S]);
                    fma4_packed(acc[ky * 3 + 2], v2, gy[d / S]);
                }
            }
        }
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&bar_empty[slot]));
        if (++slot == t.stages) { slot = 0; parity ^= 1u; }
    }
    // four output columns of a warp share a channel quad; then the eight warps
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        float* v = reinterpret_cast<float*>(&acc[k]);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            v[e] += __shfl_xor_sync(0xffffffffu, v[e], 8);
            v[e] += __shfl_xor_sync(0xffffffffu, v[e], 16);
        }
        if (lane < DG_QUADS) red[warp][k][lane] = acc[k];
    }
    asm volatile("bar.sync 1, %0;" ::"n"(DG_THREADS) : "memory");  // the compute warps
    const int c = cb * DG_CB + (tid % DG_QUADS) * 4;
    if (tid < 9 * DG_QUADS && c < C) {
        const int k = tid / DG_QUADS;
        float4 s = red[0][k][tid % DG_QUADS];
#pragma unroll
        for (int w = 1; w < DG_THREADS / 32; ++w) {
            const float4 v = red[w][k][tid % DG_QUADS];
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        if (!finite4(s)) {
            float* v = &s.x;
            for (int e = 0; e < 4; ++e)
                if (!isfinite(v[e])) v[e] = sum_of_existing(d, t, S, T::TH, TW, C, pt, pl, c + e, k, first, step);
        }
        *reinterpret_cast<float4*>(partial + ((int64_t)(first / t.c_blocks) * 9 + k) * C + c) = s;
    }
}

template <int S, int TW, int R>
void fill(DepthwiseGradPlan* p) {
    using T = DgTile<S, TW, R>;
    p->th = T::TH; p->tw = TW; p->thin = T::THIN; p->twin = T::TWIN; p->stage_bytes = T::STAGE_BYTES;
}

template <int S, int TW, int R>
cudaError_t launch_instance(const DepthwiseGradPlan& p, float* out, unsigned int* dev_status, cudaStream_t s) {
    auto kernel = depthwise3x3_backprop_filter_kernel<S, TW, R>;
    cudaError_t e = smem_attr_once(reinterpret_cast<const void*>(kernel), DG_SMEM_BUDGET);
    if (e != cudaSuccess) return e;
    const DgTiling t{p.tiles_x, p.tiles_y, p.c_blocks, p.stages, p.num_tiles};
    const DgTensors d{p.x, p.dy, p.g.H, p.g.W, p.g.Ho, p.g.Wo};
    return launch_k(kernel, dim3(p.slices * p.c_blocks), dim3(DG_ALL_THREADS), (size_t)p.stages * p.stage_bytes + 128, s, p.map_x, p.map_dy,
                    out, p.g.C, p.g.pt, p.g.pl, t, d, dev_status);
}

bool encode_nhwc(tfjsb_ctx* ctx, CUtensorMap* map, const float* base, int64_t n, int h, int w, int c, int box_h, int box_w) {
    cuuint64_t dims[4] = {(cuuint64_t)c, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)n};
    cuuint64_t strides[3] = {(cuuint64_t)c * 4, (cuuint64_t)w * c * 4, (cuuint64_t)h * w * c * 4};
    cuuint32_t box[4] = {DG_CB, (cuuint32_t)box_w, (cuuint32_t)box_h, 1u};
    cuuint32_t elem[4] = {1u, 1u, 1u, 1u};
    return ctx->encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float*>(base), dims, strides, box, elem,
                             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool depthwise_grad_plan(tfjsb_ctx* ctx, const float* x, const float* dy, const ConvGeom& g, DepthwiseGradPlan* p) {
    if (g.fh != 3 || g.fw != 3 || g.mult != 1 || g.sh != g.sw || g.sh > 2 || g.dh != 1 || g.dw != 1 || g.C % 4 != 0 || !ctx->encode_tiled)
        return false;
    p->g = g;
    p->x = x; p->dy = dy;
    // eight columns per tile where that wastes fewer of them
    const bool narrow = (g.Wo + 7) / 8 * 8 < (g.Wo + 15) / 16 * 16;
    p->variant = (g.sh == 1 ? 0 : 2) + (narrow ? 1 : 0);
    switch (p->variant) {
        case 0: fill<1, 16, 4>(p); break;
        case 1: fill<1, 8, 2>(p); break;
        case 2: fill<2, 16, 2>(p); break;
        default: fill<2, 8, 2>(p); break;
    }
    p->tiles_x = (g.Wo + p->tw - 1) / p->tw;
    p->tiles_y = (g.Ho + p->th - 1) / p->th;
    p->c_blocks = (g.C + DG_CB - 1) / DG_CB;
    const int64_t spatial = (int64_t)p->tiles_x * p->tiles_y * g.N;
    if (spatial * p->c_blocks > 0x7fffffff) return false;  // tile indices are 32-bit in the kernel
    p->num_tiles = (int)(spatial * p->c_blocks);
    p->stages = DG_SMEM_BUDGET / p->stage_bytes;
    if (p->stages > DG_MAX_STAGES) p->stages = DG_MAX_STAGES;
    // two CTAs per SM, the same number of them on every channel block
    int64_t slices = 2 * (int64_t)ctx->sm_count / p->c_blocks;
    if (slices < 1) slices = 1;
    p->slices = (int)(slices < spatial ? slices : spatial);
    return encode_nhwc(ctx, &p->map_x, x, g.N, g.H, g.W, g.C, p->thin, p->twin) &&
           encode_nhwc(ctx, &p->map_dy, dy, g.N, g.Ho, g.Wo, g.C, p->th, p->tw);
}

cudaError_t launch_depthwise_grad(const DepthwiseGradPlan& p, float* df, float* partial, unsigned int* dev_status, cudaStream_t s,
                                  int64_t* launches) {
    float* out = p.slices > 1 ? partial : df;
    cudaError_t e;
    switch (p.variant) {
        case 0: e = launch_instance<1, 16, 4>(p, out, dev_status, s); break;
        case 1: e = launch_instance<1, 8, 2>(p, out, dev_status, s); break;
        case 2: e = launch_instance<2, 16, 2>(p, out, dev_status, s); break;
        default: e = launch_instance<2, 8, 2>(p, out, dev_status, s); break;
    }
    ++*launches;
    if (e != cudaSuccess || p.slices == 1) return e;
    return launch_sum_rows(partial, df, nullptr, p.slices, 9 * (int64_t)p.g.C, 1, s, launches);
}

}  // namespace tfjsb
