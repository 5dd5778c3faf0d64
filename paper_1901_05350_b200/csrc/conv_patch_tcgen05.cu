// 3x3 convolution with stride 1 on the tensor cores (tcgen05) from input patches: conv2d forward, and its gradient with respect
// to the input, which is the same sum over dy with the taps reversed.
//
//     y[n, oy, ox, co] = act( sum over taps (ky, kx) and channels c of  x[n, oy + ky - pt, ox + kx - pl, c] . w[tap, c, co] + bias )
//
// A tile is 16 x 8 output pixels (the 128 rows of a tensor-core tile: 16 groups of 8 neighbours along W).  For 32 channels
// the input patch that all taps of the tile read, 18 x 10 pixels of 128 bytes, is copied once, with the 128-byte swizzle.  The
// A operand of a tap is then that patch from a pixel on: a K-major tile of 8-pixel groups whose start is shifted by the tap and
// whose groups are one patch row apart (the stride byte offset).  The swizzle works on addresses, so any start is a valid one,
// and as fast: 41, 49, 66 and 129 cycles per MMA of 32, 64, 128 and 256 columns wherever it starts.  Im2col copies bring the
// same pixels nine times, 128 of them in about 600 cycles.
//   warp 0       producer of patches
//   warp 1       MMA issuer
//   warp 2       producer of filter tiles [32 k x block_n], one per (channel block, tap); a filter that fits stays in shared
//                memory for the whole kernel
//   warp 3       tensor memory
//   warps 4-11   epilogue
// The forward filter [tap][Cin][Cout] is read as it is stored (MN-major tiles), the gradient's [tap][Cin][Cout] too (its
// summed index, Cout, is the contiguous one: K-major tiles), so nothing is packed.
// One thread issues everything, and every instruction around its MMAs counts: the nine taps are unrolled, an operand is the low
// word of its descriptor, worked out by the converged warp, and tiles are stepped without divisions (with the window as a loop
// and descriptors inside the elected thread's branch a tap took 880 cycles).
// What bounds it: two to four patches in flight per SM and the copies and stores of single pixels; [64,56,56,64] -> 64 takes 372
// cycles a tap where its MMAs take 196.
//
// SPLIT (gradients): fp32 accuracy from TF32 products as in conv_grad_tcgen05.cu: every operand tile has a lo tile beside it,
// made by warps 12-23 (four for patches, eight for filter tiles), three products per 8 of k, large products summed in
// segments.  A patch is split once and not once per tap.  24 warps leave a thread 80 registers; it spills 124 bytes.
// Every wait is bounded (ptx_sm100.cuh).
#include <algorithm>
#include <cstdlib>

#include "common.cuh"
#include "ptx_sm100.cuh"
#include "umma_tile.cuh"

namespace tfjsb {

using namespace ptx;
using namespace tile;

namespace {

constexpr int PC_TH = 16, PC_TW = 8;  // output pixels of a tile
constexpr int PC_PH = PC_TH + 2, PC_PW = PC_TW + 2, PC_TAPS = 9;
constexpr int PC_PATCH_BYTES = PC_PH * PC_PW * 128, PC_PATCH_STRIDE = (PC_PATCH_BYTES + 1023) / 1024 * 1024;
constexpr int PC_EPI_WARPS = 8, PC_SPLIT_P = 4, PC_SPLIT_B = 8;
constexpr int PC_MAX_PATCHES = 4, PC_MAX_B = 40;
constexpr int pc_threads(bool split) { return (4 + PC_EPI_WARPS + (split ? PC_SPLIT_P + PC_SPLIT_B : 0)) * 32; }

// A tile's coordinates, fastest first: part of the K loop, column tile, column and row of the image, image.
struct TileDigits {
    int split, nt, tx, ty, img;
};
struct PatchConvArgs {
    int C, Co, Ho, Wo;           // channels summed over, output channels, output size
    int H, W;                    // of x
    int pt, pl;
    int tiles_x, tiles_y, n_tiles, splits, num_tiles;
    TileDigits step;             // gridDim.x in the tiles' digits
    int images;
    int c_blocks, block_n, acc_stages;
    int patch_stages, b_stages, b_resident;
    int segment;                 // k-blocks per accumulator of the large products (SPLIT)
    const float *x, *w;          // for results that are not finite (SPLIT)
    const float* bias;
    int act;
    unsigned int* dev_status;
};

TileDigits tile_digits(int t, int splits, int n_tiles, int tiles_x, int tiles_y) {
    TileDigits d;
    d.split = t % splits; t /= splits;
    d.nt = t % n_tiles; t /= n_tiles;
    d.tx = t % tiles_x; t /= tiles_x;
    d.ty = t % tiles_y;
    d.img = t / tiles_y;
    return d;
}

// The tiles of a CTA one after the other.
struct PatchTile {
    TileDigits at;
    int index, cb_begin, cb_end;
    __device__ __forceinline__ explicit PatchTile(const PatchConvArgs& g) : index((int)blockIdx.x) {
        int t = index;
        at.split = t % g.splits; t /= g.splits;
        at.nt = t % g.n_tiles; t /= g.n_tiles;
        at.tx = t % g.tiles_x; t /= g.tiles_x;
        at.ty = t % g.tiles_y;
        at.img = t / g.tiles_y;
        part(g);
    }
    __device__ __forceinline__ void part(const PatchConvArgs& g) {
        cb_begin = 0;
        cb_end = g.c_blocks;
        if (g.splits > 1) {
            cb_begin = g.c_blocks * at.split / g.splits;
            cb_end = g.c_blocks * (at.split + 1) / g.splits;
        }
    }
    __device__ __forceinline__ bool live(const PatchConvArgs& g) const { return index < g.num_tiles; }
    __device__ __forceinline__ void next(const PatchConvArgs& g) {
        index += (int)gridDim.x;
        at.split += g.step.split; at.nt += g.step.nt; at.tx += g.step.tx; at.ty += g.step.ty; at.img += g.step.img;
        if (at.split >= g.splits) { at.split -= g.splits; ++at.nt; }
        if (at.nt >= g.n_tiles) { at.nt -= g.n_tiles; ++at.tx; }
        if (at.tx >= g.tiles_x) { at.tx -= g.tiles_x; ++at.ty; }
        if (at.ty >= g.tiles_y) { at.ty -= g.tiles_y; ++at.img; }
        part(g);
    }
    __device__ __forceinline__ int n0(const PatchConvArgs& g) const { return at.nt * g.block_n; }
    __device__ __forceinline__ int x0() const { return at.tx * PC_TW; }
    __device__ __forceinline__ int y0() const { return at.ty * PC_TH; }
};

// D[tmem] (+)= A . B^T with the descriptors' words apart: the high ones are constants.
__device__ __forceinline__ void mma_words(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "mov.b64 a, {%1, %2};\n\t"
        "mov.b64 b, {%3, %4};\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], a, b, %5, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}

// One result of a tile once more by fp32 multiply-adds, over the samples that exist (in the copied patches those outside the
// image are zeros, which an infinite filter value turns into NaN).
__device__ __noinline__ float patch_conv_in_fp32(const PatchConvArgs& g, const PatchTile& r, int oy, int ox, int co) {
    float acc = 0.f;
    for (int tap = 0; tap < PC_TAPS; ++tap) {
        const int iy = oy + tap / 3 - g.pt, ix = ox + tap % 3 - g.pl;
        if (iy < 0 || iy >= g.H || ix < 0 || ix >= g.W) continue;
        const float* x = g.x + (((long long)r.at.img * g.H + iy) * g.W + ix) * g.C;
        const float* w = g.w + ((long long)(PC_TAPS - 1 - tap) * g.Co + co) * g.C;
        for (int c = r.cb_begin * BLOCK_K; c < min(r.cb_end * BLOCK_K, g.C); ++c) acc = fmaf(load_global(x + c), load_global(w + c), acc);
        if (acc != acc) break;
    }
    return acc;
}

template <bool SPLIT>
__global__ void __launch_bounds__(pc_threads(SPLIT), 1)
conv_patch_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
                  const __grid_constant__ CUtensorMap map_y, const __grid_constant__ PatchConvArgs g) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_p_full[PC_MAX_PATCHES], bar_p_empty[PC_MAX_PATCHES], bar_p_split[PC_MAX_PATCHES];
    __shared__ __align__(8) uint64_t bar_b_full[PC_MAX_B], bar_b_empty[PC_MAX_B], bar_b_split[PC_MAX_B];
    __shared__ __align__(8) uint64_t bar_acc_full[MAX_ACC_STAGES], bar_acc_empty[MAX_ACC_STAGES], bar_small_empty, bar_drain;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag_s;
    volatile int* abort_flag = &abort_flag_s;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr uint32_t HALVES = SPLIT ? 2 : 1;
    const uint32_t b_bytes = (uint32_t)g.block_n * 128u;
    // dynamic shared memory: [epilogue slabs][patches, each hi | lo][filter tiles, each hi | lo]
    const uint32_t epi_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t patch_base = epi_base + PC_EPI_WARPS * EPI_SLAB_BYTES;
    const uint32_t b_base = patch_base + (uint32_t)(g.patch_stages * PC_PATCH_STRIDE) * HALVES;
    auto patch_addr = [&](int s) { return patch_base + (uint32_t)(s * PC_PATCH_STRIDE) * HALVES; };
    auto b_addr = [&](int s) { return b_base + (uint32_t)s * b_bytes * HALVES; };

    if (threadIdx.x == 0) {
        for (int s = 0; s < g.patch_stages; ++s) {
            mbar_init(smem_u32(&bar_p_full[s]), 1);
            mbar_init(smem_u32(&bar_p_empty[s]), 1);
            mbar_init(smem_u32(&bar_p_split[s]), PC_SPLIT_P);
        }
        for (int s = 0; s < g.b_stages; ++s) {
            mbar_init(smem_u32(&bar_b_full[s]), 1);
            mbar_init(smem_u32(&bar_b_empty[s]), 1);
            mbar_init(smem_u32(&bar_b_split[s]), PC_SPLIT_B);
        }
        for (int s = 0; s < MAX_ACC_STAGES; ++s) {
            mbar_init(smem_u32(&bar_acc_full[s]), 1);
            mbar_init(smem_u32(&bar_acc_empty[s]), PC_EPI_WARPS);
        }
        mbar_init(smem_u32(&bar_small_empty), PC_EPI_WARPS);
        mbar_init(smem_u32(&bar_drain), 1);
        abort_flag_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_x) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_w) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_y) : "memory");
    }
    uint32_t tmem_cols = 32;  // SPLIT: [large 0 | large 1 | small | sum]
    while (tmem_cols < (uint32_t)((SPLIT ? 4 : g.acc_stages) * g.block_n)) tmem_cols <<= 1;
    if (warp == 3) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    pdl_launch_dependents();
    pdl_wait();

    if (warp == 0) {
        // ---------------------------------------------------------------- patches
        int ps = 0, filled = 0;
        uint32_t phase = 0;
        const bool leader = elect_one();
        bool ok = true;  // the leader's
        for (PatchTile r(g); r.live(g); r.next(g)) {
            for (int cb = r.cb_begin; cb < r.cb_end; ++cb) {
                if (leader && ok && (ok = bounded_wait(smem_u32(&bar_p_empty[ps]), phase ^ 1u, abort_flag))) {
                    const uint32_t full = smem_u32(&bar_p_full[ps]);
                    mbar_arrive_expect_tx(full, (uint32_t)PC_PATCH_BYTES);
                    tma_load_4d(patch_addr(ps), &map_x, full, cb * BLOCK_K, r.x0() - g.pl, r.y0() - g.pt, r.at.img);
                    ++filled;
                }
                if (++ps == g.patch_stages) { ps = 0; phase ^= 1u; }
            }
        }
        if (!ok) {
            give_up(abort_flag, g.dev_status, DEV_STATUS_TIMEOUT_PRODUCER);
            for (int k = filled > g.patch_stages ? filled - g.patch_stages : 0; k < filled; ++k)
                drain(smem_u32(&bar_p_full[k % g.patch_stages]), (uint32_t)((k / g.patch_stages) & 1), g.dev_status);
        }
        __syncwarp();
    } else if (warp == 2) {
        // ---------------------------------------------------------------- filter tiles
        int bs = 0, filled = 0;
        uint32_t phase = 0;
        const bool leader = elect_one();
        bool ok = true;  // the leader's
        for (PatchTile r(g); r.live(g); r.next(g)) {
            if (g.b_resident && r.index != (int)blockIdx.x) break;  // loaded with the first tile
            for (int cb = r.cb_begin; cb < r.cb_end; ++cb)
                for (int tap = 0; tap < PC_TAPS; ++tap) {
                    const int wt = SPLIT ? PC_TAPS - 1 - tap : tap;
                    if (leader && ok && (ok = bounded_wait(smem_u32(&bar_b_empty[bs]), phase ^ 1u, abort_flag))) {
                        const uint32_t full = smem_u32(&bar_b_full[bs]);
                        mbar_arrive_expect_tx(full, b_bytes);
                        if (!SPLIT) {  // [tap][C][Co]: MN-major; the gradient's [tap][Co][C]: K-major
#pragma unroll 1
                            for (int i = 0; i < g.block_n >> 5; ++i)
                                tma_load_3d(b_addr(bs) + (uint32_t)i * 4096u, &map_w, full, r.n0(g) + 32 * i, cb * BLOCK_K, wt);
                        } else {
                            tma_load_3d(b_addr(bs), &map_w, full, cb * BLOCK_K, r.n0(g), wt);
                        }
                        ++filled;
                    }
                    if (++bs == g.b_stages) { bs = 0; phase ^= 1u; }
                }
        }
        if (!ok) {
            give_up(abort_flag, g.dev_status, DEV_STATUS_TIMEOUT_PRODUCER);
            for (int k = filled > g.b_stages ? filled - g.b_stages : 0; k < filled; ++k)
                drain(smem_u32(&bar_b_full[k % g.b_stages]), (uint32_t)((k / g.b_stages) & 1), g.dev_status);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA issuer
        constexpr bool B_MN = !SPLIT;
        const uint32_t idesc = make_idesc_tf32(BLOCK_M, g.block_n) | (B_MN ? IDESC_B_MN : 0u);
        // descriptor words (see make_kmajor_sw128_desc, make_mnmajor_desc); A: groups of eight rows a patch row apart
        constexpr uint32_t A_HI = (uint32_t)(PC_PW * 128 >> 4) | 1u << 14 | 2u << 29;
        constexpr uint32_t B_HI = (uint32_t)((B_MN ? 512 : 1024) >> 4) | 1u << 14 | (B_MN ? 1u : 2u) << 29, B_LO = B_MN ? (4096u >> 4) << 16 : 0u;
        constexpr uint32_t B_STEP = B_MN ? 64 : 2, A_SMALL = PC_PATCH_STRIDE >> 4;
        const uint32_t b_units = b_bytes >> 4, b_first = (b_base >> 4) | B_LO;
        const uint32_t small = tmem + (uint32_t)(2 * g.block_n);
        const bool resident = g.b_resident != 0;
        int ps = 0, bs = 0, acc = 0, in_seg = 0;
        uint32_t p_phase = 0, b_phase = 0, acc_phase = 0, small_phase = 0;
        const bool leader = elect_one();
        bool ok = true, issued = false;  // the leader's
        bool wait_b = true;
        for (PatchTile r(g); r.live(g); r.next(g)) {
            if (leader && ok) {
                if (SPLIT) ok = bounded_wait(smem_u32(&bar_small_empty), small_phase ^ 1u, abort_flag);  // the tile before has been added up
                else ok = bounded_wait(smem_u32(&bar_acc_empty[acc]), acc_phase ^ 1u, abort_flag);
            }
            small_phase ^= 1u;
            uint32_t begun = 0;  // whether the tile's accumulator (SPLIT: of the small products) holds anything
            for (int cb = r.cb_begin; cb < r.cb_end; ++cb) {
                const bool last_cb = cb + 1 == r.cb_end;
                if (leader && ok) {
                    ok = bounded_wait(smem_u32(&bar_p_full[ps]), p_phase, abort_flag);
                    if (SPLIT && ok) ok = bounded_wait(smem_u32(&bar_p_split[ps]), p_phase, abort_flag);
                    tc_fence_after();
                }
                const uint32_t patch = patch_addr(ps) >> 4;
#pragma unroll
                for (int tap = 0; tap < PC_TAPS; ++tap) {
                    const uint32_t a = patch + (uint32_t)((tap / 3 * PC_PW + tap % 3) * 8), b = b_first + (uint32_t)bs * b_units * HALVES;
                    const uint32_t d = tmem + (uint32_t)(acc * g.block_n), large_begun = SPLIT ? (in_seg != 0 ? 1u : 0u) : begun;
                    const uint32_t b_full = smem_u32(&bar_b_full[bs]), b_split = smem_u32(&bar_b_split[bs]), b_empty = smem_u32(&bar_b_empty[bs]);
                    const bool close = (last_cb && tap + 1 == PC_TAPS) || (SPLIT && in_seg + 1 == g.segment);
                    if (leader && ok) {
                        if (SPLIT && in_seg == 0) ok = bounded_wait(smem_u32(&bar_acc_empty[acc]), acc_phase ^ 1u, abort_flag);
                        if (wait_b && ok) {
                            ok = bounded_wait(b_full, b_phase, abort_flag);
                            if (SPLIT && ok) ok = bounded_wait(b_split, b_phase, abort_flag);
                        }
                        if (ok) {
                            if (wait_b || SPLIT) tc_fence_after();
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                mma_words(d, a + 2 * k, A_HI, b + B_STEP * k, B_HI, idesc, k == 0 ? large_begun : 1u);
                                if (SPLIT) {
                                    mma_words(small, a + 2 * k, A_HI, b + b_units + B_STEP * k, B_HI, idesc, k == 0 ? begun : 1u);
                                    mma_words(small, a + A_SMALL + 2 * k, A_HI, b + B_STEP * k, B_HI, idesc, 1u);
                                }
                            }
                            issued = true;
                            if (!resident) tc_commit(b_empty);
                            if (tap + 1 == PC_TAPS) tc_commit(smem_u32(&bar_p_empty[ps]));
                            if (close) tc_commit(smem_u32(&bar_acc_full[acc]));
                        }
                    }
                    begun = 1u;
                    ++in_seg;
                    if (close) {
                        in_seg = 0;
                        if (++acc == (SPLIT ? 2 : g.acc_stages)) { acc = 0; acc_phase ^= 1u; }
                    }
                    if (++bs == g.b_stages) { bs = 0; b_phase ^= 1u; }
                }
                if (++ps == g.patch_stages) { ps = 0; p_phase ^= 1u; }
            }
            if (resident) wait_b = false;
        }
        if (!ok) {
            give_up(abort_flag, g.dev_status, DEV_STATUS_TIMEOUT_MMA);
            if (issued) {
                tc_commit(smem_u32(&bar_drain));
                drain(smem_u32(&bar_drain), 0u, g.dev_status);
            }
        }
        __syncwarp();
    } else if (warp >= 4 && warp < 4 + PC_EPI_WARPS) {
        // ---------------------------------------------------------------- epilogue
        // Two warps per lane quadrant (32 rows of the accumulator: 4 x 8 pixels).  They take 32-column chunks of the result in turn;
        // SPLIT halves the columns of every segment between them (the 32 columns of a narrow tile go to the first).
        const int quad = warp & 3, half = (warp - 4) >> 2;
        const uint32_t slab = epi_base + (uint32_t)(warp - 4) * EPI_SLAB_BYTES;
        const uint32_t lanes = tmem + ((uint32_t)(quad * 32) << 16);
        int acc = 0;
        uint32_t acc_phase = 0;
        bool ok = true;
        int turn = half;  // the first chunk of this warp: with an odd number of chunks the two warps take turns
        for (PatchTile r(g); ok && r.live(g); r.next(g)) {
            const int n0 = r.n0(g), row0 = r.y0() + quad * 4, live = min(g.block_n, g.Co - n0);
            const bool rows_live = row0 < g.Ho;
            uint32_t result;  // the columns that hold it
            if (SPLIT) {
                const int kbs = (r.cb_end - r.cb_begin) * PC_TAPS, cols = g.block_n > 32 ? g.block_n / 2 : half == 0 ? 32 : 0;
                const uint32_t mine = (uint32_t)(half * cols);
                for (int kb = 0; kb < kbs; kb += g.segment) {
                    const bool got = bounded_wait(smem_u32(&bar_acc_full[acc]), acc_phase, abort_flag), last = kb + g.segment >= kbs;
                    if (!(ok = __all_sync(0xffffffffu, got))) break;
                    tc_fence_after();
                    add_segment<16>(lanes + (uint32_t)(acc * g.block_n) + mine, lanes + (uint32_t)(2 * g.block_n) + mine,
                                    lanes + (uint32_t)(3 * g.block_n) + mine, cols, kb == 0, last);
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&bar_acc_empty[acc]));
                    if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
                }
                result = lanes + (uint32_t)(3 * g.block_n);
            } else {
                const bool got = bounded_wait(smem_u32(&bar_acc_full[acc]), acc_phase, abort_flag);
                ok = __all_sync(0xffffffffu, got);
                tc_fence_after();
                result = lanes + (uint32_t)(acc * g.block_n);
            }
            if (!ok) {
                if (lane == 0) give_up(abort_flag, g.dev_status, DEV_STATUS_TIMEOUT_EPILOGUE);
                break;
            }
            // SPLIT: a warp stores the chunks whose columns it has added
            const int chunks = (live + EPI_COLS - 1) / EPI_COLS, per_half = g.block_n / 64;
            const int c_first = SPLIT ? half * per_half : turn, c_step = SPLIT ? 1 : 2;
            if (chunks & 1) turn ^= 1;
            const int c_last = !SPLIT ? chunks : g.block_n == 32 ? (half == 0 ? chunks : 0) : min(chunks, c_first + per_half);
            bool released = false;
            for (int ch = c_first; ch < c_last; ch += c_step) {
                uint32_t u[32];
                tc_ld_32x32(result + (uint32_t)(ch * EPI_COLS), u);
                tc_ld_wait();
                if (ch + c_step >= c_last) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(SPLIT ? smem_u32(&bar_small_empty) : smem_u32(&bar_acc_empty[acc]));
                    released = true;
                }
                if (!rows_live) continue;
                const int col0 = n0 + ch * EPI_COLS;
                if (lane == 0) tma_store_wait_read<0>();
                __syncwarp();
                const float* bias = !SPLIT && g.bias != nullptr ? g.bias + col0 : nullptr;
                const uint32_t row_addr = slab + (uint32_t)lane * 128u;
                if (SPLIT) stage_chunk<TFJSB_ACT_NONE>(u, nullptr, 0, row_addr, lane);  // a gradient has neither
                else if (g.act == TFJSB_ACT_RELU6) stage_chunk<TFJSB_ACT_RELU6>(u, bias, g.Co - col0, row_addr, lane);
                else if (g.act == TFJSB_ACT_RELU) stage_chunk<TFJSB_ACT_RELU>(u, bias, g.Co - col0, row_addr, lane);
                else stage_chunk<TFJSB_ACT_NONE>(u, bias, g.Co - col0, row_addr, lane);
                if (SPLIT) {
                    const int oy = row0 + (lane >> 3), ox = r.x0() + (lane & 7);
                    bool odd = false;
#pragma unroll
                    for (int e = 0; e < 32; ++e) odd = odd || not_finite(u[e]);
                    for (int e = 0; odd && oy < g.Ho && ox < g.Wo && e < min(32, g.Co - col0); ++e) {
                        const uint32_t at = row_addr + (uint32_t)((((e >> 2) ^ (lane & 7)) << 4) + (e & 3) * 4);
                        uint32_t bits;
                        asm volatile("ld.shared.b32 %0, [%1];" : "=r"(bits) : "r"(at) : "memory");
                        if (!not_finite(bits)) continue;
                        const float v = patch_conv_in_fp32(g, r, oy, ox, col0 + e);
                        asm volatile("st.shared.f32 [%0], %1;" ::"r"(at), "f"(v) : "memory");
                    }
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    tma_store_4d(&map_y, slab, col0, r.x0(), row0, r.at.split * g.images + r.at.img);
                    tma_store_commit();
                }
            }
            if (!released) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(SPLIT ? smem_u32(&bar_small_empty) : smem_u32(&bar_acc_empty[acc]));
            }
            if (!SPLIT && ++acc == g.acc_stages) { acc = 0; acc_phase ^= 1u; }
        }
        if (lane == 0) tma_store_wait_all();
        __syncwarp();
    } else if (SPLIT && warp >= 4 + PC_EPI_WARPS) {
        // ---------------------------------------------------------------- lo tiles
        const int sw = warp - 4 - PC_EPI_WARPS;
        const bool patches = sw < PC_SPLIT_P;
        const uint32_t mine = (uint32_t)((patches ? sw : sw - PC_SPLIT_P) * 32 + lane) * 16u;
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        const int stages = patches ? g.patch_stages : g.b_stages, bytes = patches ? PC_PATCH_BYTES : (int)b_bytes;
        const int step = (patches ? PC_SPLIT_P : PC_SPLIT_B) * 512;
        const uint32_t lo_offset = patches ? (uint32_t)PC_PATCH_STRIDE : b_bytes, round = patches ? SPLIT_UP : SPLIT_NEAREST;
        for (PatchTile r(g); ok && r.live(g); r.next(g)) {
            if (!patches && g.b_resident && r.index != (int)blockIdx.x) break;
            const int turns = (r.cb_end - r.cb_begin) * (patches ? 1 : PC_TAPS);
            for (int k = 0; k < turns; ++k) {
                const bool got = bounded_wait(patches ? smem_u32(&bar_p_full[stage]) : smem_u32(&bar_b_full[stage]), phase, abort_flag);
                if (!__all_sync(0xffffffffu, got)) {
                    if (lane == 0) give_up(abort_flag, g.dev_status, DEV_STATUS_TIMEOUT_PRODUCER);
                    ok = false;
                    break;
                }
                const uint32_t src = (patches ? patch_addr(stage) : b_addr(stage)) + mine;
#pragma unroll 4
                for (int o = 0; o < bytes - (int)mine; o += step) {
                    const float4 v = lds4(src + (uint32_t)o);
                    sts4(src + lo_offset + (uint32_t)o, tf32_rest(v.x, round), tf32_rest(v.y, round), tf32_rest(v.z, round), tf32_rest(v.w, round));
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(patches ? smem_u32(&bar_p_split[stage]) : smem_u32(&bar_b_split[stage]));
                if (++stage == stages) { stage = 0; phase ^= 1u; }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 3) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
    }
}

constexpr int PC_SMEM = SMEM_LIMIT - 2048;  // beside the barriers

// Tile width, rings and shared memory for a geometry (as the sum is written above: of the input gradient, the transposed one).
struct PatchTiling {
    int block_n = 0, splits = 1, patch_stages = 0, b_stages = 0, c_blocks = 0, n_tiles = 0;
    bool resident = false;
    int64_t pixel_tiles = 0, tiles = 0;
    double us = 0;  // estimate, to choose between widths and kernels only
};

bool rings_fit(PatchTiling* t, bool split) {
    const int halves = split ? 2 : 1, room = PC_SMEM - 1024 - PC_EPI_WARPS * EPI_SLAB_BYTES;
    const int patch = PC_PATCH_STRIDE * halves, b = t->block_n * 128 * halves;
    const int64_t all = (int64_t)t->c_blocks * PC_TAPS;  // filter tiles in all
    t->resident = t->n_tiles == 1 && t->splits == 1 && all <= PC_MAX_B && 2 * patch + all * b <= room;
    if (t->resident) {
        t->b_stages = (int)all;
        t->patch_stages = std::min(PC_MAX_PATCHES, (room - (int)all * b) / patch);
        return true;
    }
    t->patch_stages = split ? 2 : 3;
    if (t->patch_stages * patch + 3 * b > room) t->patch_stages = 2;
    t->b_stages = std::min(8, (room - t->patch_stages * patch) / b);
    return t->patch_stages * patch < room && t->b_stages >= 2;
}

// What a launch takes, in microseconds, fitted to 500 shapes of 7 to 224 squared, 16 to 512 channels each way, 1 to 64 images, all
// widths (nine in ten within 7 %): a start, and for every round of tiles an epilogue and its k-blocks, of 32 channels of one tap.
struct PatchCost {
    double round, kb;
};
constexpr PatchCost kRing[] = {{0.45, 0.215}, {0.55, 0.221}, {1.3, 0.24}, {2.55, 0.386}};  // 32, 64, 128, 256 columns
constexpr PatchCost kResident[] = {{0.0, 0.205}, {0.0, 0.205}, {0.0, 0.245}};              // the filter stays in shared memory
constexpr PatchCost kSplit[] = {{2.9, 0.54}, {3.6, 0.60}, {6.4, 0.69}};                    // SPLIT

bool patch_tiling(const ConvGeom& g, bool split, int sms, PatchTiling* best) {
    PatchTiling t;
    t.c_blocks = (g.C + BLOCK_K - 1) / BLOCK_K;
    t.pixel_tiles = g.N * ((g.Ho + PC_TH - 1) / PC_TH) * ((g.Wo + PC_TW - 1) / PC_TW);
    const double out_mb = (double)g.N * g.Ho * g.Wo * g.Co * 4e-6;
    bool any = false;
    for (int i = 0; i < (split ? 3 : 4); ++i) {
        const int bn = 32 << i;
        t.block_n = bn;
        t.n_tiles = (g.Co + bn - 1) / bn;
        t.tiles = t.pixel_tiles * t.n_tiles;
        t.splits = 1;
        if (split && 2 * t.tiles <= sms) t.splits = (int)std::min<int64_t>(std::min<int64_t>(sms / t.tiles, t.c_blocks), 16);
        if (rings_fit(&t, split)) {
            const PatchCost c = split ? kSplit[i] : t.resident ? kResident[i] : kRing[i];
            const int64_t rounds = (t.tiles * t.splits + sms - 1) / sms;
            const int kbs = (t.c_blocks + t.splits - 1) / t.splits * PC_TAPS;
            t.us = (!split && t.resident ? 5.2 : 4.7) + rounds * (c.round + c.kb * kbs) + (t.splits > 1 ? 0.7 + t.splits * out_mb : 0.0);
            if (!any || t.us < best->us) *best = t;
            any = true;
        }
        if (bn >= g.Co) break;
    }
    return any;
}

tfjsb_status launch(tfjsb_ctx* ctx, const float* x, const float* w, const float* bias, int act, float* y, const ConvGeom& g,
                    bool split, PatchTiling t, cudaStream_t s) {
    PatchConvArgs a{};
    a.C = g.C; a.Co = g.Co; a.Ho = g.Ho; a.Wo = g.Wo; a.H = g.H; a.W = g.W;
    a.pt = g.pt; a.pl = g.pl;
    a.tiles_x = (g.Wo + PC_TW - 1) / PC_TW;
    a.tiles_y = (g.Ho + PC_TH - 1) / PC_TH;
    a.images = (int)g.N;
    a.x = x; a.w = w; a.bias = bias; a.act = act;
    a.dev_status = ctx->dev_status;
    const int64_t out_elems = g.N * g.Ho * g.Wo * g.Co;
    if (t.splits > 1) {
        t.splits = (int)scratch_parts(ctx->scratch_c, t.splits, (size_t)out_elems * 4, s);
        if (!rings_fit(&t, split)) return fail(ctx, TFJSB_ERR_UNSUPPORTED, "convolution window too large");
    }
    a.n_tiles = t.n_tiles; a.splits = t.splits; a.num_tiles = (int)(t.tiles * t.splits);
    a.c_blocks = t.c_blocks; a.block_n = t.block_n;
    a.acc_stages = t.block_n > 128 ? 2 : MAX_ACC_STAGES;
    a.patch_stages = t.patch_stages;
    a.b_stages = t.b_stages; a.b_resident = t.resident;
    a.segment = split_segment((int64_t)t.c_blocks * PC_TAPS * BLOCK_K);
    tfjsb_status st;
    float* out = y;
    if (t.splits > 1) {
        if ((st = ensure_scratch(ctx, &ctx->scratch_c, (size_t)t.splits * out_elems * 4)) != TFJSB_OK) return st;
        out = ctx->scratch_c.ptr;
    }
    CUtensorMap map_x, map_w, map_y;
    const int64_t xd[4] = {g.C, g.W, g.H, g.N}, yd[4] = {g.Co, g.Wo, g.Ho, g.N * t.splits};
    const uint32_t xb[4] = {32u, (uint32_t)PC_PW, (uint32_t)PC_PH, 1u}, yb[4] = {32u, 8u, 4u, 1u};
    const int64_t wd[3] = {split ? g.C : g.Co, split ? g.Co : g.C, PC_TAPS};
    const uint32_t wb[3] = {32u, split ? (uint32_t)t.block_n : 32u, 1u};
    if ((st = encode_tile_map(ctx, &map_x, x, 4, xd, xb, "x")) != TFJSB_OK) return st;
    if ((st = encode_tile_map(ctx, &map_w, w, 3, wd, wb, "the filter", split ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B)) != TFJSB_OK) return st;
    if ((st = encode_tile_map(ctx, &map_y, out, 4, yd, yb, "y")) != TFJSB_OK) return st;
    auto kernel = split ? conv_patch_kernel<true> : conv_patch_kernel<false>;
    cudaError_t e = smem_attr_once(reinterpret_cast<const void*>(kernel), PC_SMEM);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "shared-memory limit");
    const size_t smem = 1024 + (size_t)PC_EPI_WARPS * EPI_SLAB_BYTES + (split ? 2 : 1) * ((size_t)t.patch_stages * PC_PATCH_STRIDE + (size_t)t.b_stages * t.block_n * 128);
    const int grid = std::min(a.num_tiles, ctx->sm_count);
    a.step = tile_digits(grid, a.splits, a.n_tiles, a.tiles_x, a.tiles_y);
    if ((e = launch_k(kernel, dim3(grid), dim3(pc_threads(split)), smem, s, map_x, map_w, map_y, a)) != cudaSuccess)
        return cuda_fail(ctx, e, "conv_patch launch");
    ++ctx->launches;
    if (t.splits > 1 && (e = launch_sum_rows(out, y, nullptr, t.splits, out_elems, 1, s, &ctx->launches)) != cudaSuccess)
        return cuda_fail(ctx, e, "partial-sum launch");
    return TFJSB_OK;
}

bool shape_ok(const ConvGeom& g) {
    constexpr int64_t LIM = 1LL << 30;
    return g.sh == 1 && g.sw == 1 && g.fh == 3 && g.fw == 3 && g.dh == 1 && g.dw == 1 && g.C % 4 == 0 && g.Co % 4 == 0 && g.C >= 16 && g.Co >= 4 &&
           g.pt >= 0 && g.pl >= 0 && g.N > 0 && g.Ho > 0 && g.Wo > 0 && g.N * 16 < LIM &&
           g.N * ((g.Ho + PC_TH - 1) / PC_TH) * ((g.Wo + PC_TW - 1) / PC_TW) * ((g.Co + 31) / 32) * 16 < LIM;
}

// The input gradient as a forward convolution over dy: dx[i] = sum over k of dy[i + pt - k d] f[k], k from last to first.
ConvGeom transposed(const ConvGeom& g) {
    ConvGeom t = g;
    t.H = g.Ho; t.W = g.Wo; t.C = g.Co;
    t.Ho = g.H; t.Wo = g.W; t.Co = g.C;
    t.pt = 2 - g.pt;
    t.pl = 2 - g.pl;
    return t;
}

}  // namespace

// By how much the estimate of this kernel has to be the lower one: both are a few percent off.  On 500 other shapes than those
// that the estimates were fitted to
//   forward   153 are taken, at 0.90 of the time of the im2col kernel and its filter packing on average, the worst at 1.04
//             ([64,112,112,32] -> 32: 108 and 84 us, [1,224,224,16] -> 16: 12.9 and 10.9, [16,28,28,128] -> 128: 15.6 and 15.2; not
//             taken, images that tiles of 16 x 8 fill badly: [63,28,28,128] -> 256: 50 and 69, [9,135,135,72] -> 64: 63 and 68)
//   gradient  132, at 0.87, the worst at 1.04 (most where im2col tiles have the K loop in fewer parts: [4,14,14,512] of 512 91.6 and
//             39.7, but also [16,28,28,128] of 128: 38.3 and 37.1, [2,172,172,128] of 96: 109 and 99; not taken: [61,28,28,128]
//             of 120: 106 and 125, [63,8,8,256] of 312: 66 and 73, [32,56,56,64] of 64: 103 and 108)
constexpr double PC_AHEAD = 0.95;

bool conv_patch_input_preferred(const ConvGeom& g, int sm_count) {
    PatchTiling t;
    if (!shape_ok(g) || !patch_tiling(g, false, sm_count, &t)) return false;
    if (const char* env = getenv("TFJSB_CONV_PATCH")) return atoi(env) != 0;  // for tests: 1 = wherever it can, 0 = never
    return t.us < PC_AHEAD * conv_im2col_us(g, sm_count);
}

tfjsb_status run_conv_patch_input(tfjsb_ctx* ctx, const float* x, const float* f, const float* bias, int act, float* y, const ConvGeom& g, cudaStream_t s) {
    PatchTiling t;
    if (!shape_ok(g) || !patch_tiling(g, false, ctx->sm_count, &t)) return fail(ctx, TFJSB_ERR_UNSUPPORTED, "not a convolution of this kernel");
    return launch(ctx, x, f, bias, act, y, g, false, t, s);
}

bool conv_patch_gradient_preferred(const ConvGeom& g, int sm_count) {
    PatchTiling t;
    const ConvGeom b = transposed(g);
    if (!shape_ok(b) || !patch_tiling(b, true, sm_count, &t) || (int64_t)PC_TAPS * t.c_blocks * 32 > SPLIT_MAX_K) return false;
    if (const char* env = getenv("TFJSB_CONV_PATCH")) return atoi(env) != 0;
    if (getenv("TFJSB_GRAD_INPUT")) return false;  // which decides between the two kernels for any window
    return conv2d_grad_input_preferred(g, sm_count) && t.us < PC_AHEAD * conv2d_grad_input_us(g, sm_count);
}

tfjsb_status run_conv_patch_gradient(tfjsb_ctx* ctx, const float* dy, const float* f, float* dx, const ConvGeom& g, cudaStream_t s) {
    PatchTiling t;
    const ConvGeom b = transposed(g);
    if (!shape_ok(b) || !patch_tiling(b, true, ctx->sm_count, &t)) return fail(ctx, TFJSB_ERR_UNSUPPORTED, "not a convolution of this kernel");
    return launch(ctx, dy, f, nullptr, TFJSB_ACT_NONE, dx, b, true, t, s);
}

}  // namespace tfjsb
