// Tile constants and the epilogue staging routine shared by the tcgen05 kernels (plain GEMM,
// implicit-GEMM convolution, fused depthwise + pointwise block).
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"
#include "ptx_sm100.cuh"

namespace tfjsb {
namespace tile {

constexpr int BLOCK_M = 128;
constexpr int BLOCK_K = 32;  // fp32 elements: one 128-byte swizzle row
constexpr int UMMA_K = 8;    // tf32 elements per tcgen05.mma
constexpr int MAX_ACC_STAGES = 4;
constexpr int EPI_COLS = 32;
constexpr int A_STAGE_BYTES = BLOCK_M * BLOCK_K * 4;             // 16 KiB
constexpr int EPI_SLAB_BYTES = 32 * EPI_COLS * 4;                // 4 KiB: 32 rows x 128 B
constexpr int EPI_BYTES = 8 /*epilogue warps*/ * EPI_SLAB_BYTES;      // 32 KiB
constexpr int SMEM_LIMIT = 232448;                               // 227 KiB

// Rows of the copy box of an A tile: those that exist, when the whole matrix is less than a tile (a multiple of 8, the
// swizzle's period).  The other rows of the operand tile keep what was there; their results are never stored.  The copy
// unit spends as long on rows outside the tensor as on rows inside ([1,1024] . [1024,1000]: 8.3 us with 128-row boxes).
inline int a_box_rows(int64_t M) { return M >= BLOCK_M ? BLOCK_M : (int)((M + 7) / 8 * 8); }

// Fused epilogue of one 32-row x 32-column accumulator block held one row per lane: bias add,
// activation, and the swizzled store into the staging slab the bulk tensor store reads from
// (16-byte chunk j of row `lane` lives at chunk j ^ (lane % 8): the 128-byte swizzle).
template <int ACT>
__device__ __forceinline__ void stage_chunk(const uint32_t (&r)[32], const float* bias, int cols_left,
                                            uint32_t row_addr, int lane) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        float4 v;
        v.x = __uint_as_float(r[4 * j + 0]); v.y = __uint_as_float(r[4 * j + 1]);
        v.z = __uint_as_float(r[4 * j + 2]); v.w = __uint_as_float(r[4 * j + 3]);
        // ld_global where it stands: fp32 models of few images 0 to 1 % faster than with loads that the compiler may move; bfloat16 models
        // of few images are 0.5 to 1 % slower so, those of many 0.2 to 0.6 % faster, and keep the latter kind
        if (bias != nullptr && 4 * j < cols_left) {  // N % 4 == 0: a quad is all in or all out
            const float4 b = ld_global4(bias + 4 * j);
            v.x = v.x + b.x; v.y = v.y + b.y; v.z = v.z + b.z; v.w = v.w + b.w;
        }
        v.x = apply_act_t<ACT>(v.x); v.y = apply_act_t<ACT>(v.y);
        v.z = apply_act_t<ACT>(v.z); v.w = apply_act_t<ACT>(v.w);
        const uint32_t dst = row_addr + (uint32_t)((j ^ (lane & 7)) << 4);
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                     : "memory");
    }
}

// ---- fp32 accuracy from TF32 products ----------------------------------------------------------------
// An fp32 operand v is used as two TF32 values (the tensor core drops the low 13 bits of what it reads), hi + lo, and a
// product as hi * hi + hi * lo + lo * hi.
//
// Where threads write the operand tiles themselves, hi is v rounded to nearest and lo the rest, exact in fp32 and cut to
// TF32 after the addition of half a unit (7e-8 of v on average; values that lo represents exactly stay as they are).  The
// rounding of hi carries a NaN of all ones over to -0, but lo is then a NaN.
__device__ __forceinline__ void tf32_split(float v, float& hi, float& lo) {
    const uint32_t up = __float_as_uint(v) + 0x1000u;
    hi = __uint_as_float(up);
    const float rest = v - __uint_as_float(up & 0xffffe000u);
    lo = fmaf(rest, 0.00048828125f, rest);
}
// Where the tile is left as it was copied, hi is v cut to TF32, and lo the rest, rounded by an integer addition.  The
// product lo * lo that is left out then has the sign of the whole: on average 2^-23 of it, a bias.  The lo half of one
// operand is therefore rounded away from zero (SPLIT_UP), which adds as much on average, that of the other to nearest.
constexpr uint32_t SPLIT_UP = 0x1fffu, SPLIT_NEAREST = 0x1000u;
__device__ __forceinline__ float tf32_rest(float v, uint32_t round) {
    const float hi = __uint_as_float(__float_as_uint(v) & 0xffffe000u);
    return __uint_as_float(__float_as_uint(v - hi) + round);
}

// The tensor core cuts every sum it makes towards zero, so an accumulator's error grows with the number of additions,
// where the errors of fp32 fused multiply-adds, which round to nearest, mostly cancel.  The large products (hi * hi)
// therefore go to an accumulator for a segment of a few k-blocks only (4 additions of 8 products each), and these parts are
// added by threads, in tensor memory: two accumulators in turn, one for the small products, which are 2^-11 of the large
// ones, and the sum:  columns [large 0 | large 1 | small | sum].
//
// Length of a segment, in k-blocks, for sums of K products.  Measured against 64 bits: 7e-8 of the result per k-block of a
// segment, 1.5e-7 if all products have one sign, beside 1.2e-7 from the operands; sums by fp32 multiply-adds 1.8e-8 sqrt(K).
// Without segments a 3x3 convolution's input gradient over 512 channels was 1.0e-5 off (multiply-adds: 1.2e-6).
inline int split_segment(int64_t K) {
    int n = 1;
    while ((int64_t)(n + 1) * (n + 1) * 196 <= K) ++n;  // sqrt(K) / 14
    return n;
}
// Of longer sums the small products' accumulator would be the less exact part.
constexpr int64_t SPLIT_MAX_K = 1LL << 22;

// What is not finite may be a result of the split: with an infinite operand lo is NaN or the opposite infinity, a value
// above the largest TF32 number is rounded to infinity, and a NaN with low bits only is cut to infinity.  Such a result is
// summed again in fp32 by the thread that has it, as the CUDA-core kernels do.  (A result that is finite had none of these
// among its operands: every one of them leaves an infinity or a NaN in hi or in lo.)
__device__ __forceinline__ bool not_finite(uint32_t bits) { return (bits & 0x7f800000u) == 0x7f800000u; }

// One 32-lane x `cols`-column part of  sum = (first ? 0 : sum) + large, and + small after the last segment; both addresses
// and `cols` (a multiple of STEP, 8 or 16) are of the caller's lanes and columns.
template <int STEP>
__device__ __forceinline__ void add_segment(uint32_t large, uint32_t small, uint32_t sum, int cols, bool first, bool last) {
#pragma unroll 1
    for (int c = 0; c < cols; c += STEP) {
        uint32_t u[STEP], v[STEP], w[STEP];
        ptx::tc_ld_cols(large + (uint32_t)c, u);
        if (!first) ptx::tc_ld_cols(sum + (uint32_t)c, v);
        if (last) ptx::tc_ld_cols(small + (uint32_t)c, w);
        ptx::tc_ld_wait();
#pragma unroll
        for (int e = 0; e < STEP; ++e) {
            float s = __uint_as_float(u[e]);
            if (!first) s = __uint_as_float(v[e]) + s;
            if (last) s += __uint_as_float(w[e]);
            u[e] = __float_as_uint(s);
        }
        ptx::tc_st_cols(sum + (uint32_t)c, u);
    }
    ptx::tc_st_wait();
}

// ---- shared memory, time-outs, copies ---------------------------------------------------------------
__device__ __forceinline__ float4 lds4(uint32_t a) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts4(uint32_t a, float x, float y, float z, float w) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}

// Raises the abort flag; the first role to do so reports the reason.
__device__ __forceinline__ void give_up(volatile int* abort_flag, unsigned int* dev_status, unsigned int code) {
    if (!*abort_flag) {
        *abort_flag = 1;
        atomicOr(dev_status, code);
    }
}
// Waits (bounded) until the phase has completed, whatever the abort flag says.
__device__ __forceinline__ void drain(uint32_t bar, uint32_t parity, unsigned int* dev_status) {
    const unsigned long long t0 = ptx::global_ns();
    while (!ptx::mbar_try_wait(bar, parity)) {
        if (ptx::global_ns() - t0 > ptx::WAIT_LIMIT_NS) {
            atomicOr(dev_status, DEV_STATUS_TIMEOUT_DRAIN);
            break;
        }
    }
}

// An operand tile of 32 k whose rows of memory run along M or N: one copy of 32 k x 32 columns per group.
template <bool BATCHED>
__device__ __forceinline__ void load_mn_groups(uint32_t dst, const CUtensorMap* map, uint32_t bar, int row0, int k0, int batch, int groups) {
#pragma unroll 1
    for (int i = 0; i < groups; ++i) {
        if (BATCHED) ptx::tma_load_3d(dst + (uint32_t)i * 4096u, map, bar, row0 + 32 * i, k0, batch);
        else ptx::tma_load_2d(dst + (uint32_t)i * 4096u, map, bar, row0 + 32 * i, k0);
    }
}

// ---- bfloat16 storage ------------------------------------------------------------------------------
// Instruction descriptor: fp32 accumulator, bfloat16 A and B (format 1), both K-major.
__device__ __forceinline__ uint32_t make_idesc_bf16(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// One 32-row x 32-column accumulator block, one row per lane: bias, activation, rounding to bfloat16,
// and the store into the staging slab in the 64-byte swizzle the bulk tensor store expects (rows of
// 64 bytes; 16-byte piece j of row r lives at piece j ^ ((r / 2) % 4)).
template <int ACT>
__device__ __forceinline__ void stage_chunk_bf16(const uint32_t (&r)[32], const float* bias, int cols_left,
                                                 uint32_t slab, int lane) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(r[8 * j + e]);
        if (bias != nullptr && 8 * j < cols_left) {  // N % 8 == 0: a group of eight is all in or all out
            const float4 b0 = load_global(reinterpret_cast<const float4*>(bias + 8 * j));
            const float4 b1 = load_global(reinterpret_cast<const float4*>(bias + 8 * j + 4));
            v[0] += b0.x; v[1] += b0.y; v[2] += b0.z; v[3] += b0.w;
            v[4] += b1.x; v[5] += b1.y; v[6] += b1.z; v[7] += b1.w;
        }
        uint32_t p[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(apply_act_t<ACT>(v[2 * e]), apply_act_t<ACT>(v[2 * e + 1]));
            p[e] = *reinterpret_cast<const uint32_t*>(&h);
        }
        const uint32_t dst = slab + (uint32_t)lane * 64u + (uint32_t)((j ^ ((lane >> 1) & 3)) << 4);
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(p[0]), "r"(p[1]), "r"(p[2]), "r"(p[3])
                     : "memory");
    }
}

}  // namespace tile
}  // namespace tfjsb
