// Shared declarations of the CUDA library: context, error helpers, the fused epilogue,
// and the host-side launchers each kernel file exports to the API layer.
#pragma once

#include <cuda_runtime.h>
#include <cuda.h>
#include <stdint.h>

#include <string>
#include <utility>
#include <vector>

#include "tfjsb.h"

namespace tfjsb {

// ---- device status word -------------------------------------------------------------------
// Kernels with bounded waits OR a code into this word when a wait gives up; the host reads it
// in tfjsb_check_device_status.
enum : unsigned int {
    DEV_STATUS_OK = 0u,
    DEV_STATUS_TIMEOUT_PRODUCER = 1u,  // TMA producer waited too long for a free stage
    DEV_STATUS_TIMEOUT_MMA = 2u,       // MMA issuer waited too long for data or for a free accumulator
    DEV_STATUS_TIMEOUT_EPILOGUE = 4u,  // epilogue waited too long for an accumulator
    DEV_STATUS_TIMEOUT_DRAIN = 8u,     // teardown waited too long for copies in flight
    DEV_STATUS_TIMEOUT_DEPTHWISE = 16u // depthwise kernel waited too long for an input tile
};

// ---- fused epilogue (bias add, then activation), identical in every kernel -----------------
//   v = acc + bias ; relu: v > 0 ? v : +0 (NaN stays NaN, -0 -> +0) ; relu6: min(relu(v), 6)
// max.NaN / min.NaN return NaN when an input is NaN and order -0 below +0, which is exactly that
// definition in two instructions (a compare-and-select chain costs four times as many, and the
// bandwidth-bound kernels turned out to be bound by instruction issue).
__device__ __forceinline__ float relu_nan(float v) {
    float r;
    asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float relu6_nan(float v) {
    float r;
    asm("max.NaN.f32 %0, %1, 0f00000000;\n\tmin.NaN.f32 %0, %0, 0f40C00000;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float apply_act(float v, int act) {
    const float r = relu_nan(v);
    const float r6 = relu6_nan(v);
    return act == TFJSB_ACT_NONE ? v : (act == TFJSB_ACT_RELU6 ? r6 : r);
}
// Two independent fp32 FMAs in one instruction (sm_100 packed fp32): acc.{x,y} += a.{x,y} * b.{x,y},
// each lane rounded exactly like a scalar fmaf.  Halves the issue slots of the CUDA-core kernels,
// which are bound by instruction issue.
__device__ __forceinline__ void fma2(float2& acc, const float2& a, const float2& b) {
    unsigned long long& d = reinterpret_cast<unsigned long long&>(acc);
    asm("fma.rn.f32x2 %0, %1, %2, %0;"
        : "+l"(d)
        : "l"(reinterpret_cast<const unsigned long long&>(a)), "l"(reinterpret_cast<const unsigned long long&>(b)));
}
// acc.{x,y,z,w} += a * b of four bfloat16 each, as they lie in memory: exact products, one rounding, as fmaf of the widened
// values, without widening them.
__device__ __forceinline__ void fma4_bf16(float4& acc, const uint2& a, const uint2& b) {
    asm("{\n\t.reg .b16 a0, a1, a2, a3, b0, b1, b2, b3;\n\t"
        "mov.b32 {a0, a1}, %4;\n\tmov.b32 {a2, a3}, %5;\n\tmov.b32 {b0, b1}, %6;\n\tmov.b32 {b2, b3}, %7;\n\t"
        "fma.rn.f32.bf16 %0, a0, b0, %0;\n\tfma.rn.f32.bf16 %1, a1, b1, %1;\n\t"
        "fma.rn.f32.bf16 %2, a2, b2, %2;\n\tfma.rn.f32.bf16 %3, a3, b3, %3;\n\t}"
        : "+f"(acc.x), "+f"(acc.y), "+f"(acc.z), "+f"(acc.w)
        : "r"(a.x), "r"(a.y), "r"(b.x), "r"(b.y));
}
__device__ __forceinline__ float2 add2(const float2& a, const float2& b) {
    float2 r;
    asm("add.rn.f32x2 %0, %1, %2;"
        : "=l"(reinterpret_cast<unsigned long long&>(r))
        : "l"(reinterpret_cast<const unsigned long long&>(a)), "l"(reinterpret_cast<const unsigned long long&>(b)));
    return r;
}
// relu / relu6 of two bfloat16: their bounds are bfloat16 values and rounding is monotonic, so this after the rounding is the
// rounded activation, in half the instructions.
template <int ACT>
__device__ __forceinline__ uint32_t apply_act_bf16x2(uint32_t v) {
    if (ACT == TFJSB_ACT_RELU || ACT == TFJSB_ACT_RELU6) asm("max.NaN.bf16x2 %0, %0, %1;" : "+r"(v) : "r"(0u));
    if (ACT == TFJSB_ACT_RELU6) asm("min.NaN.bf16x2 %0, %0, %1;" : "+r"(v) : "r"(0x40c040c0u));
    return v;
}
__device__ __forceinline__ void fma4_packed(float4& acc, const float4& a, const float4& b) {
    fma2(reinterpret_cast<float2*>(&acc)[0], reinterpret_cast<const float2*>(&a)[0], reinterpret_cast<const float2*>(&b)[0]);
    fma2(reinterpret_cast<float2*>(&acc)[1], reinterpret_cast<const float2*>(&a)[1], reinterpret_cast<const float2*>(&b)[1]);
}

template <int ACT>
__device__ __forceinline__ float apply_act_t(float v) {
    if (ACT == TFJSB_ACT_NONE) return v;
    if (ACT == TFJSB_ACT_RELU6) return relu6_nan(v);
    return relu_nan(v);
}

__device__ __forceinline__ bool finite4(const float4& v) {
    return isfinite(v.x) && isfinite(v.y) && isfinite(v.z) && isfinite(v.w);
}

// Of sums of values times zero: false when one of the values was not finite.
__device__ __forceinline__ bool all_zero(const float4& v) { return v.x + v.y + (v.z + v.w) == 0.f; }

// ---- context --------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

typedef CUresult (*EncodeIm2colFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                   const int*, const int*, cuuint32_t, cuuint32_t, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct Scratch {
    float* ptr = nullptr;
    size_t bytes = 0;
};

}  // namespace tfjsb

struct tfjsb_ctx {
    int device = 0;
    int sm_count = 0;
    tfjsb_math math = TFJSB_MATH_TF32;
    std::string last_error;
    unsigned int* dev_status = nullptr;  // device status word
    tfjsb::EncodeTiledFn encode_tiled = nullptr;
    tfjsb::EncodeIm2colFn encode_im2col = nullptr;
    tfjsb::Scratch scratch_a, scratch_b;  // transposed operands of tfjsb_matmul
    tfjsb::Scratch scratch_c;             // partial sums of the filter / bias gradients
    std::vector<void*> retired;            // outgrown scratch blocks, freed at shutdown
    int64_t launches = 0;
    int live_models = 0;
};

namespace tfjsb {

tfjsb_status fail(tfjsb_ctx* ctx, tfjsb_status st, const std::string& msg);
tfjsb_status cuda_fail(tfjsb_ctx* ctx, cudaError_t err, const char* what);
// Grows `s` to at least `bytes`.  Never synchronises: an outgrown block may still be read by kernels in
// flight on any stream, so it is kept until tfjsb_shutdown; growth is geometric, so all outgrown blocks
// together are smaller than the live one.  tfjsb_reserve_scratch sizes the blocks up front.
tfjsb_status ensure_scratch(tfjsb_ctx* ctx, Scratch* s, size_t bytes);
// Whether `s` has less than `bytes` and cannot grow, because `stream` is being captured (an allocation would end the
// capture): a call that can do with less scratch then does.
bool scratch_is_short(const Scratch& s, size_t bytes, cudaStream_t stream);
// How many of `wanted` partial results of `each` bytes there is room for, 1 at least (one needs no scratch).
int64_t scratch_parts(const Scratch& s, int64_t wanted, size_t each, cudaStream_t stream);

// Raises a kernel's dynamic shared-memory limit once per (kernel, device): function attributes belong to
// a device's copy of the function, and contexts on several devices or host threads may launch the same kernel.
cudaError_t smem_attr_once(const void* kernel, int bytes);
// Number of SMs of the current device (cached per device): grid caps of the grid-stride kernels.
int current_sm_count();

// ---- kernel launch with optional programmatic dependent launch --------------------------------------
// Every kernel launched through launch_k calls pdl_wait() before it touches global memory, reads or writes, so it may be
// launched while the previous kernel of the stream drains, and only its prologue (barrier set-up, tensor-map prefetch,
// TMEM allocation) and the launch itself overlap.  Between kernels of op calls this saves 1 to 3 us (eleven small ops
// 61 -> 38 us, a block's forward and backward pass 229 -> 210, one 512^3 matMul after another 8.4 -> 7.3).
// On unless TFJSB_NO_PDL is set; the executor switches it by the model's setting while it enqueues one.
// What starts early is put where there is room and not one block to an SM, so it costs more than it saves where blocks of either
// kernel run long and share SMs.  Long reductions of few blocks are therefore launched after the kernel before (launch_k_if:
// global pools, softmax), and kernels of small blocks, or of two CTAs to an SM, that another such kernel may follow say
// pdl_launch_dependents() late or not at all, in which case the next one starts as they end.
extern thread_local bool g_launch_pdl;

// A load of what the kernel before may still be writing when this one starts: an ordinary one, also through pointers to
// const (__ldg and const __restrict__ pointers read through the non-coherent path, which wants data that nobody writes
// while the kernel runs).
template <typename T>
__device__ __forceinline__ T load_global(const T* p) { return *p; }
// The other kind, for what nothing writes while any kernel runs that reads it: a model's filters and biases.
template <typename T>
__device__ __forceinline__ T load_fixed(const T* p) { return __ldg(p); }
// load_global as an instruction that stays where it is written, for loops that load ahead with few registers to spare (the
// strided GEMM's loaders spill 16 to 40 bytes with load_global and nothing with these) or whose loads the compiler spreads out
// (max and global pools).
__device__ __forceinline__ float ld_global(const float* p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 ld_global4(const float* p) {
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}

template <typename... KArgs, typename... Args>
cudaError_t launch_k_if(bool early, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = early && g_launch_pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}
template <typename... KArgs, typename... Args>
cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args) {
    return launch_k_if(true, kernel, grid, block, smem, s, std::forward<Args>(args)...);
}

// The same launch without the attribute, whatever the executor's setting: for kernels made of many
// small blocks with little shared memory.  Launched early, their first blocks become resident beside
// the predecessor's CTAs and wait there, and that costs the predecessor more than the overlap returns
// (measured: a model whose depthwise layers are such kernels ran 4 % slower with the attribute on
// them, and the fp32 model 9 % slower when its depthwise layers were swapped for such a kernel; the
// persistent kernels with large shared-memory footprints cannot become resident early and only
// overlap their prologue).  Such a kernel still executes griddepcontrol.launch_dependents, so its
// successor may start early.
template <typename... KArgs, typename... Args>
cudaError_t launch_k_serial(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args) {
    return launch_k_if(false, kernel, grid, block, smem, s, std::forward<Args>(args)...);
}

// ---- geometry of one convolution / pooling call -----------------------------------------------
struct ConvGeom {
    int64_t N;
    int H, W, C;        // input
    int fh, fw;         // filter window
    int Co;             // output channels (conv: Cout; depthwise: C*mult; pool: C)
    int mult;           // depthwise channel multiplier (1 otherwise)
    int sh, sw, dh, dw; // strides, dilations
    int pt, pl;         // padding before (top, left)
    int Ho, Wo;
    // 3x3 depthwise kernels: taps read last to first, which turns the forward pass over dy into the gradient with
    // respect to the input (stride 1)
    int reversed = 0;
    int gather_only = 0;  // conv2d: no im2col copies, whose packed filter is the larger one
};

// ---- launchers (each returns the CUDA launch error; `launches` is incremented per kernel) -----
cudaError_t launch_bias_act(const float* x, const float* bias, float* y, int64_t rows, int64_t C, int act,
                            cudaStream_t s, int64_t* launches);
cudaError_t launch_avg_pool(const float* x, float* y, const ConvGeom& g, cudaStream_t s, int64_t* launches);
cudaError_t launch_softmax(const float* x, float* y, int64_t rows, int64_t cols, cudaStream_t s, int64_t* launches);
cudaError_t launch_max_pool(const float* x, float* y, const ConvGeom& g, cudaStream_t s, int64_t* launches);
// out[i] = a[i] op b[i % b_len] (op: tfjsb_binary_op)
cudaError_t launch_binary(int op, const float* a, const float* b, float* out, int64_t n, int64_t b_len, cudaStream_t s,
                          int64_t* launches);
// out[c, r] = in[r, c] for in of shape [rows, cols]
cudaError_t launch_transpose(const float* in, float* out, int64_t rows, int64_t cols, cudaStream_t s,
                             int64_t* launches);

// C[M,N] = act(A' B' + bias), CUDA-core fp32.  A' element (i,k) at a[i*a_rs + k*a_cs]; B' element
// (k,j) at b[k*b_rs + j*b_cs]; C row pitch ldc.
cudaError_t launch_gemm_fp32(const float* a, int64_t a_rs, int64_t a_cs, const float* b, int64_t b_rs, int64_t b_cs,
                             const float* bias, int act, float* c, int64_t ldc, int64_t M, int64_t N, int64_t K,
                             cudaStream_t s, int64_t* launches);

// The same with fp32 accuracy on the tensor cores, for operands with either dimension contiguous and any alignment
// (gemm_strided_tcgen05.cu); `batches` products stored one after the other.
bool gemm_strided_supported(int64_t batches, int64_t M, int64_t N, int64_t K, int sm_count);
cudaError_t launch_gemm_strided(const float* a, int64_t a_rs, int64_t a_ks, const float* b, int64_t b_ks, int64_t b_cs, const float* bias,
                                int act, float* c, int64_t batches, int64_t M, int64_t N, int64_t K, int sm_count,
                                unsigned int* dev_status, cudaStream_t s, int64_t* launches);

// Direct convolution on CUDA cores (any window, stride, dilation).  filter [fh,fw,Cin,Cout].
cudaError_t launch_conv2d_fp32(const float* x, const float* f, const float* bias, int act, float* y,
                               const ConvGeom& g, cudaStream_t s, int64_t* launches);

// Depthwise convolution.  filter [fh,fw,C,mult].  A plan picks the kernel and, for the bulk-copy
// pipelined 3x3 kernel, holds the tensor map of the input; it stays valid while `x` and the
// geometry stay the same.
struct DepthwisePlan {
    int variant = -1;  // -1: register kernel / scalar kernel; >= 0: index of the pipelined instance
    CUtensorMap map_x;
    int tiles_x = 0, tiles_y = 0, c_blocks = 0;
    int64_t num_tiles = 0;
    int grid = 0, stages = 0;
    size_t smem_bytes = 0;
    bool narrow = false;  // planned for bfloat16 storage
    // Whether the next kernel may start while this one runs, for a model's layers, whose next kernel has an SM's shared memory for
    // itself, and not for calls, whose next may be such a kernel again: two of its CTAs fit an SM, and those that wait beside the last
    // ones of this call get the tiles of two long CTAs as often as not (one call after another, [11,30,30,1000] 16.6 us without an
    // early start, 18.4 with one, 15.2 started as the call ends; [10,71,71,752] 57.8, 63.2 and 56.4).
    bool next_early = true;
};
// `narrow`: x is bfloat16 (narrow storage); the plan then runs through launch_depthwise_tma_narrow, and
// variant stays -1 where the pipelined kernel has no instance for the shape.
tfjsb_status depthwise_plan(tfjsb_ctx* ctx, const void* x, const ConvGeom& g, DepthwisePlan* plan, bool narrow = false);
cudaError_t launch_depthwise_tma_narrow(const DepthwisePlan& plan, const float* f, const float* bias, int act, void* y,
                                        bool y_is_bf16, const ConvGeom& g, unsigned int* dev_status, cudaStream_t s,
                                        int64_t* launches);
cudaError_t launch_depthwise(const DepthwisePlan& plan, const float* x, const float* f, const float* bias, int act,
                             float* y, const ConvGeom& g, unsigned int* dev_status, cudaStream_t s,
                             int64_t* launches);

// Tensor-core GEMM: C[M,N] = act(A[M,K] . Bt[N,K]^T + bias); all three row-major with K (resp. N)
// contiguous, or operands with their other dimension contiguous (a_mn: A as [K,M], M % 4 == 0; b_mn: B as [K,N]), whose
// products have the same bits.  A plan holds the tensor maps and tile choice; it can be built once and reused while
// the pointers stay the same.
struct GemmTf32Plan {
    CUtensorMap map_a, map_b, map_c;
    int64_t M, N, K;
    int64_t batches = 1;  // independent products of this shape in one launch (single-CTA kernel only)
    int block_n;       // 32..256
    int stages;
    int acc_stages;
    int num_tiles;
    int grid;
    size_t smem_bytes;
    // CTA-pair kernel (gemm_pair.cu): 256 x block_n tiles shared by two CTAs
    bool pair = false;
    bool a_mn = false, b_mn = false;   // A is stored [K, M], B is stored [K, N]
    // cluster split-K kernel (gemm_tf32_splitk.cu): `splits` CTAs per tile, reduced through shared memory
    bool cluster_split = false;
    int splits = 1, kb_per_split = 0;  // slices of the K loop (= cluster size) and k-blocks per slice
    bool next_early = true;            // of the cluster kernel, whose CTAs may share an SM: see DepthwisePlan
    float* c = nullptr;                // C, which that kernel stores directly
    // implicit-GEMM convolution: A is gathered from x by the kernel instead of copied, or copied by im2col loads
    bool gather = false;
    bool im2col = false;
    const float* x = nullptr;
    ConvGeom g{};
};
bool gemm_tf32_supported(int64_t M, int64_t N, int64_t K);
// `batches` > 1: that many products of the same shape, operands and results stored one after the other.
tfjsb_status gemm_tf32_plan(tfjsb_ctx* ctx, const float* a, const float* bt, float* c, int64_t M, int64_t N,
                            int64_t K, GemmTf32Plan* plan, int64_t batches = 1, bool a_mn = false, bool b_mn = false);
// The same GEMM on CTA pairs; gemm_tf32_plan picks it where it is the faster kernel (environment
// variable TFJSB_GEMM_PAIR: 0 = never, 1 = wherever the shape allows, unset = by shape).
bool gemm_tf32_pair_preferred(int64_t M, int64_t N, int64_t K, int sm_count);
tfjsb_status gemm_tf32_pair_plan(tfjsb_ctx* ctx, const float* a, const float* bt, float* c, int64_t M, int64_t N,
                                 int64_t K, GemmTf32Plan* plan, bool a_mn, bool b_mn);
cudaError_t launch_gemm_tf32_pair(const GemmTf32Plan& plan, const float* bias, int act, unsigned int* dev_status,
                                  cudaStream_t s, int64_t* launches);
// Split K across the CTAs of a cluster, for GEMMs with too few tiles for the SMs (gemm_tf32_splitk.cu).
bool gemm_tf32_splitk_choice(int64_t M, int64_t N, int64_t K, int sm_count, int64_t whole_ns, int* block_n, int* splits);
tfjsb_status gemm_tf32_splitk_plan(tfjsb_ctx* ctx, const float* a, const float* bt, float* c, int64_t M, int64_t N,
                                   int64_t K, int block_n, int splits, GemmTf32Plan* plan, bool a_mn, bool b_mn);
cudaError_t launch_gemm_tf32_splitk(const GemmTf32Plan& plan, const float* bias, int act, unsigned int* dev_status,
                                    cudaStream_t s, int64_t* launches);
// Implicit-GEMM convolution on the same kernel: M = N*Ho*Wo output pixels, K = fh*fw*Cin, N = Cout.
// `bt` is the filter packed as [Cout, k_pad] by launch_pack_conv_filter (K-contiguous, zero padded to whole k-blocks of
// 32: each tap for itself where A comes by im2col loads, the whole window otherwise).
bool conv_igemm_supported(const ConvGeom& g);
bool conv_igemm_uses_im2col(const ConvGeom& g);
double conv_im2col_us(const ConvGeom& g, int sm_count);  // estimate of the filter packing and the im2col kernel
int64_t conv_igemm_k_pad(const ConvGeom& g);
cudaError_t launch_pack_conv_filter(const float* f, float* out, const ConvGeom& g, cudaStream_t s, int64_t* launches);
tfjsb_status conv_igemm_plan(tfjsb_ctx* ctx, const float* x, const float* bt, float* y, const ConvGeom& g,
                             GemmTf32Plan* plan);
// out[n, t * c_pad + c] = c < C ? f[t, c, n] : 0 for f of shape [taps, C, N], out of shape [N, taps * c_pad]
cudaError_t launch_pack_filter(const float* f, float* out, int64_t taps, int64_t C, int64_t N, int64_t c_pad, cudaStream_t s,
                               int64_t* launches);
cudaError_t launch_gemm_tf32(const GemmTf32Plan& plan, const float* bias, int act, unsigned int* dev_status,
                             cudaStream_t s, int64_t* launches);

// ---- narrow storage (bfloat16 in memory, fp32 sums) -------------------------------------------------
// Tensor-core GEMM on bfloat16 operands: C[M,N] = act(A[M,K] . Bt[N,K]^T + bias), C bfloat16 or fp32.
struct GemmBf16Plan {
    CUtensorMap map_a, map_b, map_c;
    int64_t M = 0, N = 0, K = 0;
    bool c_is_bf16 = true;
    bool pair = false;  // CTA-pair kernel (gemm_pair.cu): 256 x block_n tiles shared by two CTAs
    int block_n = 0, stages = 0, acc_stages = 0, num_tiles = 0, grid = 0;
    int epi_warps = 16;  // epilogue warps of the single-CTA kernel: 16 for short K loops, 8 otherwise
    size_t smem_bytes = 0;
};
bool gemm_bf16_supported(int64_t M, int64_t N, int64_t K);
tfjsb_status gemm_bf16_plan(tfjsb_ctx* ctx, const void* a, const void* bt, void* c, bool c_is_bf16, int64_t M, int64_t N,
                            int64_t K, GemmBf16Plan* plan);
cudaError_t launch_gemm_bf16(const GemmBf16Plan& plan, const float* bias, int act, unsigned int* dev_status,
                             cudaStream_t s, int64_t* launches);
// The same GEMM (bfloat16 output only) on CTA pairs; gemm_bf16_plan picks it where it is the faster
// kernel (TFJSB_GEMM_PAIR: 0 = never, 1 = wherever the shape allows, unset = by shape).
bool gemm_bf16_pair_preferred(int64_t M, int64_t N, int64_t K, int sm_count);
tfjsb_status gemm_bf16_pair_plan(tfjsb_ctx* ctx, const void* a, const void* bt, void* c, int64_t M, int64_t N, int64_t K,
                                 GemmBf16Plan* plan);
cudaError_t launch_gemm_bf16_pair(const GemmBf16Plan& plan, const float* bias, int act, unsigned int* dev_status,
                                  cudaStream_t s, int64_t* launches);
// CUDA-core layers of the same mode.  Filters are fp32 arrays holding bfloat16 values.
cudaError_t launch_conv_narrow(const void* x, bool x_is_f32, const float* f, const float* bias, int act, void* y,
                               bool y_is_bf16, const ConvGeom& g, cudaStream_t s, int64_t* launches);
bool depthwise_narrow_supported(const ConvGeom& g);
cudaError_t launch_depthwise_narrow(const void* x, const float* f, const float* bias, int act, void* y, bool y_is_bf16,
                                    const ConvGeom& g, cudaStream_t s, int64_t* launches);
cudaError_t launch_avg_pool_global_narrow(const void* x, void* y, bool y_is_bf16, int64_t images, int positions, int C,
                                          cudaStream_t s, int64_t* launches);
cudaError_t launch_f32_to_bf16(const float* in, void* out, int64_t n, cudaStream_t s, int64_t* launches);
cudaError_t launch_bf16_to_f32(const void* in, float* out, int64_t n, cudaStream_t s, int64_t* launches);
cudaError_t launch_round_to_bf16_in_place(float* v, int64_t n, cudaStream_t s, int64_t* launches);
// out [r*N, r*K] = r copies of km [N, K] down the diagonal, zeros elsewhere
cudaError_t launch_block_diagonal(const float* km, float* out, int64_t N, int64_t K, int r, cudaStream_t s, int64_t* launches);

// ---- gradients (backprop.cu) ----------------------------------------------------------------------
// `g` is the geometry of the FORWARD op (H, W, C the forward input; Ho, Wo, Co the forward output).
int backprop_slices(int64_t rows, int sm_count);
int sum_rows_slices(int64_t rows, int64_t C, int sm_count);  // slices that launch_sum_rows wants for this shape
cudaError_t launch_conv2d_backprop_input(const float* dy, const float* f, float* dx, const ConvGeom& g, int sm_count,
                                         cudaStream_t s, int64_t* launches);
// `partial` holds slices * fh*fw*C*Co floats (unused when slices == 1)
cudaError_t launch_conv2d_backprop_filter(const float* x, const float* dy, float* df, float* partial, int slices,
                                          const ConvGeom& g, cudaStream_t s, int64_t* launches);
// The input gradient of a stride-1 3x3 depthwise convolution is a forward one over dy (taps reversed): whether the
// 3x3 kernels of depthwise.cu can run it for this forward geometry, and the geometry that they get.
bool depthwise_backprop_is_forward(const ConvGeom& g);
ConvGeom depthwise_backprop_geometry(const ConvGeom& g);
// The same for fh*fw*Cin <= 32 and Cout % 4 == 0 (the first layer's filter); `partial` holds slices * fh*fw*C*Co floats.
bool conv2d_small_filter_supported(const ConvGeom& g);
int conv2d_small_filter_slices(const ConvGeom& g, int sm_count);
cudaError_t launch_conv2d_small_filter(const float* x, const float* dy, float* df, float* partial, int slices, const ConvGeom& g,
                                       cudaStream_t s, int64_t* launches);
cudaError_t launch_depthwise_backprop_input(const float* dy, const float* f, float* dx, const ConvGeom& g, int sm_count,
                                            cudaStream_t s, int64_t* launches);
// `partial` holds slices * fh*fw*Co floats (unused when slices == 1)
cudaError_t launch_depthwise_backprop_filter(const float* x, const float* dy, float* df, float* partial, int slices,
                                             const ConvGeom& g, cudaStream_t s, int64_t* launches);
// Gradients of conv2d on the tensor cores (conv_grad_tcgen05.cu).  fp32 results: operands as two TF32 values each, except
// the filter gradient with `split` false, which reads them as TF32.  Scratch for partial sums is the context's.
bool conv2d_grad_input_supported(const ConvGeom& g);
double conv2d_grad_input_us(const ConvGeom& g, int sm_count);  // estimate for stride 1, to compare it with patches
bool conv2d_grad_input_preferred(const ConvGeom& g, int sm_count);  // to the CUDA-core kernel (TFJSB_GRAD_INPUT=1: always)
tfjsb_status run_conv2d_grad_input(tfjsb_ctx* ctx, const float* dy, const float* f, float* dx, const ConvGeom& g, cudaStream_t s);
bool conv2d_grad_filter_supported(const ConvGeom& g);
tfjsb_status run_conv2d_grad_filter(tfjsb_ctx* ctx, const float* x, const float* dy, float* df, const ConvGeom& g, bool split, cudaStream_t s);
// A row-major fp32 tensor of up to four dimensions, innermost first, copied in boxes (conv_grad_tcgen05.cu).
tfjsb_status encode_tile_map(tfjsb_ctx* ctx, CUtensorMap* map, const float* base, int rank, const int64_t* dims, const uint32_t* box, const char* what,
                             CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B);
// conv2d 3x3 with stride 1 from input patches (conv_patch_tcgen05.cu): the forward pass with TF32 operands, f as it is stored,
// and the input gradient with fp32 accuracy; `g` is the forward geometry of both.
bool conv_patch_input_preferred(const ConvGeom& g, int sm_count);
tfjsb_status run_conv_patch_input(tfjsb_ctx* ctx, const float* x, const float* f, const float* bias, int act, float* y, const ConvGeom& g, cudaStream_t s);
bool conv_patch_gradient_preferred(const ConvGeom& g, int sm_count);
tfjsb_status run_conv_patch_gradient(tfjsb_ctx* ctx, const float* dy, const float* f, float* dx, const ConvGeom& g, cudaStream_t s);
// Pipelined filter gradient of the 3x3 depthwise convolution (depthwise_grad.cu); depthwise_grad_plan says whether the
// shape is one of its own.  `partial` holds slices * 9 * C floats (unused when slices == 1).
struct DepthwiseGradPlan {
    CUtensorMap map_x, map_dy;
    const float *x = nullptr, *dy = nullptr;
    ConvGeom g{};
    int variant = 0, th = 0, tw = 0, thin = 0, twin = 0, stage_bytes = 0, stages = 0;
    int tiles_x = 0, tiles_y = 0, c_blocks = 0, num_tiles = 0, slices = 0;
};
bool depthwise_grad_plan(tfjsb_ctx* ctx, const float* x, const float* dy, const ConvGeom& g, DepthwiseGradPlan* plan);
cudaError_t launch_depthwise_grad(const DepthwiseGradPlan& plan, float* df, float* partial, unsigned int* dev_status, cudaStream_t s,
                                  int64_t* launches);
cudaError_t launch_act_backprop(const float* y, const float* dy, float* dz, int64_t n, int act, int sm_count, cudaStream_t s,
                                int64_t* launches);
// out[c] = sum_r in[r, c]; with slices > 1 in two steps through `partial` (slices * C floats)
cudaError_t launch_sum_rows(const float* in, float* out, float* partial, int64_t rows, int64_t C, int slices, cudaStream_t s,
                            int64_t* launches);
// out[b, c, r] = in[b, r, c] for `batches` matrices [rows, cols] stored one after the other
cudaError_t launch_transpose_batched(const float* in, float* out, int64_t batches, int64_t rows, int64_t cols, cudaStream_t s,
                                     int64_t* launches);

// Fused depthwise 3x3 (stride 1) + pointwise block: the depthwise output is produced straight into
// the tensor-core operand layout in shared memory and never written to global memory.
// `bt` is the pointwise filter stored [Cout, Cin] (K-contiguous).
struct DwPwPlan {
    CUtensorMap map_x, map_b, map_y;
    ConvGeom g{};   // geometry of the depthwise layer
    int Co = 0;
    int block_n = 0, n_sub = 1, acc_stages = 0, patch_stages = 0, a_stages = 0, b_stages = 0;
    bool b_resident = false;  // the B ring holds all of Bt for the whole kernel
    bool wide_epi = false;    // sixteen epilogue warps and one depthwise group (one k-block per tile)
    int tiles_x = 0, tiles_y = 0, num_tiles = 0, grid = 0;
    size_t smem_bytes = 0;
    int patch_bytes = 0, patch_stride = 0;
    // small-window convolution mode of the same kernel
    bool conv = false;
    bool y_bf16 = false;  // the output tensor is bfloat16 (narrow storage): small-window mode only
    int row_floats = 0, patch_rows = 0;
};
bool dwpw_fused_supported(const ConvGeom& dw, int64_t Cout);
// `narrow`: x and y are bfloat16 (narrow storage), bt holds bfloat16 values as fp32
tfjsb_status dwpw_fused_plan(tfjsb_ctx* ctx, const void* x, const float* bt, void* y, const ConvGeom& dw,
                             int64_t Cout, DwPwPlan* plan, bool narrow = false);
// conv2d with fh*fw*Cin <= 32 on the same kernel (input patch by bulk tensor copy, im2col in shared
// memory); `bt` is the filter packed [Cout, 32].  Launched with launch_dwpw_fused (pw_bias / pw_act = the
// convolution's bias and activation; the depthwise arguments are ignored).
bool conv_small_window_supported(const ConvGeom& g);
tfjsb_status conv_small_window_plan(tfjsb_ctx* ctx, const float* x, const float* bt, void* y, const ConvGeom& g, DwPwPlan* plan,
                             bool y_bf16 = false);
cudaError_t launch_dwpw_fused(const DwPwPlan& plan, const float* dw_filter, const float* dw_bias, int dw_act,
                              const float* pw_bias, int pw_act, unsigned int* dev_status, cudaStream_t s,
                              int64_t* launches);

// ---- several layers as one kernel (chain_cluster.cu) ----------------------------------------------------
enum ChainKind { CHAIN_STEM, CHAIN_BLOCK, CHAIN_POOL, CHAIN_DENSE, CHAIN_SOFTMAX };
struct ChainOp {
    int kind = CHAIN_SOFTMAX;
    int H = 0, W = 0, C = 0, Ho = 0, Wo = 0, Co = 0;  // of one image; dense and softmax: C -> Co
    int sh = 1, sw = 1, dh = 1, dw = 1, pt = 0, pl = 0;
    int act1 = 0, act2 = 0;                 // after the depthwise part, after the step
    int round1 = 0, round2 = 0, store_bf16 = 0;  // round to bfloat16 (stem: its input), and how the result is stored
    // a block's tiles: `pixels` rows for one of `groups` groups of `group_cols` columns is a unit; columns are multiplied
    // `tile_cols` at a time by warp tiles of `variant`'s shape, K divided among `k_splits` warps
    int pixels = 0, groups = 1, group_cols = 0, tile_cols = 0, units = 0, variant = 0, k_splits = 1;
    int w_stride = 0, chunk_rows = 0, n_chunks = 0, chunk_floats = 0, group_tiles = 0, tasks = 0, task_n = 0, task_rows = 0, task_cols = 0, lanes = 0, strip = 1;
    // ceil(2^32 / d) for the divisors Wo, groups, tile_cols / 4 (stem: w_stride), C / 4 (stem: in_row), tasks, task_n (0 for
    // d = 1)
    unsigned int by_wo = 0, by_groups = 0, by_pieces = 0, by_quads = 0, by_tasks = 0, by_task_n = 0;
    float lo1 = 0, hi1 = 0, lo2 = 0, hi2 = 0;       // the activations as bounds
    int in_row = 0, out_row = 0, out_origin = 0;    // floats between rows of the input and of the output, and its first element
    int64_t out_buffer = 0;                         // in the cluster's workspace
    const float *f1 = nullptr, *b1 = nullptr, *f2 = nullptr, *b2 = nullptr;  // depthwise (stem, dense) and pointwise [C,Co]
    // Layers' own output tensors that a caller may read after the run: of the operation, [images][Ho Wo][Co], and of a
    // block's depthwise part, [images][Ho Wo][C]
    float *also = nullptr, *also_dw = nullptr;
    int also_bf16 = 0, also_dw_bf16 = 0;
};
constexpr int CHAIN_MAX_OPS = 22;
struct ChainArgs {
    ChainOp ops[CHAIN_MAX_OPS];
    int n_ops = 0, cluster_size = 1;
    int64_t images = 0, in_elems = 0, out_elems = 0;  // elements per image
    int64_t cluster_elems = 0;                        // of workspace
    const float* input = nullptr;
    float* output = nullptr;
    float* workspace = nullptr;  // [clusters][cluster_elems], zero before the first launch
    unsigned int* dev_status = nullptr;
};
struct ChainPlan {
    ChainArgs args;
    int blocks = 0;
};
bool chain_stem_supported(const ConvGeom& g);
bool chain_block_supported(const ConvGeom& dw, int64_t Cout);
// Plans the first operations as one kernel where that is estimated to be faster than `separate` ns: rest[k] is what the
// layers after operation k take as their own kernels, negative where the kernel cannot end there.  Fills in everything but
// the pointers and the element counts; returns the number of operations, 0 for none.
int chain_plan(const ChainOp* ops, int n_ops, int64_t images, const double* rest, double separate, ChainPlan* plan);
// The blocks' filters in the plan's layout, `dst` of chain_packed_floats; the plan then refers to them.
int64_t chain_packed_floats(const ChainPlan& plan);
cudaError_t chain_pack(ChainPlan* plan, float* dst, cudaStream_t s, int64_t* launches);
cudaError_t launch_chain(const ChainPlan& plan, const float* input, float* output, unsigned int* dev_status, cudaStream_t s,
                         int64_t* launches);

}  // namespace tfjsb
