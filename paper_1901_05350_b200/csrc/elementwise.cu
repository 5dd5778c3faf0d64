// Bandwidth-bound helpers: the standalone bias+activation op, avgPool, softmax, and the
// 2-D transpose used to make matMul operands K-contiguous.
#include "common.cuh"
#include "ptx_sm100.cuh"

namespace tfjsb {

namespace {

constexpr int kThreads = 256;

inline int grid_for(int64_t work_items, int threads, int max_blocks) {
    int64_t b = (work_items + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > max_blocks) b = max_blocks;
    return (int)b;
}

// The elementwise kernels take STRIDED items per thread and pass, a grid apart, and load all of them before they store the
// first (add of 2 x 25.7 MB: 7.0 us, with one or two loads in flight per thread 8.3).
constexpr int STRIDED = 4;

// i % period, in 32 bits where they do (the 64-bit remainder is a hundred instructions)
__device__ __forceinline__ int64_t wrap(int64_t i, int64_t period) {
    return (uint64_t)i < (1ull << 32) && (uint64_t)period < (1ull << 32) ? (int64_t)((uint32_t)i % (uint32_t)period) : i % period;
}

// ---- bias + activation ----------------------------------------------------------------------
// out[r, c] = act(x[r, c] + bias[c]).  float4 path: C % 4 == 0, so a float4 never straddles rows.
__global__ void bias_act_vec4_kernel(const float4* x, const float* bias, float4* y, int64_t n_vec, int C4, int act) {
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_vec; i += STRIDED * stride) {
        float4 v[STRIDED];
#pragma unroll
        for (int u = 0; u < STRIDED; ++u)
            if (i + u * stride < n_vec) v[u] = x[i + u * stride];
#pragma unroll
        for (int u = 0; u < STRIDED; ++u) {
            const int64_t at = i + u * stride;
            if (at >= n_vec) break;
            if (bias) {
                const float4 b = load_global(reinterpret_cast<const float4*>(bias) + wrap(at, C4));
                v[u].x = v[u].x + b.x; v[u].y = v[u].y + b.y; v[u].z = v[u].z + b.z; v[u].w = v[u].w + b.w;
            }
            v[u].x = apply_act(v[u].x, act); v[u].y = apply_act(v[u].y, act);
            v[u].z = apply_act(v[u].z, act); v[u].w = apply_act(v[u].w, act);
            y[at] = v[u];
        }
    }
}

// Here and in binary_scalar_kernel the grid is one wave of blocks and the next kernel starts as this one ends (see
// avg_pool_window_kernel).  9 million values of 63 channels: 18.3 us with two waves, an early start and a 32-bit remainder, 15.8 so;
// 1.7 million 5.9 and 4.7; 26 million 57.5 and 55.7 (53.3 through the read-only path).
__global__ void bias_act_scalar_kernel(const float* x, const float* bias, float* y, int64_t n, int64_t C, int act) {
    ptx::pdl_wait();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        float v = x[i];
        if (bias) v = v + bias[i % C];
        y[i] = apply_act(v, act);
    }
}

// ---- avgPool ----------------------------------------------------------------------------------
// The pools over windows let the next kernel start as they end, not before: blocks of it that wait beside the last ones of a
// pool that is two waves of small blocks are spread unevenly over the SMs (one avgPool 3 x 3 after another, [64,112,112,64]
// 812 us with an early start, 787 without; [8,33,35,36] / 2 5.0 and 3.5).
// One thread per output element, channel fastest (coalesced).  Padding never counts.
__global__ void avg_pool_window_kernel(const float* x, float* __restrict__ y, ConvGeom g,
                                       int64_t n_out) {
    ptx::pdl_wait();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_out; i += stride) {
        const int c = (int)(i % g.C);
        int64_t t = i / g.C;
        const int ox = (int)(t % g.Wo); t /= g.Wo;
        const int oy = (int)(t % g.Ho);
        const int64_t n = t / g.Ho;
        float acc = 0.0f;
        int count = 0;
        for (int ky = 0; ky < g.fh; ++ky) {
            const int iy = oy * g.sh - g.pt + ky;
            if (iy < 0 || iy >= g.H) continue;
            for (int kx = 0; kx < g.fw; ++kx) {
                const int ix = ox * g.sw - g.pl + kx;
                if (ix < 0 || ix >= g.W) continue;
                acc += x[((n * g.H + iy) * (int64_t)g.W + ix) * g.C + c];
                ++count;
            }
        }
        y[i] = acc / (float)count;
    }
}

// ---- maxPool ----------------------------------------------------------------------------------
// One thread per output element, channel fastest (coalesced).  Padding never takes part; max.NaN keeps
// a NaN that is in the window.
__global__ void max_pool_window_kernel(const float* x, float* __restrict__ y, ConvGeom g,
                                       int64_t n_out) {
    ptx::pdl_wait();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_out; i += stride) {
        const int c = (int)(i % g.C);
        int64_t t = i / g.C;
        const int ox = (int)(t % g.Wo); t /= g.Wo;
        const int oy = (int)(t % g.Ho);
        const int64_t n = t / g.Ho;
        float m = __int_as_float(0xff800000);  // -inf
        for (int ky = 0; ky < g.fh; ++ky) {
            const int iy = oy * g.sh - g.pt + ky;
            if (iy < 0 || iy >= g.H) continue;
            for (int kx = 0; kx < g.fw; ++kx) {
                const int ix = ox * g.sw - g.pl + kx;
                if (ix < 0 || ix >= g.W) continue;
                const float v = x[((n * g.H + iy) * (int64_t)g.W + ix) * g.C + c];
                asm("max.NaN.f32 %0, %0, %1;" : "+f"(m) : "f"(v));
            }
        }
        y[i] = m;
    }
}

// The same with four channels per thread (C % 4 == 0): one 16-byte load per window element, a warp
// reads 512 contiguous bytes per tap; neighbouring outputs' windows overlap in L1/L2.
__device__ __forceinline__ void max4_nan(float4& m, const float4& v) {
    asm("max.NaN.f32 %0, %0, %1;" : "+f"(m.x) : "f"(v.x));
    asm("max.NaN.f32 %0, %0, %1;" : "+f"(m.y) : "f"(v.y));
    asm("max.NaN.f32 %0, %0, %1;" : "+f"(m.z) : "f"(v.z));
    asm("max.NaN.f32 %0, %0, %1;" : "+f"(m.w) : "f"(v.w));
}
// W: windows of up to W x W, all samples on their way before the first comparison, -inf where there is none; 0: any window, one
// sample after the other (ld_global: with loads that the compiler may move, 5 x 5 over [32,55,55,172] takes 146 us, 117 so).
// [32,55,55,172]: 3 x 3 / 2 22.6 us with W = 0 and 17.6 with W = 3, 2 x 2 / 2 16.5 and 10.2 with W = 2 (17.3 with W = 3), 1 x 3
// 41.9 with W = 0 and 45.8 with W = 3.
template <int W>
__global__ void max_pool_vec4_kernel(const float* x, float* __restrict__ y, ConvGeom g, int64_t n_out4) {
    ptx::pdl_wait();
    const int C4 = g.C >> 2;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_out4; i += stride) {
        const int c = (int)(i % C4) * 4;
        int64_t t = i / C4;
        const int ox = (int)(t % g.Wo); t /= g.Wo;
        const int oy = (int)(t % g.Ho);
        const int64_t n = t / g.Ho;
        const float ninf = __int_as_float(0xff800000);
        float4 m = make_float4(ninf, ninf, ninf, ninf);
        const int iy0 = oy * g.sh - g.pt, ix0 = ox * g.sw - g.pl;
        const int ky0 = iy0 < 0 ? -iy0 : 0, ky1 = min(g.fh, g.H - iy0);
        const int kx0 = ix0 < 0 ? -ix0 : 0, kx1 = min(g.fw, g.W - ix0);
        if constexpr (W > 0) {
            float4 v[W][W];
#pragma unroll
            for (int ky = 0; ky < W; ++ky)
#pragma unroll
                for (int kx = 0; kx < W; ++kx) {
                    v[ky][kx] = m;
                    if (ky >= ky0 && ky < ky1 && kx >= kx0 && kx < kx1)
                        v[ky][kx] = load_global(reinterpret_cast<const float4*>(x + ((n * g.H + iy0 + ky) * (int64_t)g.W + ix0 + kx) * g.C + c));
                }
#pragma unroll
            for (int k = 0; k < W * W; ++k) max4_nan(m, v[k / W][k % W]);
        } else {
            for (int ky = ky0; ky < ky1; ++ky) {
                const float* row = x + ((n * g.H + iy0 + ky) * (int64_t)g.W + ix0) * g.C + c;
                for (int kx = kx0; kx < kx1; ++kx) max4_nan(m, ld_global4(row + (int64_t)kx * g.C));
            }
        }
        *reinterpret_cast<float4*>(y + i * 4) = m;
    }
}

// ---- elementwise binary ops (the addition shader of the paper's Fig. 3: one output value per thread) ----
// out[i] = a[i] op b[i % b_len]; OP 0 add, 1 subtract, 2 multiply: one fp32 operation, so bit-exact.
template <int OP>
__device__ __forceinline__ float binary_op(float u, float v) {
    return OP == 0 ? __fadd_rn(u, v) : (OP == 1 ? __fsub_rn(u, v) : __fmul_rn(u, v));
}
// float4 path: n and b_len multiples of 4 (a float4 never straddles a period of b)
template <int OP>
__global__ void binary_vec4_kernel(const float4* a, const float4* b, float4* out, int64_t n4, int64_t b_len4) {
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += STRIDED * stride) {
        float4 u[STRIDED], v[STRIDED];
#pragma unroll
        for (int k = 0; k < STRIDED; ++k) {
            const int64_t at = i + k * stride;
            if (at >= n4) break;
            u[k] = a[at];
            v[k] = b[b_len4 == n4 ? at : wrap(at, b_len4)];
        }
#pragma unroll
        for (int k = 0; k < STRIDED; ++k) {
            if (i + k * stride >= n4) break;
            out[i + k * stride] = make_float4(binary_op<OP>(u[k].x, v[k].x), binary_op<OP>(u[k].y, v[k].y), binary_op<OP>(u[k].z, v[k].z),
                                              binary_op<OP>(u[k].w, v[k].w));
        }
    }
}
template <int OP>
__global__ void binary_scalar_kernel(const float* a, const float* b, float* out, int64_t n, int64_t b_len) {
    ptx::pdl_wait();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        out[i] = binary_op<OP>(a[i], b[i % b_len]);
}

// Global pools of more positions than this (2 us) are launched after the kernel before: early, their blocks, fewer than SMs as a
// rule, are put several to an SM and share its bandwidth for as long as they run ([34,45,45,336], 102 blocks, 16.5 us and 37.6;
// [59,79,79,64] 45 and 101; after a pointwise convolution of 100352 pixels the pair 76 and 155).
constexpr int SHORT_POOL = 256;

// Global pool: a block owns (image n, 128 consecutive channels).  Lane = 4 channels (one float4, so a
// warp reads 512 contiguous bytes per position), the 8 warps stride over the H*W positions, partial
// sums meet in shared memory.  C % 4 == 0.
template <int U>
__device__ __forceinline__ void add_positions(float4& acc, const float* base, int p, int C) {
    float4 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = ld_global4(base + (int64_t)(p + 8 * u) * C);
#pragma unroll
    for (int u = 0; u < U; ++u) { acc.x += v[u].x; acc.y += v[u].y; acc.z += v[u].z; acc.w += v[u].w; }
}
__global__ void avg_pool_global_vec4_kernel(const float* x, float* __restrict__ y, int HW, int C) {
    __shared__ float4 partial[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = (blockIdx.x * 32 + lane) * 4;
    const int64_t n = blockIdx.y;
    if (HW <= SHORT_POOL) ptx::pdl_launch_dependents();
    ptx::pdl_wait();
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c < C) {
        const float* base = x + n * (int64_t)HW * C + c;
        // eight loads in flight per thread, then four (the sum order stays p ascending); ld_global: [59,79,79,64] 35.9 us, 40.3 with
        // loads that the compiler may move and 41.0 with four of those
        int p = warp;
        for (; p + 56 < HW; p += 64) add_positions<8>(acc, base, p, C);
        for (; p + 24 < HW; p += 32) add_positions<4>(acc, base, p, C);
        for (; p < HW; p += 8) {
            const float4 v = *reinterpret_cast<const float4*>(base + (int64_t)p * C);
            acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
        }
    }
    partial[warp][lane] = acc;
    __syncthreads();
    if (warp == 0 && c < C) {
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const float4 v = partial[w][lane];
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        const float inv = (float)HW;
        *reinterpret_cast<float4*>(y + n * C + c) = make_float4(s.x / inv, s.y / inv, s.z / inv, s.w / inv);
    }
}

// The same with one channel per lane, for channel counts that are not multiples of 4.
__global__ void avg_pool_global_kernel(const float* x, float* __restrict__ y, int HW, int C) {
    __shared__ float partial[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * 32 + lane;
    const int64_t n = blockIdx.y;
    if (HW <= SHORT_POOL) ptx::pdl_launch_dependents();
    ptx::pdl_wait();
    float acc = 0.0f;
    if (c < C) {
        const float* base = x + n * (int64_t)HW * C + c;
        int p = warp;
        for (; p + 56 < HW; p += 64) {  // eight loads in flight
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = load_global(base + (int64_t)(p + 8 * u) * C);
#pragma unroll
            for (int u = 0; u < 8; ++u) acc += v[u];
        }
        for (; p < HW; p += 8) acc += load_global(base + (int64_t)p * C);
    }
    partial[warp][lane] = acc;
    __syncthreads();
    if (warp == 0 && c < C) {
        float s = 0.0f;
#pragma unroll
        for (int w = 0; w < 8; ++w) s += partial[w][lane];
        y[n * C + c] = s / (float)HW;
    }
}

// ---- softmax ----------------------------------------------------------------------------------
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Rows of more columns than this are launched after the kernel before, as long global pools are: 60 rows of 30000 columns and an add
// of 16.8 MB take 25 us so and 36 launched early; 100 rows of 4096 and the add 9.1 early, 10.4 so.
constexpr int64_t SHORT_ROW = 4096;

// One block (kThreads) per row: max, then sum of exp(x - max), then the quotient.
__global__ void softmax_rows_kernel(const float* x, float* __restrict__ y, int64_t cols) {
    __shared__ float red[kThreads / 32];
    __shared__ float bcast;
    const float* xr = x + (int64_t)blockIdx.x * cols;
    float* yr = y + (int64_t)blockIdx.x * cols;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (cols <= SHORT_ROW) ptx::pdl_launch_dependents();
    ptx::pdl_wait();

    float m = -INFINITY;
    for (int64_t j = threadIdx.x; j < cols; j += kThreads) m = fmaxf(m, xr[j]);
    m = warp_max(m);
    if (lane == 0) red[warp] = m;
    __syncthreads();
    if (warp == 0) {
        float v = lane < kThreads / 32 ? red[lane] : -INFINITY;
        v = warp_max(v);
        if (lane == 0) bcast = v;
    }
    __syncthreads();
    m = bcast;

    float sum = 0.0f;
    for (int64_t j = threadIdx.x; j < cols; j += kThreads) sum += expf(xr[j] - m);
    sum = warp_sum(sum);
    __syncthreads();  // red[] and bcast are reused
    if (lane == 0) red[warp] = sum;
    __syncthreads();
    if (warp == 0) {
        float v = lane < kThreads / 32 ? red[lane] : 0.0f;
        v = warp_sum(v);
        if (lane == 0) bcast = v;
    }
    __syncthreads();
    sum = bcast;

    for (int64_t j = threadIdx.x; j < cols; j += kThreads) yr[j] = expf(xr[j] - m) / sum;
}

// ---- transpose --------------------------------------------------------------------------------
// out[b, c, r] = in[b, r, c]: a 32 x 32 tile through shared memory per block.  The grid covers (columns, rows, matrices) and
// walks on over rows and matrices beyond its limits.
__global__ void transpose_kernel(const float* in, float* __restrict__ out, int64_t batches, int64_t rows, int64_t cols) {
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();
    __shared__ float tile[32][33];
    const int64_t c0 = (int64_t)blockIdx.x * 32;
    for (int64_t b = blockIdx.z; b < batches; b += gridDim.z) {
        const float* from = in + b * rows * cols;
        float* to = out + b * rows * cols;
        for (int64_t r0 = (int64_t)blockIdx.y * 32; r0 < rows; r0 += (int64_t)gridDim.y * 32) {
            for (int j = threadIdx.y; j < 32; j += 8) {
                const int64_t r = r0 + j, c = c0 + threadIdx.x;
                if (r < rows && c < cols) tile[j][threadIdx.x] = from[r * cols + c];
            }
            __syncthreads();
            for (int j = threadIdx.y; j < 32; j += 8) {
                const int64_t c = c0 + j, r = r0 + threadIdx.x;
                if (r < rows && c < cols) to[c * rows + r] = tile[threadIdx.x][j];
            }
            __syncthreads();
        }
    }
}

// ---- filter packing for the implicit-GEMM convolution ------------------------------------------------
// out[n, t * c_pad + c] = c < C ? f[t, c, n] : 0.  A 32 x 32 transpose through shared memory per block, so that both
// sides are read and written in 128-byte runs.
__global__ void pack_filter_kernel(const float* f, float* __restrict__ out, int64_t C, int64_t N, int64_t c_pad) {
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();
    __shared__ float tile[32][33];
    const int64_t n0 = (int64_t)blockIdx.x * 32, t = blockIdx.z;
    for (int64_t c0 = (int64_t)blockIdx.y * 32; c0 < c_pad; c0 += (int64_t)gridDim.y * 32) {
        for (int j = threadIdx.y; j < 32; j += 8) {
            const int64_t c = c0 + j, n = n0 + threadIdx.x;
            tile[j][threadIdx.x] = c < C && n < N ? f[(t * C + c) * N + n] : 0.0f;
        }
        __syncthreads();
        for (int j = threadIdx.y; j < 32; j += 8) {
            const int64_t n = n0 + j, c = c0 + threadIdx.x;
            if (n < N && c < c_pad) out[(n * gridDim.z + t) * c_pad + c] = tile[threadIdx.x][j];
        }
        __syncthreads();
    }
}

}  // namespace

cudaError_t launch_pack_filter(const float* f, float* out, int64_t taps, int64_t C, int64_t N, int64_t c_pad, cudaStream_t s,
                               int64_t* launches) {
    if (taps * N * c_pad == 0) return cudaSuccess;
    if (taps > 65535) return cudaErrorInvalidConfiguration;  // im2col copies have 128 x 128 at most
    const int64_t gy = (c_pad + 31) / 32;                    // the grid walks on where there are more
    ++*launches;
    return launch_k(pack_filter_kernel, dim3((unsigned)((N + 31) / 32), (unsigned)(gy < 65535 ? gy : 65535), (unsigned)taps), dim3(32, 8), 0, s, f, out, C, N, c_pad);
}

cudaError_t launch_bias_act(const float* x, const float* bias, float* y, int64_t rows, int64_t C, int act,
                            cudaStream_t s, int64_t* launches) {
    const int64_t n = rows * C;
    if (n == 0) return cudaSuccess;
    ++*launches;
    if (C % 4 == 0) {
        const int64_t n_vec = n / 4;
        return launch_k(bias_act_vec4_kernel, dim3(grid_for(n_vec, kThreads, current_sm_count() * 16)), dim3(kThreads), 0, s,
                        reinterpret_cast<const float4*>(x), bias, reinterpret_cast<float4*>(y), n_vec, (int)(C / 4), act);
    }
    return launch_k(bias_act_scalar_kernel, dim3(grid_for(n, kThreads, current_sm_count() * 8)), dim3(kThreads), 0, s, x, bias, y, n, C, act);
}

cudaError_t launch_avg_pool(const float* x, float* y, const ConvGeom& g, cudaStream_t s, int64_t* launches) {
    const int64_t n_out = g.N * g.Ho * g.Wo * g.C;
    if (n_out == 0) return cudaSuccess;
    const bool global = g.Ho == 1 && g.Wo == 1 && g.fh == g.H && g.fw == g.W && g.pt == 0 && g.pl == 0 &&
                        g.N <= 65535;
    ++*launches;
    if (!global) return launch_k(avg_pool_window_kernel, dim3(grid_for(n_out, kThreads, current_sm_count() * 16)), dim3(kThreads), 0, s, x, y, g, n_out);
    auto global_kernel = g.C % 4 == 0 ? avg_pool_global_vec4_kernel : avg_pool_global_kernel;
    const dim3 grid(g.C % 4 == 0 ? (g.C / 4 + 31) / 32 : (g.C + 31) / 32, (unsigned)g.N);
    return launch_k_if(g.H * g.W <= SHORT_POOL, global_kernel, grid, dim3(256), 0, s, x, y, g.H * g.W, g.C);
}

cudaError_t launch_max_pool(const float* x, float* y, const ConvGeom& g, cudaStream_t s, int64_t* launches) {
    const int64_t n_out = g.N * g.Ho * g.Wo * g.C;
    if (n_out == 0) return cudaSuccess;
    ++*launches;
    auto vec4 = g.fh <= 2 && g.fw <= 2 ? max_pool_vec4_kernel<2> : g.fh == 3 && g.fw == 3 ? max_pool_vec4_kernel<3> : max_pool_vec4_kernel<0>;
    if (g.C % 4 == 0)
        return launch_k(vec4, dim3(grid_for(n_out / 4, kThreads, current_sm_count() * 32)), dim3(kThreads), 0, s, x, y, g, n_out / 4);
    return launch_k(max_pool_window_kernel, dim3(grid_for(n_out, kThreads, current_sm_count() * 16)), dim3(kThreads), 0, s, x, y, g, n_out);
}

template <int OP>
static cudaError_t launch_binary_op(const float* a, const float* b, float* out, int64_t n, int64_t b_len, cudaStream_t s) {
    if (n % 4 == 0 && b_len % 4 == 0)
        return launch_k(binary_vec4_kernel<OP>, dim3(grid_for(n / 4, kThreads, current_sm_count() * 16)), dim3(kThreads), 0, s,
                        reinterpret_cast<const float4*>(a), reinterpret_cast<const float4*>(b), reinterpret_cast<float4*>(out), n / 4, b_len / 4);
    return launch_k(binary_scalar_kernel<OP>, dim3(grid_for(n, kThreads, current_sm_count() * 8)), dim3(kThreads), 0, s, a, b, out, n, b_len);
}

cudaError_t launch_binary(int op, const float* a, const float* b, float* out, int64_t n, int64_t b_len, cudaStream_t s,
                          int64_t* launches) {
    if (n == 0) return cudaSuccess;
    ++*launches;
    if (op == TFJSB_BINARY_ADD) return launch_binary_op<0>(a, b, out, n, b_len, s);
    if (op == TFJSB_BINARY_SUB) return launch_binary_op<1>(a, b, out, n, b_len, s);
    return launch_binary_op<2>(a, b, out, n, b_len, s);
}

cudaError_t launch_softmax(const float* x, float* y, int64_t rows, int64_t cols, cudaStream_t s,
                           int64_t* launches) {
    if (rows == 0) return cudaSuccess;
    // gridDim.x is 2^31-1: enough for any tensor that fits in memory
    cudaError_t e = launch_k_if(cols <= SHORT_ROW, softmax_rows_kernel, dim3((unsigned)rows), dim3(kThreads), 0, s, x, y, cols);
    ++*launches;
    return e;
}

cudaError_t launch_transpose_batched(const float* in, float* out, int64_t batches, int64_t rows, int64_t cols, cudaStream_t s,
                                     int64_t* launches) {
    if (rows == 0 || cols == 0 || batches == 0) return cudaSuccess;
    const int64_t gy = (rows + 31) / 32;
    const dim3 grid((unsigned)((cols + 31) / 32), (unsigned)(gy < 65535 ? gy : 65535), (unsigned)(batches < 65535 ? batches : 65535));
    ++*launches;
    return launch_k(transpose_kernel, grid, dim3(32, 8), 0, s, in, out, batches, rows, cols);
}

cudaError_t launch_transpose(const float* in, float* out, int64_t rows, int64_t cols, cudaStream_t s, int64_t* launches) {
    return launch_transpose_batched(in, out, 1, rows, cols, s, launches);
}

}  // namespace tfjsb
