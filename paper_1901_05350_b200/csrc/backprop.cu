// Gradient kernels of conv2d, depthwiseConv2d and the bias + activation epilogue (the per-kernel
// gradient functions that eager differentiation calls, Sec. 3.5 of the paper): CUDA-core kernels for
// any window, stride and dilation.  The pointwise (1x1, stride 1) convolution, whose two gradients are
// plain matrix products, runs on the tensor-core GEMMs instead (see the entry points in api.cu).
//
//   dx[n,iy,ix,ci]   = sum over the (output pixel, tap) pairs that read (iy,ix) in the forward pass, and co,
//                      of dy[n,oy,ox,co] * f[ky,kx,ci,co]
//   df[ky,kx,ci,co]  = sum over n,oy,ox of x[n, oy*sh - pt + ky*dh, ox*sw - pl + kx*dw, ci] * dy[n,oy,ox,co]
// and the depthwise forms with co = c*mult + q.  Sums over pixels (filter and bias gradients) are taken
// in two steps, partial sums per slice of the pixels into scratch and then a sum over the slices in slice
// order, so that the result does not depend on scheduling.
#include "common.cuh"
#include "ptx_sm100.cuh"

namespace tfjsb {

namespace {

constexpr int BP_THREADS = 256;

// Output row / column that tap k of a forward window maps input coordinate i to, or -1 when none does:
// o*s - p + k*d = i.
__device__ __forceinline__ int source_of(int i, int p, int k, int d, int s, int limit) {
    const int t = i + p - k * d;
    if (t < 0) return -1;
    const int o = t / s;
    return (o * s == t && o < limit) ? o : -1;
}

// ---- conv2d, gradient with respect to the input ---------------------------------------------------
// thread = one input sample (n, iy, ix, ci), ci fastest; the dy row of a source pixel is the same address
// for the threads of a pixel (a broadcast), the filter row f[tap, ci, :] is contiguous per thread.
__global__ void __launch_bounds__(BP_THREADS)
conv2d_backprop_input_kernel(const float* dy, const float* f, float* __restrict__ dx, ConvGeom g,
                             int64_t total) {
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += stride) {
        const int ci = (int)(e % g.C);
        int64_t p = e / g.C;
        const int ix = (int)(p % g.W);
        p /= g.W;
        const int iy = (int)(p % g.H);
        const int64_t n = p / g.H;
        float acc = 0.f;
        for (int ky = 0; ky < g.fh; ++ky) {
            const int oy = source_of(iy, g.pt, ky, g.dh, g.sh, g.Ho);
            if (oy < 0) continue;
            for (int kx = 0; kx < g.fw; ++kx) {
                const int ox = source_of(ix, g.pl, kx, g.dw, g.sw, g.Wo);
                if (ox < 0) continue;
                const float* gp = dy + ((n * g.Ho + oy) * (int64_t)g.Wo + ox) * g.Co;
                const float* fp = f + ((int64_t)(ky * g.fw + kx) * g.C + ci) * g.Co;
                for (int co = 0; co < g.Co; ++co) acc = fmaf(load_global(gp + co), load_global(fp + co), acc);
            }
        }
        dx[e] = acc;
    }
}

// ---- conv2d, gradient with respect to the filter: partial sums ---------------------------------------
// Block = a 32 x 32 tile of (ci, co) for one tap and one slice of the output pixels; 32 pixels at a time go
// through shared memory (x samples [32 pixels][32 ci], dy [32 pixels][32 co]); thread (tx = co, ty = ci).
__global__ void __launch_bounds__(1024)
conv2d_backprop_filter_partial_kernel(const float* x, const float* dy, float* __restrict__ partial,
                                      ConvGeom g, int64_t pixels, int64_t pixels_per_slice, int ci_tiles, int co_tiles) {
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();
    __shared__ float xs[32][33];
    __shared__ float gs[32][33];
    int b = blockIdx.x;
    const int co0 = (b % co_tiles) * 32;
    b /= co_tiles;
    const int ci0 = (b % ci_tiles) * 32;
    const int tap = b / ci_tiles;
    const int ky = tap / g.fw, kx = tap - ky * g.fw;
    const int slice = blockIdx.y;
    const int64_t p_begin = (int64_t)slice * pixels_per_slice;
    const int64_t p_end = min(pixels, p_begin + pixels_per_slice);
    const int tx = threadIdx.x, ty = threadIdx.y;
    float acc = 0.f;
    for (int64_t p0 = p_begin; p0 < p_end; p0 += 32) {
        // row ty of both tiles is output pixel p0 + ty; column tx is channel ci0 + tx (resp. co0 + tx)
        const int64_t p = p0 + ty;
        float xv = 0.f, gv = 0.f;
        if (p < p_end) {
            const int ox = (int)(p % g.Wo);
            const int64_t r = p / g.Wo;
            const int oy = (int)(r % g.Ho);
            const int64_t n = r / g.Ho;
            const int iy = oy * g.sh - g.pt + ky * g.dh, ix = ox * g.sw - g.pl + kx * g.dw;
            if (iy >= 0 && iy < g.H && ix >= 0 && ix < g.W && ci0 + tx < g.C)
                xv = load_global(x + ((n * g.H + iy) * (int64_t)g.W + ix) * g.C + ci0 + tx);
            if (co0 + tx < g.Co) gv = load_global(dy + p * g.Co + co0 + tx);
        }
        xs[ty][tx] = xv;
        gs[ty][tx] = gv;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 32; ++k) acc = fmaf(xs[k][ty], gs[k][tx], acc);
        __syncthreads();
    }
    if (ci0 + ty < g.C && co0 + tx < g.Co)
        partial[((int64_t)slice * g.fh * g.fw + tap) * g.C * g.Co + (int64_t)(ci0 + ty) * g.Co + co0 + tx] = acc;
}

// ---- conv2d, gradient with respect to a small filter: partial sums ----------------------------------------
// fh * fw * Cin <= 32 (the 3x3 filter of an RGB image: 27), Cout % 4 == 0.  Block = all window elements x 4 CG output
// channels for one slice of the output pixels, 32 pixels at a time through shared memory: the window's samples, gathered
// ([pixel][32]), and dy ([pixel][4 CG]), the next 32 pixels' values in registers meanwhile.  Thread = 4 window elements x
// 4 channels; a warp reads one 16-byte piece of samples (a broadcast) and up to 512 bytes of dy per pixel for 16
// multiply-adds, so shared memory and the FMA pipe are about equally busy.  With fewer than 32 channel groups the block's
// threads take pixels in turn and meet at the end.  For [49,48,48,3] -> 224 channels:
// 69 + 9 us (101 MB of dy; 22 us of multiply-adds); the 32 x 32 tiles per tap, 3 of 32 rows of each in use, took 3.3 ms.
template <int CG>
__global__ void __launch_bounds__(BP_THREADS)
conv2d_backprop_small_filter_kernel(const float* x, const float* dy, float* __restrict__ partial, ConvGeom g,
                                    int64_t pixels, int64_t pixels_per_slice, int window) {
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();
    constexpr int PIX = 32, LANES = BP_THREADS / (8 * CG), CO = 4 * CG;
    constexpr int DY4 = PIX * CG / BP_THREADS;  // 16-byte pieces of dy per thread and step
    __shared__ __align__(16) float xs[2][PIX][32];
    __shared__ __align__(16) float gs[2][PIX][CO];
    const int tid = threadIdx.x;
    const int co0 = blockIdx.x * CO;
    const int64_t p_begin = (int64_t)blockIdx.y * pixels_per_slice, p_end = min(pixels, p_begin + pixels_per_slice);
    // gathering: this thread's window element, and every eighth pixel
    const int e = tid & 31, first_px = tid >> 5;
    const int tap = e / g.C, ky = tap / g.fw, off_y = ky * g.dh, off_x = (tap - ky * g.fw) * g.dw, ci = e - tap * g.C;
    float xv[PIX / 8];
    float4 gv[DY4];
    auto fetch = [&](int64_t p0) {
        // the thread's pixels p0 + first_px + 8 i: one division, then steps
        int64_t p = p0 + first_px;
        int64_t row = p / g.Wo;
        int ox = (int)(p - row * g.Wo);
        int64_t n = row / g.Ho;
        int oy = (int)(row - n * g.Ho);
#pragma unroll
        for (int i = 0; i < PIX / 8; ++i) {
            const int iy = oy * g.sh - g.pt + off_y, ix = ox * g.sw - g.pl + off_x;
            xv[i] = p < p_end && e < window && iy >= 0 && iy < g.H && ix >= 0 && ix < g.W
                        ? load_global(x + ((n * g.H + iy) * (int64_t)g.W + ix) * g.C + ci) : 0.f;
            p += 8;
            for (ox += 8; ox >= g.Wo; ox -= g.Wo)
                if (++oy == g.Ho) { oy = 0; ++n; }
        }
#pragma unroll
        for (int i = 0; i < DY4; ++i) {
            const int j = tid + i * BP_THREADS, px = j / CG, c = co0 + 4 * (j % CG);
            gv[i] = p0 + px < p_end && c < g.Co ? load_global(reinterpret_cast<const float4*>(dy + (p0 + px) * g.Co + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    const int eg = (tid / CG) & 7, cg = tid % CG, lane = tid / (8 * CG);
    float4 acc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    int buf = 0;
    if (p_begin < p_end) fetch(p_begin);
    for (int64_t p0 = p_begin; p0 < p_end; p0 += PIX, buf ^= 1) {
#pragma unroll
        for (int i = 0; i < PIX / 8; ++i) xs[buf][first_px + 8 * i][e] = xv[i];
#pragma unroll
        for (int i = 0; i < DY4; ++i) {
            const int j = tid + i * BP_THREADS;
            *reinterpret_cast<float4*>(&gs[buf][j / CG][4 * (j % CG)]) = gv[i];
        }
        __syncthreads();
        if (p0 + PIX < p_end) fetch(p0 + PIX);
#pragma unroll 8
        for (int px = lane; px < PIX; px += LANES) {
            const float4 a = *reinterpret_cast<const float4*>(&xs[buf][px][4 * eg]);
            const float4 b = *reinterpret_cast<const float4*>(&gs[buf][px][4 * cg]);
            fma4_packed(acc[0], make_float4(a.x, a.x, a.x, a.x), b);
            fma4_packed(acc[1], make_float4(a.y, a.y, a.y, a.y), b);
            fma4_packed(acc[2], make_float4(a.z, a.z, a.z, a.z), b);
            fma4_packed(acc[3], make_float4(a.w, a.w, a.w, a.w), b);
        }
        // the other buffer is written next: its readers passed the barrier above
    }
    if (LANES > 1) {
        // the lanes' sums, in a tree through gs: LANES / 2 <= 2 rows of [32][CO], which is what gs holds
        float4* red = reinterpret_cast<float4*>(&gs[0][0][0]);  // [lane][element][CG]
#pragma unroll
        for (int half = LANES / 2; half > 0; half >>= 1) {
            __syncthreads();
            if (lane >= half && lane < 2 * half) {
#pragma unroll
                for (int k = 0; k < 4; ++k) red[((lane - half) * 32 + 4 * eg + k) * CG + cg] = acc[k];
            }
            __syncthreads();
            if (lane < half) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float4 v = red[(lane * 32 + 4 * eg + k) * CG + cg];
                    acc[k].x += v.x; acc[k].y += v.y; acc[k].z += v.z; acc[k].w += v.w;
                }
            }
        }
    }
    if (lane == 0 && co0 + 4 * cg < g.Co) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (4 * eg + k < window)
                *reinterpret_cast<float4*>(partial + ((int64_t)blockIdx.y * window + 4 * eg + k) * g.Co + co0 + 4 * cg) = acc[k];
    }
}

// ---- column sums ------------------------------------------------------------------------------------
// out[c] = sum over r < rows of in[r, c].  Block = blockDim.x column lanes (V columns each) x blockDim.y row
// lanes; a lane adds every blockDim.y-th row (UNROLL of them in flight), the row lanes meet in shared memory in
// lane order.  blockIdx.y cuts the rows into slices of `rows_per_slice`, one row of `out` per slice: the same
// kernel makes the partial sums and adds them up.  The order of the additions depends on the shape alone.
// Bound: memory.  One thread per column with a serial walk over 392 partial rows, and 4-byte loads with one in
// flight per thread before that, took 24 + 26 us for [100352, 128] (51 MB); now 16 + 5 us with a cold cache.
template <int V>
__global__ void __launch_bounds__(1024)
column_sums_kernel(const float* in, float* __restrict__ out, int64_t rows, int64_t C, int64_t rows_per_slice) {
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();
    constexpr int UNROLL = 8;
    __shared__ float red[1024 * V];
    const int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * V;
    const int64_t r_begin = (int64_t)blockIdx.y * rows_per_slice;
    const int64_t r_end = min(rows, r_begin + rows_per_slice);
    const int lanes = blockDim.y;
    float acc[V];
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = 0.f;
    if (c < C) {
        const float* p = in + c;
        // the last rows of a slice stay in the unrolled form (predicated): one by one, each would cost a memory latency
        for (int64_t r = r_begin + threadIdx.y; r < r_end; r += (int64_t)UNROLL * lanes) {
            float t[UNROLL][V];
#pragma unroll
            for (int u = 0; u < UNROLL; ++u) {
                const int64_t row = r + (int64_t)u * lanes;
#pragma unroll
                for (int v = 0; v < V; ++v) t[u][v] = 0.f;
                if (row < r_end) {
                    if (V == 4) *reinterpret_cast<float4*>(t[u]) = load_global(reinterpret_cast<const float4*>(p + row * C));
                    else t[u][0] = load_global(p + row * C);
                }
            }
#pragma unroll
            for (int u = 0; u < UNROLL; ++u)
#pragma unroll
                for (int v = 0; v < V; ++v) acc[v] += t[u][v];
        }
    }
    // [row lane][V][column lane]: neighbouring threads of a warp write neighbouring words
#pragma unroll
    for (int v = 0; v < V; ++v) red[(threadIdx.y * V + v) * blockDim.x + threadIdx.x] = acc[v];
    for (int half = lanes >> 1; half > 0; half >>= 1) {
        __syncthreads();
        if (threadIdx.y < half) {
#pragma unroll
            for (int v = 0; v < V; ++v)
                red[(threadIdx.y * V + v) * blockDim.x + threadIdx.x] += red[((threadIdx.y + half) * V + v) * blockDim.x + threadIdx.x];
        }
    }
    if (threadIdx.y == 0 && c < C) {
#pragma unroll
        for (int v = 0; v < V; ++v) out[(int64_t)blockIdx.y * C + c + v] = red[v * blockDim.x + threadIdx.x];
    }
}

// ---- depthwise, gradient with respect to the input ---------------------------------------------------
__global__ void __launch_bounds__(BP_THREADS)
depthwise_backprop_input_kernel(const float* dy, const float* f, float* __restrict__ dx, ConvGeom g,
                                int64_t total) {
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += stride) {
        const int c = (int)(e % g.C);
        int64_t p = e / g.C;
        const int ix = (int)(p % g.W);
        p /= g.W;
        const int iy = (int)(p % g.H);
        const int64_t n = p / g.H;
        float acc = 0.f;
        for (int ky = 0; ky < g.fh; ++ky) {
            const int oy = source_of(iy, g.pt, ky, g.dh, g.sh, g.Ho);
            if (oy < 0) continue;
            for (int kx = 0; kx < g.fw; ++kx) {
                const int ox = source_of(ix, g.pl, kx, g.dw, g.sw, g.Wo);
                if (ox < 0) continue;
                const float* gp = dy + ((n * g.Ho + oy) * (int64_t)g.Wo + ox) * g.Co + (int64_t)c * g.mult;
                const float* fp = f + ((int64_t)(ky * g.fw + kx) * g.C + c) * g.mult;
                // the first apart: with it in the loop the taps' loads come one after the other (5 x 5 over [8,56,56,64] 147 us
                // for 120, and 136 with read-only loads)
                acc = fmaf(load_global(gp), load_global(fp), acc);
                for (int q = 1; q < g.mult; ++q) acc = fmaf(load_global(gp + q), load_global(fp + q), acc);
            }
        }
        dx[e] = acc;
    }
}

// 3x3, stride 2, multiplier 1, C % 4 == 0.  In padded coordinates u = iy + pt, v = ix + pl the 2x2 group of samples
// (u, v) = (2q, 2r) .. (2q+1, 2r+1) is reached from the four output pixels (q-1..q, r-1..r) only:
//   (2q, 2r): four taps (corners), (2q, 2r+1) and (2q+1, 2r): two each, (2q+1, 2r+1): the centre tap.
// Thread = 4 channels x one column pair x a strip of ROWS row pairs: 2 (ROWS + 1) 16-byte loads, all issued before
// the first use, feed 4 ROWS 16-byte stores.  Bound by memory (dx is four times dy).
template <int ROWS>
__global__ void __launch_bounds__(BP_THREADS)
depthwise3x3_s2_backprop_input_kernel(const float* dy, const float* f, float* __restrict__ dx, ConvGeom g,
                                      int tc, int c4_tiles) {
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();
    const int C4 = g.C >> 2;
    const int c4 = (blockIdx.x % c4_tiles) * tc + (threadIdx.x % tc);
    const int r = (blockIdx.x / c4_tiles) * (BP_THREADS / tc) + threadIdx.x / tc;
    const int q0 = blockIdx.y * ROWS;
    const int ix = 2 * r - g.pl;
    if (c4 >= C4 || ix >= g.W) return;
    const int c = c4 * 4;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 w[9];
#pragma unroll
    for (int t = 0; t < 9; ++t) w[t] = load_global(reinterpret_cast<const float4*>(f + (int64_t)t * g.C + c));
    const int64_t n = blockIdx.z;
    const float* gy = dy + n * (int64_t)g.Ho * g.Wo * g.C + c;
    float4 a[ROWS + 1], b[ROWS + 1];  // columns r - 1 and r of rows q0 - 1 .. q0 + ROWS - 1
#pragma unroll
    for (int j = 0; j <= ROWS; ++j) {
        const int oy = q0 - 1 + j;
        const bool row = oy >= 0 && oy < g.Ho;
        const float* p = gy + ((int64_t)oy * g.Wo + r) * g.C;
        a[j] = row && r >= 1 && r - 1 < g.Wo ? load_global(reinterpret_cast<const float4*>(p - g.C)) : zero;
        b[j] = row && r < g.Wo ? load_global(reinterpret_cast<const float4*>(p)) : zero;
    }
    float* out = dx + n * (int64_t)g.H * g.W * g.C + c;
    // a filter that is not finite: only taps that meet an output pixel take part, where the zeros make NaNs of the others
    float4 nil = zero;
#pragma unroll
    for (int t = 0; t < 9; ++t) fma4_packed(nil, w[t], zero);
    const bool odd = !all_zero(nil);
    for (int e = 0; odd && e < 4 * ROWS; ++e) {
        const int iy = 2 * (q0 + (e >> 2)) - g.pt + ((e >> 1) & 1), jx = ix + (e & 1);
        if (iy < 0 || iy >= g.H || jx < 0 || jx >= g.W) continue;
        float4 v = zero;
        for (int t = 0; t < 9; ++t) {
            const int oy = source_of(iy, g.pt, t / 3, 1, 2, g.Ho), ox = source_of(jx, g.pl, t % 3, 1, 2, g.Wo);
            if (oy < 0 || ox < 0) continue;
            fma4_packed(v, load_global(reinterpret_cast<const float4*>(gy + ((int64_t)oy * g.Wo + ox) * g.C)),
                        load_global(reinterpret_cast<const float4*>(f + (int64_t)t * g.C + c)));
        }
        *reinterpret_cast<float4*>(out + ((int64_t)iy * g.W + jx) * g.C) = v;
    }
    if (odd) return;
#pragma unroll
    for (int j = 1; j <= ROWS; ++j) {
        const int iy = 2 * (q0 + j - 1) - g.pt;
        float4 v00 = zero, v01 = zero, v10 = zero, v11 = zero;
        fma4_packed(v00, b[j], w[0]); fma4_packed(v00, a[j], w[2]); fma4_packed(v00, b[j - 1], w[6]); fma4_packed(v00, a[j - 1], w[8]);
        fma4_packed(v01, b[j], w[1]); fma4_packed(v01, b[j - 1], w[7]);
        fma4_packed(v10, b[j], w[3]); fma4_packed(v10, a[j], w[5]);
        fma4_packed(v11, b[j], w[4]);
        float* o = out + ((int64_t)iy * g.W + ix) * g.C;
        if (iy >= 0 && iy < g.H) {
            if (ix >= 0) *reinterpret_cast<float4*>(o) = v00;
            if (ix + 1 < g.W) *reinterpret_cast<float4*>(o + g.C) = v01;
        }
        if (iy + 1 < g.H) {
            o += (int64_t)g.W * g.C;
            if (ix >= 0) *reinterpret_cast<float4*>(o) = v10;
            if (ix + 1 < g.W) *reinterpret_cast<float4*>(o + g.C) = v11;
        }
    }
}

// ---- depthwise, gradient with respect to the filter: partial sums ------------------------------------
// Block = 32 output channels (tx) x 8 pixel lanes (ty) for one tap (blockIdx.z) and one slice of the
// output pixels (blockIdx.y).
__global__ void __launch_bounds__(BP_THREADS)
depthwise_backprop_filter_partial_kernel(const float* x, const float* dy, float* __restrict__ partial,
                                         ConvGeom g, int64_t pixels, int64_t pixels_per_slice) {
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();
    __shared__ float red[8][32];
    const int oc = blockIdx.x * 32 + threadIdx.x;
    const int tap = blockIdx.z;
    const int ky = tap / g.fw, kx = tap - ky * g.fw;
    const int64_t p_begin = (int64_t)blockIdx.y * pixels_per_slice;
    const int64_t p_end = min(pixels, p_begin + pixels_per_slice);
    float acc = 0.f;
    if (oc < g.Co) {
        const int c = oc / g.mult;
        for (int64_t p = p_begin + threadIdx.y; p < p_end; p += 8) {
            const int ox = (int)(p % g.Wo);
            const int64_t r = p / g.Wo;
            const int oy = (int)(r % g.Ho);
            const int64_t n = r / g.Ho;
            const int iy = oy * g.sh - g.pt + ky * g.dh, ix = ox * g.sw - g.pl + kx * g.dw;
            if (iy >= 0 && iy < g.H && ix >= 0 && ix < g.W)
                acc = fmaf(load_global(x + ((n * g.H + iy) * (int64_t)g.W + ix) * g.C + c), load_global(dy + p * g.Co + oc), acc);
        }
    }
    red[threadIdx.y][threadIdx.x] = acc;
    __syncthreads();
    if (threadIdx.y == 0 && oc < g.Co) {
        float v = red[0][threadIdx.x];
#pragma unroll
        for (int k = 1; k < 8; ++k) v += red[k][threadIdx.x];
        partial[((int64_t)blockIdx.y * g.fh * g.fw + tap) * g.Co + oc] = v;
    }
}

// ---- epilogue ---------------------------------------------------------------------------------------
// dz = dy where the activation passed its input through (judged by the forward output y), +0 elsewhere.  Bound by
// memory (two operands in, one out); four values per thread and step: 26 -> 24 us for 3 x 51 MB.
__device__ __forceinline__ float act_grad(float y, float dy, int act) {
    const bool pass = act == TFJSB_ACT_NONE || (y > 0.f && (act == TFJSB_ACT_RELU || y < 6.f));
    return pass ? dy : 0.f;
}
// One group of four per thread and pass, and the next kernel starts as this one ends: two groups loaded ahead of the first store
// and an early start take 11.5 us for 7.8 million values, this 9.2 (before dependent launches 10.4), 17 million 31.2 and 29.5.
__global__ void __launch_bounds__(BP_THREADS)
act_backprop_kernel(const float* y, const float* dy, float* __restrict__ dz, int64_t n, int act) {
    ptx::pdl_wait();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t n4 = n >> 2;
    for (int64_t i = first; i < (n + 3) >> 2; i += stride) {
        if (i == n4) {  // the last three values at most, by a thread of their own where there are enough
            for (int64_t e = 4 * n4; e < n; ++e) dz[e] = act_grad(y[e], dy[e], act);
            break;
        }
        const float4 v = reinterpret_cast<const float4*>(y)[i], g = reinterpret_cast<const float4*>(dy)[i];
        reinterpret_cast<float4*>(dz)[i] =
            make_float4(act_grad(v.x, g.x, act), act_grad(v.y, g.y, act), act_grad(v.z, g.z, act), act_grad(v.w, g.w, act));
    }
}

int blocks_for(int64_t items, int sm_count) {
    int64_t b = (items + BP_THREADS - 1) / BP_THREADS;
    const int64_t cap = (int64_t)sm_count * 16;
    return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

}  // namespace

int backprop_slices(int64_t rows, int sm_count) {
    // enough slices for a few blocks per SM, at least 256 rows each
    int64_t s = rows / 256;
    if (s > 4 * (int64_t)sm_count) s = 4 * (int64_t)sm_count;
    return (int)(s < 1 ? 1 : s);
}

cudaError_t launch_conv2d_backprop_input(const float* dy, const float* f, float* dx, const ConvGeom& g, int sm_count,
                                         cudaStream_t s, int64_t* launches) {
    const int64_t total = g.N * g.H * g.W * g.C;
    ++*launches;
    return launch_k(conv2d_backprop_input_kernel, dim3(blocks_for(total, sm_count)), dim3(BP_THREADS), 0, s, dy, f, dx, g, total);
}

namespace {

int pow2_at_least(int64_t v, int limit) {
    int p = 1;
    while (p < v && p < limit) p <<= 1;
    return p;
}

// One launch of column_sums_kernel over `slices` slices of the rows.
cudaError_t launch_column_sums(const float* in, float* out, int64_t rows, int64_t C, int slices, cudaStream_t s, int64_t* launches) {
    const int64_t per = (rows + slices - 1) / slices;
    // four columns per thread where rows start on 16 bytes and there are columns enough to fill the SMs that way
    const bool vec = C % 4 == 0 && C * slices >= 8192;
    const int64_t cols = vec ? C / 4 : C;
    const int tx = pow2_at_least(cols, 32);
    // eight rows per lane and pass, up to 1024 threads; one warp at least
    int ty = pow2_at_least((per + 7) / 8, 1024 / tx);
    if (ty * tx < 32) ty = 32 / tx;
    const dim3 grid((unsigned)((cols + tx - 1) / tx), (unsigned)slices), block(tx, ty);
    ++*launches;
    return launch_k(vec ? column_sums_kernel<4> : column_sums_kernel<1>, grid, block, 0, s, in, out, rows, C, per);
}

}  // namespace

int sum_rows_slices(int64_t rows, int64_t C, int sm_count) {
    // One step while the 1024 threads of a block read their column strip in one pass.  Beyond that, slices of at least
    // 128 rows and two blocks of 1024 threads per SM, one wave.
    const int64_t strips = C % 4 == 0 ? (C + 127) / 128 : (C + 31) / 32;
    if (rows <= 1024) return 1;
    int64_t s = (2 * (int64_t)sm_count + strips - 1) / strips;
    if (s > rows / 128) s = rows / 128;
    return (int)(s < 1 ? 1 : (s > 65535 ? 65535 : s));
}

cudaError_t launch_sum_rows(const float* in, float* out, float* partial, int64_t rows, int64_t C, int slices, cudaStream_t s,
                            int64_t* launches) {
    if (slices <= 1) return launch_column_sums(in, out, rows, C, 1, s, launches);
    cudaError_t e = launch_column_sums(in, partial, rows, C, slices, s, launches);
    return e != cudaSuccess ? e : launch_column_sums(partial, out, slices, C, 1, s, launches);
}

bool conv2d_small_filter_supported(const ConvGeom& g) {
    return (int64_t)g.fh * g.fw * g.C <= 32 && g.Co % 4 == 0 && g.Co > 0 && (g.Co + 31) / 32 <= 0x7fffffff;
}

int conv2d_small_filter_slices(const ConvGeom& g, int sm_count) {
    // four blocks per SM over the channel tiles; a slice has at least 128 pixels
    const int tiles = (g.Co + (g.Co > 64 ? 127 : g.Co > 32 ? 63 : 31)) / (g.Co > 64 ? 128 : g.Co > 32 ? 64 : 32);
    int64_t s = (4 * (int64_t)sm_count + tiles - 1) / tiles;
    const int64_t most = g.N * g.Ho * g.Wo / 128;
    if (s > most) s = most;
    return (int)(s < 1 ? 1 : s > 65535 ? 65535 : s);
}

cudaError_t launch_conv2d_small_filter(const float* x, const float* dy, float* df, float* partial, int slices, const ConvGeom& g,
                                       cudaStream_t s, int64_t* launches) {
    const int64_t pixels = g.N * g.Ho * g.Wo, per = ((pixels + slices - 1) / slices + 31) / 32 * 32;
    const int window = g.fh * g.fw * g.C;
    float* out = slices > 1 ? partial : df;
    auto kernel = g.Co > 64 ? conv2d_backprop_small_filter_kernel<32> : g.Co > 32 ? conv2d_backprop_small_filter_kernel<16> : conv2d_backprop_small_filter_kernel<8>;
    const unsigned tiles = g.Co > 64 ? (unsigned)((g.Co + 127) / 128) : 1u;
    cudaError_t e = launch_k(kernel, dim3(tiles, (unsigned)slices), dim3(BP_THREADS), 0, s, x, dy, out, g, pixels, per, window);
    ++*launches;
    if (e != cudaSuccess || slices <= 1) return e;
    return launch_sum_rows(partial, df, nullptr, slices, (int64_t)window * g.Co, 1, s, launches);
}

cudaError_t launch_conv2d_backprop_filter(const float* x, const float* dy, float* df, float* partial, int slices,
                                          const ConvGeom& g, cudaStream_t s, int64_t* launches) {
    const int64_t pixels = g.N * g.Ho * g.Wo;
    const int64_t per = ((pixels + slices - 1) / slices + 31) / 32 * 32;
    const int ci_tiles = (g.C + 31) / 32, co_tiles = (g.Co + 31) / 32;
    const int64_t blocks = (int64_t)g.fh * g.fw * ci_tiles * co_tiles;
    if (blocks >= (1LL << 31)) return cudaErrorInvalidConfiguration;
    const int64_t elems = (int64_t)g.fh * g.fw * g.C * g.Co;
    cudaError_t e = launch_k(conv2d_backprop_filter_partial_kernel, dim3((unsigned)blocks, (unsigned)slices), dim3(32, 32), 0, s, x, dy, slices > 1 ? partial : df, g, pixels, per, ci_tiles, co_tiles);
    ++*launches;
    if (e != cudaSuccess || slices <= 1) return e;
    return launch_sum_rows(partial, df, nullptr, slices, elems, 1, s, launches);
}

bool depthwise_backprop_is_forward(const ConvGeom& g) {
    return g.fh == 3 && g.fw == 3 && g.mult == 1 && g.sh == 1 && g.sw == 1 && g.C % 4 == 0 && g.dh == g.dw &&
           (g.dh == 1 || g.dh == 2 || g.dh == 4) && g.N <= 65535 && (g.H + 3) / 4 <= 65535;
}

ConvGeom depthwise_backprop_geometry(const ConvGeom& g) {
    ConvGeom t = g;
    t.H = g.Ho; t.W = g.Wo; t.Ho = g.H; t.Wo = g.W;
    t.pt = (g.fh - 1) * g.dh - g.pt;  // dx[i] = sum over k of dy[i + pt - k d] f[k], k from last to first
    t.pl = (g.fw - 1) * g.dw - g.pl;
    t.reversed = 1;
    return t;
}

cudaError_t launch_depthwise_backprop_input(const float* dy, const float* f, float* dx, const ConvGeom& g, int sm_count,
                                            cudaStream_t s, int64_t* launches) {
    if (g.fh == 3 && g.fw == 3 && g.mult == 1 && g.sh == 2 && g.sw == 2 && g.dh == 1 && g.dw == 1 && g.C % 4 == 0 && g.N <= 65535) {
        constexpr int ROWS = 4;
        const int tc = pow2_at_least(g.C / 4, 32);
        const int c4_tiles = (g.C / 4 + tc - 1) / tc;
        const int cols = BP_THREADS / tc;
        const int64_t gx = (int64_t)c4_tiles * (((g.W + g.pl + 1) / 2 + cols - 1) / cols);
        const int gy = ((g.H + g.pt + 1) / 2 + ROWS - 1) / ROWS;
        if (gx <= 2147483647LL && gy <= 65535) {
            ++*launches;
            return launch_k(depthwise3x3_s2_backprop_input_kernel<ROWS>, dim3((unsigned)gx, (unsigned)gy, (unsigned)g.N), dim3(BP_THREADS), 0, s, dy, f, dx, g, tc, c4_tiles);
        }
    }
    const int64_t total = g.N * g.H * g.W * g.C;
    ++*launches;
    return launch_k(depthwise_backprop_input_kernel, dim3(blocks_for(total, sm_count)), dim3(BP_THREADS), 0, s, dy, f, dx, g, total);
}

cudaError_t launch_depthwise_backprop_filter(const float* x, const float* dy, float* df, float* partial, int slices,
                                             const ConvGeom& g, cudaStream_t s, int64_t* launches) {
    const int64_t pixels = g.N * g.Ho * g.Wo;
    const int64_t per = (pixels + slices - 1) / slices;
    const int taps = g.fh * g.fw;
    if (taps > 65535 || slices > 65535) return cudaErrorInvalidConfiguration;
    cudaError_t e = launch_k(depthwise_backprop_filter_partial_kernel, dim3((unsigned)((g.Co + 31) / 32), (unsigned)slices, (unsigned)taps), dim3(32, 8), 0, s, x, dy, slices > 1 ? partial : df, g, pixels, per);
    ++*launches;
    if (e != cudaSuccess || slices <= 1) return e;
    return launch_sum_rows(partial, df, nullptr, slices, (int64_t)taps * g.Co, 1, s, launches);
}

cudaError_t launch_act_backprop(const float* y, const float* dy, float* dz, int64_t n, int act, int sm_count, cudaStream_t s,
                                int64_t* launches) {
    ++*launches;
    return launch_k(act_backprop_kernel, dim3(blocks_for((n + 3) / 4, sm_count)), dim3(BP_THREADS), 0, s, y, dy, dz, n, act);
}

}  // namespace tfjsb
