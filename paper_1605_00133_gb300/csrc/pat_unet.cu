// pat_unet.cu - layers of the learned warm start (a 3D U-Net mapping A^T C^T f to a starting image
// for the TV-Bregman solver): the C ABI of the 3x3x3 convolutions, their data and weight gradients
// (on the tcgen05 tensor cores, pat_unet_tc.cu), and the elementwise layers around them (pooling,
// upsampling, ReLU backward, the input and output layers, the loss and Adam).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <string>

#include "../../include/pat_unet.h"
#include "pat_fft.cuh"
#include "pat_internal.h"

namespace pat {
cudaError_t conv3_tc(const void* x, int ldx, int cin, const void* w, int cout, void* y, int ldy, int D, int H,
                     int W, int relu, const void* mask, int ldm, cudaStream_t st);
cudaError_t unet_take_status(int* word, cudaStream_t st);
void unet_set_copy_fault(int stop_after, int polls);
int64_t wgrad_tc_scratch(int cin, int cout, int D, int H, int W);
cudaError_t wgrad_tc(const void* x, int ldx, int cin, const void* dy, int ldy, int cout, int D, int H, int W,
                     float* partial, float* dw, cudaStream_t st);
}  // namespace pat

namespace {

typedef __nv_bfloat16 bf16;
using pat::launch_pdl;
using pat::pdl_trigger;
using pat::pdl_wait;


__global__ void cast_weights_kernel(const float* __restrict__ w32, int cin, int cout, bf16* __restrict__ wb,
                                    bf16* __restrict__ wt) {
    const int n = 27 * cin * cout;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int t = i / (cout * cin), r = i - t * cout * cin, co = r / cin, ci = r - co * cin;
        const bf16 b = __float2bfloat16(w32[i]);
        wb[i] = b;
        wt[((size_t)(26 - t) * cin + ci) * cout + co] = b;
    }
}

// ---- elementwise layers.  Each has a vector form, eight channels (16 bytes) per thread with 32-bit indices,
// taken when the channel count and strides are multiples of 8 and the pointers 16-byte aligned (every layer of
// the network), and a scalar form for anything else.  One thread per channel with a 64-bit division and 2-byte
// accesses, they ran at a tenth of the memory bandwidth (up 132 us, ReLU backward 43, pool backward 79 at
// 64x128x128 voxels); the vector forms are bound by memory.  MASK: the gradient is also taken through the
// ReLU whose output is y (zero where y is not positive), which saves a pass of its own.  The vector forms are
// launched with programmatic stream serialisation, as the convolutions are (pat_unet_tc.cu).

struct V8 {
    uint4 u;
};
// (through L2: written by the kernel before, which may still run when this one starts)
__device__ __forceinline__ V8 ld8(const bf16* p) { return V8{__ldcg(reinterpret_cast<const uint4*>(p))}; }
__device__ __forceinline__ void st8(bf16* p, V8 v) { *reinterpret_cast<uint4*>(p) = v.u; }
__device__ __forceinline__ void unpack8(V8 v, float* f) {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v.u);
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const float2 t = __bfloat1622float2(h[i]);
        f[2 * i] = t.x;
        f[2 * i + 1] = t.y;
    }
}
__device__ __forceinline__ V8 pack8(const float* f) {
    V8 v;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&v.u);
#pragma unroll
    for (int i = 0; i < 4; i++) h[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
    return v;
}
// f, zero where the activation y is not positive
__device__ __forceinline__ void mask8(float* f, V8 y) {
    float a[8];
    unpack8(y, a);
#pragma unroll
    for (int i = 0; i < 8; i++) f[i] = a[i] > 0.f ? f[i] : 0.f;
}
// voxel and channel octet of element i of n = voxels * c8
struct Vox {
    unsigned v, c;
};
__device__ __forceinline__ Vox vox_of(unsigned i, unsigned c8) {
    const unsigned v = i / c8;
    return Vox{v, 8 * (i - v * c8)};
}
// the eight children of voxel p of an H x W (x D) volume in the twice as large one
__device__ __forceinline__ unsigned child0(unsigned p, unsigned H, unsigned W) {
    const unsigned z = p / (H * W), r = p - z * (H * W), y = r / W, x = r - y * W;
    return ((2 * z) * (2 * H) + 2 * y) * (2 * W) + 2 * x;
}
__device__ __forceinline__ unsigned child(unsigned c0, int k, unsigned H2, unsigned W2) {
    return c0 + ((k >> 2) * H2 + ((k >> 1) & 1)) * W2 + (k & 1);
}

__global__ void __launch_bounds__(256) relu_bwd8_kernel(bf16* __restrict__ g, int ldg, const bf16* __restrict__ y, int ldy,
                                                        unsigned c8, unsigned n) {
    for (unsigned i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) {
        const Vox e = vox_of(i, c8);
        bf16* p = g + (size_t)e.v * ldg + e.c;
        float f[8];
        unpack8(ld8(p), f);
        mask8(f, ld8(y + (size_t)e.v * ldy + e.c));
        st8(p, pack8(f));
    }
}
__global__ void relu_bwd_kernel(bf16* __restrict__ g, int ldg, const bf16* __restrict__ y, int ldy, int C, long long V) {
    const long long n = V * C;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const long long v = i / C;
        const int c = (int)(i - v * C);
        if (!(__bfloat162float(y[v * ldy + c]) > 0.f)) g[v * ldg + c] = __float2bfloat16(0.f);
    }
}

// D, H, W: the pooled (small) volume
__global__ void __launch_bounds__(256) pool8_kernel(const bf16* __restrict__ x, int ldx, unsigned c8, unsigned H, unsigned W,
                                                    bf16* __restrict__ y, int ldy, unsigned n) {
    pdl_wait();
    pdl_trigger();
    for (unsigned i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) {
        const Vox e = vox_of(i, c8);
        const unsigned c0 = child0(e.v, H, W);
        V8 in[8];
#pragma unroll
        for (int k = 0; k < 8; k++) in[k] = ld8(x + (size_t)child(c0, k, 2 * H, 2 * W) * ldx + e.c);
        float s[8] = {};
#pragma unroll
        for (int k = 0; k < 8; k++) {
            float f[8];
            unpack8(in[k], f);
#pragma unroll
            for (int j = 0; j < 8; j++) s[j] += f[j];
        }
#pragma unroll
        for (int j = 0; j < 8; j++) s[j] *= 0.125f;
        st8(y + (size_t)e.v * ldy + e.c, pack8(s));
    }
}
__global__ void pool_kernel(const bf16* __restrict__ x, int ldx, int C, int D, int H, int W, bf16* __restrict__ y, int ldy) {
    const int D2 = D / 2, H2 = H / 2, W2 = W / 2;
    const long long n = (long long)D2 * H2 * W2 * C;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % C);
        const long long p = i / C;
        const int z = (int)(p / (H2 * W2)), r = (int)(p - (long long)z * H2 * W2), yy = r / W2, xx = r - yy * W2;
        float s = 0.f;
        for (int k = 0; k < 8; k++) {
            const int cz = 2 * z + (k >> 2), cy = 2 * yy + ((k >> 1) & 1), cx = 2 * xx + (k & 1);
            s += __bfloat162float(x[((size_t)(cz * H + cy) * W + cx) * ldx + c]);
        }
        y[p * ldy + c] = __float2bfloat16(0.125f * s);
    }
}

// D, H, W: the pooled volume; mask: activation of the large one (NULL: none)
__global__ void __launch_bounds__(256) pool_bwd_add8_kernel(const bf16* __restrict__ dy, int ldd, unsigned c8, unsigned H,
                                                            unsigned W, bf16* __restrict__ dx, int ldx,
                                                            const bf16* __restrict__ mask, int ldm, unsigned n) {
    pdl_wait();
    pdl_trigger();
    for (unsigned i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) {
        const Vox e = vox_of(i, c8);
        const unsigned c0 = child0(e.v, H, W);
        float g[8];
        unpack8(ld8(dy + (size_t)e.v * ldd + e.c), g);
#pragma unroll
        for (int j = 0; j < 8; j++) g[j] *= 0.125f;
        V8 in[8], mk[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const size_t v = child(c0, k, 2 * H, 2 * W);
            in[k] = ld8(dx + v * ldx + e.c);
            if (mask) mk[k] = ld8(mask + v * ldm + e.c);
        }
#pragma unroll
        for (int k = 0; k < 8; k++) {
            float f[8];
            unpack8(in[k], f);
#pragma unroll
            for (int j = 0; j < 8; j++) f[j] += g[j];
            if (mask) mask8(f, mk[k]);
            st8(dx + (size_t)child(c0, k, 2 * H, 2 * W) * ldx + e.c, pack8(f));
        }
    }
}
__global__ void pool_bwd_add_kernel(const bf16* __restrict__ dy, int ldd, int C, int D, int H, int W, bf16* __restrict__ dx, int ldx) {
    const long long n = (long long)D * H * W * C;
    const int H2 = H / 2, W2 = W / 2;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % C);
        const long long v = i / C;
        const int z = (int)(v / (H * W)), r = (int)(v - (long long)z * H * W), yy = r / W, xx = r - yy * W;
        const long long pp = ((long long)(z / 2) * H2 + yy / 2) * W2 + xx / 2;
        const float g = 0.125f * __bfloat162float(dy[pp * ldd + c]);
        dx[v * ldx + c] = __float2bfloat16(__bfloat162float(dx[v * ldx + c]) + g);
    }
}

// D, H, W: the small volume
__global__ void __launch_bounds__(256) up8_kernel(const bf16* __restrict__ x, int ldx, unsigned c8, unsigned H, unsigned W,
                                                  bf16* __restrict__ y, int ldy, unsigned n) {
    pdl_wait();
    pdl_trigger();
    for (unsigned i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) {
        const Vox e = vox_of(i, c8);
        const unsigned c0 = child0(e.v, H, W);
        const V8 v = ld8(x + (size_t)e.v * ldx + e.c);
#pragma unroll
        for (int k = 0; k < 8; k++) st8(y + (size_t)child(c0, k, 2 * H, 2 * W) * ldy + e.c, v);
    }
}
__global__ void up_kernel(const bf16* __restrict__ x, int ldx, int C, int D, int H, int W, bf16* __restrict__ y, int ldy) {
    const int D2 = 2 * D, H2 = 2 * H, W2 = 2 * W;
    const long long n = (long long)D2 * H2 * W2 * C;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % C);
        const long long v = i / C;
        const int z = (int)(v / (H2 * W2)), r = (int)(v - (long long)z * H2 * W2), yy = r / W2, xx = r - yy * W2;
        y[v * ldy + c] = x[((size_t)((z / 2) * H + yy / 2) * W + xx / 2) * ldx + c];
    }
}

// D, H, W: the small volume; mask: its activation (NULL: none)
__global__ void __launch_bounds__(256) up_bwd8_kernel(const bf16* __restrict__ dy, int ldd, unsigned c8, unsigned H,
                                                      unsigned W, bf16* __restrict__ dx, int ldx,
                                                      const bf16* __restrict__ mask, int ldm, unsigned n) {
    pdl_wait();
    pdl_trigger();
    for (unsigned i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) {
        const Vox e = vox_of(i, c8);
        const unsigned c0 = child0(e.v, H, W);
        V8 in[8];
#pragma unroll
        for (int k = 0; k < 8; k++) in[k] = ld8(dy + (size_t)child(c0, k, 2 * H, 2 * W) * ldd + e.c);
        float s[8] = {};
#pragma unroll
        for (int k = 0; k < 8; k++) {
            float f[8];
            unpack8(in[k], f);
#pragma unroll
            for (int j = 0; j < 8; j++) s[j] += f[j];
        }
        if (mask) mask8(s, ld8(mask + (size_t)e.v * ldm + e.c));
        st8(dx + (size_t)e.v * ldx + e.c, pack8(s));
    }
}
__global__ void up_bwd_kernel(const bf16* __restrict__ dy, int ldd, int C, int D, int H, int W, bf16* __restrict__ dx, int ldx) {
    const long long n = (long long)D * H * W * C;
    const int H2 = 2 * H, W2 = 2 * W;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % C);
        const long long p = i / C;
        const int z = (int)(p / (H * W)), r = (int)(p - (long long)z * H * W), yy = r / W, xx = r - yy * W;
        float s = 0.f;
        for (int k = 0; k < 8; k++) {
            const int cz = 2 * z + (k >> 2), cy = 2 * yy + ((k >> 1) & 1), cx = 2 * xx + (k & 1);
            s += __bfloat162float(dy[((size_t)(cz * H2 + cy) * W2 + cx) * ldd + c]);
        }
        dx[p * ldx + c] = __float2bfloat16(s);
    }
}

// two 16-byte halves of a voxel's 16 channels per thread pair: consecutive threads write consecutive bytes
__global__ void __launch_bounds__(256) input8_kernel(const float* __restrict__ xin, float s, long long n, bf16* __restrict__ x16) {
    pdl_wait();
    pdl_trigger();
    for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += gridDim.x * 256LL) {
        float f[8] = {};
        if (!(i & 1)) f[0] = s * __ldcg(xin + (i >> 1));
        st8(x16 + 8 * i, pack8(f));
    }
}
__global__ void input_kernel(const float* __restrict__ xin, float s, long long V, bf16* __restrict__ x16) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < V * 16; i += (long long)gridDim.x * blockDim.x) {
        const long long v = i >> 4;
        x16[i] = __float2bfloat16((i & 15) == 0 ? s * xin[v] : 0.f);
    }
}

__global__ void __launch_bounds__(256) head8_kernel(const bf16* __restrict__ h, const float* __restrict__ head, long long V,
                                                    float* __restrict__ out) {
    pdl_wait();
    pdl_trigger();
    float w[17];
#pragma unroll
    for (int c = 0; c < 17; c++) w[c] = __ldca(head + c);
    for (long long v = blockIdx.x * 256LL + threadIdx.x; v < V; v += gridDim.x * 256LL) {
        float f[16], s = w[16];
        unpack8(ld8(h + 16 * v), f);
        unpack8(ld8(h + 16 * v + 8), f + 8);
#pragma unroll
        for (int c = 0; c < 16; c++) s = fmaf(w[c], f[c], s);
        out[v] = s;
    }
}
__global__ void head_kernel(const bf16* __restrict__ h, const float* __restrict__ head, long long V, float* __restrict__ out) {
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < V; v += (long long)gridDim.x * blockDim.x) {
        float s = head[16];
#pragma unroll
        for (int c = 0; c < 16; c++) s = fmaf(head[c], __bfloat162float(h[v * 16 + c]), s);
        out[v] = s;
    }
}

constexpr int kHeadBlocks = 304;  // two per SM
// fixed-order tree over the block's threads of the 18 sums in red; one row of partial per block
__device__ __forceinline__ void head_reduce(double (*red)[18], double* __restrict__ partial) {
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int k = 0; k < 18; k++) red[threadIdx.x][k] += red[threadIdx.x + w][k];
        __syncthreads();
    }
    if (threadIdx.x < 18) partial[(size_t)blockIdx.x * 18 + threadIdx.x] = red[0][threadIdx.x];
}

// The two BF16 of a word as doubles times 2^-896: their bits moved to a double's places without the change of
// exponent bias, exact for every finite value (a BF16 subnormal becomes a double's).
__device__ __forceinline__ double bf16_lo_scaled(uint32_t w) {
    return __hiloint2double((int)(((w & 0x7fffu) << 13) | ((w << 16) & 0x80000000u)), 0);
}
__device__ __forceinline__ double bf16_hi_scaled(uint32_t w) {
    return __hiloint2double((int)(((w & 0x7fff0000u) >> 3) | (w & 0x80000000u)), 0);
}

// per block: 16 channel sums of g h, the sum of g, the sum of squared errors, in FP64: they cover the range and the
// precision of a long sum of FP32 products, whatever the data.  mask: dh is also taken through the ReLU whose output h
// is.  What bounds it: the FP64 units, about 2 operations per cycle and SM here.  16 multiply-adds a voxel are needed,
// 16 conversions more would be its work too (107 us with them, in the scalar form), so a channel's bits are placed in a
// double by integer operations, 2^-896 too small, and the factor g carries the 2^896: the products, and so the sums,
// are those of head_bwd_kernel bit for bit.  A voxel with an infinite or NaN channel is converted.  1 M voxels, with
// the sum over the blocks: 63 us.  (Sums as pairs of floats take 38, but have FP32's range and 47 bits.)
__global__ void __launch_bounds__(256) head_bwd8_kernel(const bf16* __restrict__ h, const float* __restrict__ head,
                                                        const float* __restrict__ out, const float* __restrict__ target,
                                                        long long V, bf16* __restrict__ dh, int mask,
                                                        double* __restrict__ partial) {
    pdl_wait();
    pdl_trigger();
    __shared__ double red[256][18];
    double acc[18];
#pragma unroll
    for (int k = 0; k < 18; k++) acc[k] = 0.0;
    float w[16];
#pragma unroll
    for (int c = 0; c < 16; c++) w[c] = __ldca(head + c);
    const double gs = 2.0 / (double)V;
    for (long long v = blockIdx.x * 256LL + threadIdx.x; v < V; v += gridDim.x * 256LL) {
        const V8 h8[2] = {ld8(h + 16 * v), ld8(h + 16 * v + 8)};
        float f[16];
        unpack8(h8[0], f);
        unpack8(h8[1], f + 8);
        const double e = (double)__ldcg(out + v) - (double)__ldcg(target + v);
        const float g = (float)(gs * e);
        const double gd = (double)g;
        float d[16], odd = 0.f;
#pragma unroll
        for (int c = 0; c < 16; c++) {
            odd = fmaf(f[c], 0.f, odd);  // NaN if any channel is not finite
            d[c] = (!mask || f[c] > 0.f) ? g * w[c] : 0.f;
        }
        st8(dh + 16 * v, pack8(d));
        st8(dh + 16 * v + 8, pack8(d + 8));
        if (odd == 0.f) {
            const double gb = gd * 0x1p896;  // finite where g is
            const uint32_t* u = reinterpret_cast<const uint32_t*>(h8);
#pragma unroll
            for (int c = 0; c < 16; c += 2) {
                acc[c] = fma(gb, bf16_lo_scaled(u[c / 2]), acc[c]);
                acc[c + 1] = fma(gb, bf16_hi_scaled(u[c / 2]), acc[c + 1]);
            }
        } else {
#pragma unroll
            for (int c = 0; c < 16; c++) acc[c] = fma(gd, (double)f[c], acc[c]);
        }
        acc[16] += gd;
        acc[17] = fma(e, e, acc[17]);
    }
#pragma unroll
    for (int k = 0; k < 18; k++) red[threadIdx.x][k] = acc[k];
    head_reduce(red, partial);
}
__global__ void __launch_bounds__(256) head_bwd_kernel(const bf16* __restrict__ h, const float* __restrict__ head,
                                                       const float* __restrict__ out, const float* __restrict__ target,
                                                       long long V, bf16* __restrict__ dh, int mask,
                                                       double* __restrict__ partial) {
    __shared__ double red[256][18];
    double acc[18];
    for (int k = 0; k < 18; k++) acc[k] = 0.0;
    const double gs = 2.0 / (double)V;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < V; v += (long long)gridDim.x * blockDim.x) {
        const double e = (double)out[v] - (double)target[v];
        const float g = (float)(gs * e);
#pragma unroll
        for (int c = 0; c < 16; c++) {
            const float hv = __bfloat162float(h[v * 16 + c]);
            acc[c] = fma((double)g, (double)hv, acc[c]);
            dh[v * 16 + c] = __float2bfloat16((!mask || hv > 0.f) ? g * head[c] : 0.f);
        }
        acc[16] += (double)g;
        acc[17] = fma(e, e, acc[17]);
    }
    for (int k = 0; k < 18; k++) red[threadIdx.x][k] = acc[k];
    head_reduce(red, partial);
}

// one warp per sum: strided partial sums and a fixed-order tree
__global__ void __launch_bounds__(576) head_bwd_final_kernel(const double* __restrict__ partial, int nb, long long V,
                                                             float* __restrict__ ghead, double* __restrict__ loss) {
    pdl_wait();
    pdl_trigger();
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s = 0.0;
    for (int b = lane; b < nb; b += 32) s += __ldcg(partial + (size_t)b * 18 + k);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane) return;
    if (k < 17) ghead[k] = (float)s;
    else loss[0] = s / (double)V;
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                            long long n, float lr, float b1, float b2, float eps, float c1, float c2) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

unsigned grid_for(long long n, int nt = 256) {
    const long long b = (n + nt - 1) / nt;
    return (unsigned)std::max(1LL, std::min(b, 152LL * 16));
}

bool al16(const void* p) { return ((uintptr_t)p & 15) == 0; }
// whether the vector forms serve a layer: whole octets of channels, 16-byte aligned rows (an unused operand
// passes the alignment of a used one), and element indices that fit 32 bits
bool vec8(int C, int lda, int ldb, int ldc, const void* a, const void* b, const void* c, long long voxels) {
    return C % 8 == 0 && lda % 8 == 0 && ldb % 8 == 0 && ldc % 8 == 0 && al16(a) && al16(b) && al16(c) &&
           voxels * (C / 8) < (1LL << 31) && voxels < (1LL << 31);
}

pat_status bad(const char* msg) { return pat::set_error(PAT_ERR_INVALID_ARG, msg); }

pat_status launched(const char* where) {
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PAT_OK : pat::set_cuda_error(e, where);
}

}  // namespace

extern "C" {

static pat_status conv3(const char* who, const void* x, int32_t ldx, int32_t cin, const void* w, int32_t cout, void* y,
                        int32_t ldy, int32_t D, int32_t H, int32_t W, int32_t relu, const void* mask, int32_t ldm,
                        void* stream) {
    const auto fail = [&](const char* msg) { return bad((std::string(who) + msg).c_str()); };
    if (!x || !w || !y) return fail(": NULL pointer");
    if (cin < 16 || cin > 512 || cin % 16 || ldx < cin || ldx % 16 || ldy < cout || ldy % 16)
        return fail(": channel counts and strides must be multiples of 16 (cin <= 512)");
    if (cout < 16 || cout > 1024 || cout % 16) return fail(": cout must be a multiple of 16 (<= 1024)");
    if (D < 1 || H < 1 || W < 1 || (int64_t)D * H * W > (1LL << 30)) return fail(": bad volume");
    if (!al16(x) || !al16(w) || !al16(y)) return fail(": pointers must be 16-byte aligned");
    const cudaError_t e = pat::conv3_tc(x, ldx, cin, w, cout, y, ldy, D, H, W, relu, mask, ldm, (cudaStream_t)stream);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return pat::set_cuda_error(e, who);
    }
    return PAT_OK;
}

pat_status pat_unet_conv3(const void* x, int32_t ldx, int32_t cin, const void* w, int32_t cout, void* y,
                          int32_t ldy, int32_t D, int32_t H, int32_t W, int32_t relu, void* stream) {
    return conv3("pat_unet_conv3", x, ldx, cin, w, cout, y, ldy, D, H, W, relu, nullptr, 0, stream);
}

pat_status pat_unet_conv3_masked(const void* x, int32_t ldx, int32_t cin, const void* w, int32_t cout, void* y,
                                 int32_t ldy, int32_t D, int32_t H, int32_t W, const void* act, int32_t lda,
                                 void* stream) {
    if (!act || !al16(act) || lda < cout || lda % 16)
        return bad("pat_unet_conv3_masked: the activation must be 16-byte aligned, its stride a multiple of 16");
    return conv3("pat_unet_conv3_masked", x, ldx, cin, w, cout, y, ldy, D, H, W, 0, act, lda, stream);
}

pat_status pat_unet_debug_copy_fault(int32_t stop_after_stage, int32_t polls) {
    if (stop_after_stage < -1 || polls < 0) return bad("pat_unet_debug_copy_fault: stop_after_stage >= -1, polls >= 0");
    pat::unet_set_copy_fault(stop_after_stage, polls);
    pat::set_error(PAT_OK, "");
    return PAT_OK;
}

pat_status pat_unet_device_status(void* stream) {
    int word = 0;
    const cudaError_t e = pat::unet_take_status(&word, (cudaStream_t)stream);
    if (e != cudaSuccess) return pat::set_cuda_error(e, "pat_unet_device_status");
    if (word) return pat::set_error(PAT_ERR_TIMEOUT, "pat_unet_device_status: a tensor-core convolution gave up "
                                                     "waiting for its copies or its matrix multiplies");
    pat::set_error(PAT_OK, "");
    return PAT_OK;
}

int64_t pat_unet_wgrad_scratch(int32_t cin, int32_t cout, int32_t D, int32_t H, int32_t W) {
    if (cin < 16 || cout < 16 || D < 1 || H < 1 || W < 1) return 0;
    return pat::wgrad_tc_scratch(cin, cout, D, H, W);
}

pat_status pat_unet_conv3_wgrad(const void* x, int32_t ldx, int32_t cin, const void* dy, int32_t ldy, int32_t cout,
                                int32_t D, int32_t H, int32_t W, float* partial, float* dw, void* stream) {
    if (!x || !dy || !partial || !dw) return bad("pat_unet_conv3_wgrad: NULL pointer");
    if (cin < 16 || cin > 256 || cin % 16 || ldx < cin || ldx % 16 || ldy < cout || ldy % 16 || cout < 16 ||
        cout > 128 || cout % 16)
        return bad("pat_unet_conv3_wgrad: cin in 16..256 and cout in 16..128, multiples of 16; strides too");
    if (!al16(x) || !al16(dy) || !al16(partial)) return bad("pat_unet_conv3_wgrad: pointers must be 16-byte aligned");
    if (D < 1 || H < 1 || W < 1 || (int64_t)D * H * W > (1LL << 30)) return bad("pat_unet_conv3_wgrad: bad volume");
    const cudaError_t e = pat::wgrad_tc(x, ldx, cin, dy, ldy, cout, D, H, W, partial, dw, (cudaStream_t)stream);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return pat::set_cuda_error(e, "pat_unet_conv3_wgrad");
    }
    return PAT_OK;
}

pat_status pat_unet_cast_weights(const float* w32, int32_t cin, int32_t cout, void* wb, void* wt, void* stream) {
    if (!w32 || !wb || !wt || cin < 1 || cout < 1) return bad("pat_unet_cast_weights: bad argument");
    const long long n = 27LL * cin * cout;
    cast_weights_kernel<<<grid_for(n), 256, 0, (cudaStream_t)stream>>>(w32, cin, cout, (bf16*)wb, (bf16*)wt);
    return launched("pat_unet_cast_weights");
}

pat_status pat_unet_relu_bwd(void* g, int32_t ldg, const void* y, int32_t ldy, int32_t C, int64_t V, void* stream) {
    if (!g || !y || C < 1 || ldg < C || ldy < C || V < 0) return bad("pat_unet_relu_bwd: bad argument");
    if (vec8(C, ldg, ldy, 8, g, y, y, V))
        relu_bwd8_kernel<<<grid_for(V * C / 8), 256, 0, (cudaStream_t)stream>>>((bf16*)g, ldg, (const bf16*)y, ldy, C / 8,
                                                                               (unsigned)(V * C / 8));
    else
        relu_bwd_kernel<<<grid_for(V * C), 256, 0, (cudaStream_t)stream>>>((bf16*)g, ldg, (const bf16*)y, ldy, C, V);
    return launched("pat_unet_relu_bwd");
}

pat_status pat_unet_pool(const void* x, int32_t ldx, int32_t C, int32_t D, int32_t H, int32_t W, void* y, int32_t ldy,
                         void* stream) {
    if (!x || !y || C < 1 || ldx < C || ldy < C || D < 2 || H < 2 || W < 2 || (D | H | W) & 1)
        return bad("pat_unet_pool: bad argument (even dims >= 2)");
    const long long P = (long long)D * H * W / 8;
    if (vec8(C, ldx, ldy, 8, x, y, y, 8 * P))
        launch_pdl(pool8_kernel, grid_for(P * C / 8), 256, 0, (cudaStream_t)stream, (const bf16*)x, ldx, C / 8, H / 2, W / 2,
                   (bf16*)y, ldy, (unsigned)(P * C / 8));
    else
        pool_kernel<<<grid_for(P * C), 256, 0, (cudaStream_t)stream>>>((const bf16*)x, ldx, C, D, H, W, (bf16*)y, ldy);
    return launched("pat_unet_pool");
}

pat_status pat_unet_pool_bwd_add(const void* dy, int32_t ldd, int32_t C, int32_t D, int32_t H, int32_t W, void* dx,
                                 int32_t ldx, void* stream) {
    if (!dy || !dx || C < 1 || ldx < C || ldd < C || D < 2 || H < 2 || W < 2 || (D | H | W) & 1)
        return bad("pat_unet_pool_bwd_add: bad argument (even dims >= 2)");
    const long long P = (long long)D * H * W / 8;
    if (vec8(C, ldx, ldd, 8, dx, dy, dy, 8 * P))
        launch_pdl(pool_bwd_add8_kernel, grid_for(P * C / 8), 256, 0, (cudaStream_t)stream,
                   (const bf16*)dy, ldd, C / 8, H / 2, W / 2, (bf16*)dx, ldx, nullptr, 0, (unsigned)(P * C / 8));
    else
        pool_bwd_add_kernel<<<grid_for(8 * P * C), 256, 0, (cudaStream_t)stream>>>((const bf16*)dy, ldd, C, D, H, W,
                                                                                  (bf16*)dx, ldx);
    return launched("pat_unet_pool_bwd_add");
}

pat_status pat_unet_pool_bwd_add_masked(const void* dy, int32_t ldd, int32_t C, int32_t D, int32_t H, int32_t W, void* dx,
                                        int32_t ldx, const void* act, int32_t lda, void* stream) {
    if (!dy || !dx || !act || C < 1 || ldx < C || ldd < C || lda < C || D < 2 || H < 2 || W < 2 || (D | H | W) & 1)
        return bad("pat_unet_pool_bwd_add_masked: bad argument (even dims >= 2)");
    const long long P = (long long)D * H * W / 8;
    if (vec8(C, ldx, ldd, lda, dx, dy, act, 8 * P)) {
        launch_pdl(pool_bwd_add8_kernel, grid_for(P * C / 8), 256, 0, (cudaStream_t)stream,
                   (const bf16*)dy, ldd, C / 8, H / 2, W / 2, (bf16*)dx, ldx, (const bf16*)act, lda, (unsigned)(P * C / 8));
        return launched("pat_unet_pool_bwd_add_masked");
    }
    const pat_status s = pat_unet_pool_bwd_add(dy, ldd, C, D, H, W, dx, ldx, stream);
    return s != PAT_OK ? s : pat_unet_relu_bwd(dx, ldx, act, lda, C, 8 * P, stream);
}

pat_status pat_unet_up(const void* x, int32_t ldx, int32_t C, int32_t D, int32_t H, int32_t W, void* y, int32_t ldy,
                       void* stream) {
    if (!x || !y || C < 1 || ldx < C || ldy < C || D < 1 || H < 1 || W < 1) return bad("pat_unet_up: bad argument");
    const long long P = (long long)D * H * W;
    if (vec8(C, ldx, ldy, 8, x, y, y, 8 * P))
        launch_pdl(up8_kernel, grid_for(P * C / 8), 256, 0, (cudaStream_t)stream, (const bf16*)x, ldx, C / 8, H, W, (bf16*)y,
                   ldy, (unsigned)(P * C / 8));
    else
        up_kernel<<<grid_for(8 * P * C), 256, 0, (cudaStream_t)stream>>>((const bf16*)x, ldx, C, D, H, W, (bf16*)y, ldy);
    return launched("pat_unet_up");
}

pat_status pat_unet_up_bwd(const void* dy, int32_t ldd, int32_t C, int32_t D, int32_t H, int32_t W, void* dx, int32_t ldx,
                           void* stream) {
    if (!dy || !dx || C < 1 || ldx < C || ldd < C || D < 1 || H < 1 || W < 1) return bad("pat_unet_up_bwd: bad argument");
    const long long P = (long long)D * H * W;
    if (vec8(C, ldx, ldd, 8, dx, dy, dy, 8 * P))
        launch_pdl(up_bwd8_kernel, grid_for(P * C / 8), 256, 0, (cudaStream_t)stream,
                   (const bf16*)dy, ldd, C / 8, H, W, (bf16*)dx, ldx, nullptr, 0, (unsigned)(P * C / 8));
    else
        up_bwd_kernel<<<grid_for(P * C), 256, 0, (cudaStream_t)stream>>>((const bf16*)dy, ldd, C, D, H, W, (bf16*)dx, ldx);
    return launched("pat_unet_up_bwd");
}

pat_status pat_unet_up_bwd_masked(const void* dy, int32_t ldd, int32_t C, int32_t D, int32_t H, int32_t W, void* dx,
                                  int32_t ldx, const void* act, int32_t lda, void* stream) {
    if (!dy || !dx || !act || C < 1 || ldx < C || ldd < C || lda < C || D < 1 || H < 1 || W < 1)
        return bad("pat_unet_up_bwd_masked: bad argument");
    const long long P = (long long)D * H * W;
    if (vec8(C, ldx, ldd, lda, dx, dy, act, 8 * P)) {
        launch_pdl(up_bwd8_kernel, grid_for(P * C / 8), 256, 0, (cudaStream_t)stream,
                   (const bf16*)dy, ldd, C / 8, H, W, (bf16*)dx, ldx, (const bf16*)act, lda, (unsigned)(P * C / 8));
        return launched("pat_unet_up_bwd_masked");
    }
    const pat_status s = pat_unet_up_bwd(dy, ldd, C, D, H, W, dx, ldx, stream);
    return s != PAT_OK ? s : pat_unet_relu_bwd(dx, ldx, act, lda, C, P, stream);
}

pat_status pat_unet_input(const float* xin, float s, int64_t V, void* x16, void* stream) {
    if (!xin || !x16 || V < 0) return bad("pat_unet_input: bad argument");
    if (al16(x16)) launch_pdl(input8_kernel, grid_for(V * 2), 256, 0, (cudaStream_t)stream, xin, s, V * 2, (bf16*)x16);
    else input_kernel<<<grid_for(V * 16), 256, 0, (cudaStream_t)stream>>>(xin, s, V, (bf16*)x16);
    return launched("pat_unet_input");
}

pat_status pat_unet_head(const void* h, const float* head, int64_t V, float* out, void* stream) {
    if (!h || !head || !out || V < 0) return bad("pat_unet_head: bad argument");
    if (al16(h)) launch_pdl(head8_kernel, grid_for(V), 256, 0, (cudaStream_t)stream, (const bf16*)h, head, V, out);
    else head_kernel<<<grid_for(V), 256, 0, (cudaStream_t)stream>>>((const bf16*)h, head, V, out);
    return launched("pat_unet_head");
}

int64_t pat_unet_head_scratch(int64_t V) {
    (void)V;
    return (int64_t)kHeadBlocks * 18;
}

static pat_status head_bwd(const char* who, const void* h, const float* head, const float* out, const float* target,
                           int64_t V, void* dh, int mask, float* ghead, double* loss, double* partial, void* stream) {
    if (!h || !head || !out || !target || !dh || !ghead || !loss || !partial || V < 1)
        return bad((std::string(who) + ": bad argument").c_str());
    const cudaStream_t st = (cudaStream_t)stream;
    if (al16(h) && al16(dh))
        launch_pdl(head_bwd8_kernel, kHeadBlocks, 256, 0, st, (const bf16*)h, head, out, target, V, (bf16*)dh, mask,
                   partial);
    else
        head_bwd_kernel<<<kHeadBlocks, 256, 0, st>>>((const bf16*)h, head, out, target, V, (bf16*)dh, mask, partial);
    launch_pdl(head_bwd_final_kernel, 1, 18 * 32, 0, st, partial, kHeadBlocks, V, ghead, loss);
    return launched(who);
}

pat_status pat_unet_head_bwd(const void* h, const float* head, const float* out, const float* target, int64_t V, void* dh,
                             float* ghead, double* loss, double* partial, void* stream) {
    return head_bwd("pat_unet_head_bwd", h, head, out, target, V, dh, 0, ghead, loss, partial, stream);
}

pat_status pat_unet_head_bwd_masked(const void* h, const float* head, const float* out, const float* target, int64_t V,
                                    void* dh, float* ghead, double* loss, double* partial, void* stream) {
    return head_bwd("pat_unet_head_bwd_masked", h, head, out, target, V, dh, 1, ghead, loss, partial, stream);
}

pat_status pat_unet_adam(float* p, const float* g, float* m, float* v, int64_t n, float lr, float b1, float b2, float eps,
                         int32_t step, void* stream) {
    if (!p || !g || !m || !v || n < 0 || step < 1) return bad("pat_unet_adam: bad argument");
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    adam_kernel<<<grid_for(n), 256, 0, (cudaStream_t)stream>>>(p, g, m, v, n, lr, b1, b2, eps, c1, c2);
    return launched("pat_unet_adam");
}

}  // extern "C"
