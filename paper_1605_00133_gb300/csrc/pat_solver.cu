// pat_solver.cu - variational reconstruction on the GPU (arXiv:1605.00133, Sec. 4.5-4.6, App. A-B).
//
//   pat_tv_prox        argmin_{q >= 0} 1/2 ||q - p||^2 + alpha TV(q), TV isotropic with forward
//                      differences and Neumann boundary (App. A), by the accelerated primal-dual
//                      hybrid gradient method the paper names (App. B): one launch per iteration,
//                      the dual step (ball projection of xi + sigma grad(qbar)) fused with the
//                      primal step (divergence, data term, non-negativity clamp); step sizes follow
//                      theta = 1/sqrt(1 + 2 tau), tau <- theta tau, sigma <- sigma / theta,
//                      tau_0 = sigma_0 = 1/sqrt(12).
//   pat_bregman_solve  Bregman iterations (Eqs. BregIterA/B) around an accelerated proximal-gradient
//                      (FISTA) inner solver with restart and up to `max_backtrack` halvings of the
//                      step after a restart, eta = step_scale / L, L from power iteration (App. B).
// Fields and operators run in FP32; the data-space residual, the Bregman variable b, the objective
// and every norm and inner product are accumulated in FP64 (deterministic two-stage reductions).
// The host drives the iteration and reads one or two FP64 scalars per FISTA step.
#include <math.h>

#include <algorithm>
#include <string>

#include "pat_fft.cuh"
#include "pat_internal.h"

namespace pat {

#define PAT_CUDA(x, where)                                   \
    do {                                                     \
        cudaError_t _e = (x);                                \
        if (_e != cudaSuccess) return set_cuda_error(_e, where); \
    } while (0)

static constexpr int kRedBlocks = 512;
static constexpr int kRedThreads = 256;

static inline int ew_blocks(size_t n) {
    size_t b = (n + 255) / 256;
    return (int)std::min<size_t>(b, 152 * 16);
}

// ------------------------------------------------------------------------------ elementwise kernels

// z = a * x + b * y (float)
__global__ void axpby_kernel(float* __restrict__ z, const float* __restrict__ x, const float* __restrict__ y,
                             float a, float b, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        z[i] = fmaf(a, x[i], b * y[i]);
}

// r = (float)(ay - g)  (g in FP64)
__global__ void residual_kernel(float* __restrict__ r, const float* __restrict__ ay, const double* __restrict__ g, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        r[i] = (float)((double)ay[i] - g[i]);
}

// g = f + b (FP64)
__global__ void data_shift_kernel(double* __restrict__ g, const float* __restrict__ f, const double* __restrict__ b, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        g[i] = (double)f[i] + b[i];
}

// b += f - ax (FP64 Bregman update)
__global__ void bregman_update_kernel(double* __restrict__ b, const float* __restrict__ f, const float* __restrict__ ax, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        b[i] += (double)f[i] - (double)ax[i];
}

__global__ void clamp_copy_kernel(float* __restrict__ q, float* __restrict__ qbar, const float* __restrict__ p, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float v = fmaxf(0.f, p[i]);
        q[i] = v;
        qbar[i] = v;
    }
}

// ------------------------------------------------------------------------------ TV prox kernel

struct TvDims {
    int nz, ny, nx;
    size_t n;      // nz*ny*nx
    size_t total;  // B*n
};

// One primal-dual iteration per launch, dual and primal steps fused (App. B):
//   xi'   = project_{|.| <= alpha}(xi + sigma grad(qbar))        dual, every voxel
//   q'    = max(0, (q - tau grad^T(xi') + tau p) / (1 + tau))    primal, the clamp fused
//   qbar' = q' + theta (q' - q)
// grad: forward differences, zero past the last voxel of an axis; grad^T(xi)(v) = sum over axes of
// [xi_a(v - e_a) if v has a predecessor] - [xi_a(v) if v has a successor].
// A CTA owns a 32 x kTvRows tile of (x, y) columns over a run of z planes and marches along z:
// lanes are consecutive x, warps consecutive y, and warp 0 is the halo row y0 - 1, whose new dual
// the first output row needs.  The x neighbours come by warp shuffle (lane 31 loads qbar at
// x0 + 32, lane 0 also evaluates the dual at x0 - 1), the y neighbours through shared memory, and
// the new dual's z component of the plane below stays in a register; a run's first plane needs
// the plane before it, which the CTA evaluates first without storing it.  qbar and xi are read from
// one buffer and written to the other (neighbouring CTAs read the old values); q is read and
// written only at its own voxel.
constexpr int kTvRows = 8;
constexpr int kTvWarps = kTvRows + 1;

struct TvStep {
    const float* qb_in;
    float* qb_out;
    const float* xi_in;  // components z, y, x at offsets 0, N, 2N
    float* xi_out;
    float* q;
    const float* p;
    float sigma, alpha, tau, theta;
    int nonneg;
    int nz, ny, nx;
    int zrun, nruns;  // planes per run, runs per image
    long long n, N;   // voxels per image, B * n
};

// The projection of the dual (a, b, e) onto the ball of radius alpha multiplies it by tv_scale(its squared norm).
__device__ __forceinline__ float tv_scale(float n, float alpha) {
    const float g = sqrtf(n);
    return (g > alpha) ? alpha / g : 1.f;
}

// The squared norm.  Lines are cut into pieces of 32 voxels, and the dual of a piece's last voxel enters the
// voxel after it with the first two squares added the other way round (tv_square_seam).  Both kernels do so: the
// solver's restarts amplify a last bit of the prox to 1e-8 of its residuals, and a solve has to come out the same
// whichever kernel a length, an alignment or an odd iteration picks.
__device__ __forceinline__ float tv_square(float a, float b, float e) { return fmaf(e, e, fmaf(a, a, b * b)); }
__device__ __forceinline__ float tv_square_seam(float a, float b, float e) { return fmaf(e, e, fmaf(b, b, a * a)); }

// what a thread reads for plane z (its qbar at z itself is carried from the plane before)
struct TvIn {
    float qn;          // qbar at z + 1
    float xz, xy, xx;  // dual at the own voxel
    float qv, pv;      // q and the prox input (output voxels only)
    float qr, qd;      // qbar at x0 + 32 (lane 31) and at y + 1 (last warp)
    float qln, qld;    // lane 0 of the output rows: qbar at (z + 1, y, x0 - 1) and (z, y + 1, x0 - 1)
    float lz, ly, lx;  //   and the dual at (z, y, x0 - 1)
};

__global__ void __launch_bounds__(32 * kTvWarps) tv_step_kernel(TvStep a) {
    __shared__ float sq[kTvWarps][32];  // qbar of the current plane, one row per warp
    __shared__ float sy[kTvWarps][32];  // y component of the new dual, one row per warp
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int x0 = blockIdx.x * 32, x = x0 + lane;
    const int y = blockIdx.y * kTvRows - 1 + w;
    const int b = blockIdx.z / a.nruns, run = blockIdx.z - b * a.nruns;
    const int z0 = run * a.zrun, z1 = min(z0 + a.zrun, a.nz);
    const bool yin = y >= 0 && y < a.ny, in = yin && x < a.nx;
    const bool own = in && w > 0;                               // writes its voxel (planes z0 .. z1-1)
    const bool xn = x + 1 < a.nx, yn = y + 1 < a.ny;            // voxel has a successor along x / y
    const bool halo = lane == 0 && x0 > 0 && yin && w > 0;      // evaluates the dual at x0 - 1
    const bool right = lane == 31 && x0 + 32 < a.nx && yin;     // loads qbar at x0 + 32
    const bool down = w == kTvWarps - 1 && in && yn;            // loads qbar at y + 1
    const long long plane = (long long)a.ny * a.nx;
    const long long base = b * a.n + (long long)y * a.nx + x;   // + z * plane; dereferenced only when in
    const float* __restrict__ qb = a.qb_in;
    const float* __restrict__ xi = a.xi_in;
    auto load = [&](int z) {
        TvIn v;
        const long long o = base + z * plane;
        const bool zn = z + 1 < a.nz, store = own && z >= z0;
        v.qn = (in && zn) ? qb[o + plane] : 0.f;
        v.xz = in ? xi[o] : 0.f;
        v.xy = in ? xi[a.N + o] : 0.f;
        v.xx = in ? xi[2 * a.N + o] : 0.f;
        v.qv = store ? a.q[o] : 0.f;
        v.pv = store ? a.p[o] : 0.f;
        v.qr = right ? qb[o + 1] : 0.f;
        v.qd = down ? qb[o + a.nx] : 0.f;
        v.qln = (halo && zn) ? qb[o - 1 + plane] : 0.f;
        v.qld = (halo && yn) ? qb[o - 1 + a.nx] : 0.f;
        v.lz = halo ? xi[o - 1] : 0.f;
        v.ly = halo ? xi[a.N + o - 1] : 0.f;
        v.lx = halo ? xi[2 * a.N + o - 1] : 0.f;
        return v;
    };
    const int zs = z0 > 0 ? z0 - 1 : z0;
    float qc = in ? qb[base + zs * plane] : 0.f;         // qbar at (z, y, x)
    float qlc = halo ? qb[base - 1 + zs * plane] : 0.f;  // qbar at (z, y, x0 - 1)
    float pz = 0.f;                                      // z component of the new dual at z - 1
    // plane z from its reads `cur`.  The reads are not issued a plane ahead: a CTA barrier waits
    // for the loads in flight, so reads issued before the barriers of the plane before would
    // only add registers (measured slower).
    auto step = [&](int z, const TvIn& cur) {
        const long long o = base + z * plane;
        const bool zn = z + 1 < a.nz, store = own && z >= z0;
        sq[w][lane] = qc;
        __syncthreads();
        // new dual at the own voxel
        const float qxn = __shfl_down_sync(0xffffffffu, qc, 1);
        const float qyn = (w < kTvWarps - 1) ? sq[w + 1][lane] : cur.qd;
        const float gz = zn ? cur.qn - qc : 0.f;
        const float gy = yn ? qyn - qc : 0.f;
        const float gx = xn ? (lane < 31 ? qxn : cur.qr) - qc : 0.f;
        float dz = fmaf(a.sigma, gz, cur.xz), dy = fmaf(a.sigma, gy, cur.xy), dx = fmaf(a.sigma, gx, cur.xx);
        const float s = tv_scale(tv_square(dz, dy, dx), a.alpha);
        dz *= s;
        dy *= s;
        dx *= s;
        // new dual at x0 - 1 (lane 0 of the output rows): only its x component is used
        float dlx = 0.f;
        if (halo) {
            float ez = fmaf(a.sigma, zn ? cur.qln - qlc : 0.f, cur.lz);
            float ey = fmaf(a.sigma, yn ? cur.qld - qlc : 0.f, cur.ly);
            float ex = fmaf(a.sigma, qc - qlc, cur.lx);
            dlx = ex * tv_scale(tv_square_seam(ez, ey, ex), a.alpha);
        }
        sy[w][lane] = dy;
        __syncthreads();
        const float dxl = __shfl_up_sync(0xffffffffu, dx, 1);
        if (store) {
            float gt = 0.f;
            if (zn) gt -= dz;
            if (z > 0) gt += pz;
            if (yn) gt -= dy;
            if (y > 0) gt += sy[w - 1][lane];
            if (xn) gt -= dx;
            if (x > 0) gt += lane > 0 ? dxl : dlx;
            float qnew = fmaf(-a.tau, gt, fmaf(a.tau, cur.pv, cur.qv)) / (1.f + a.tau);
            if (a.nonneg) qnew = fmaxf(0.f, qnew);
            a.q[o] = qnew;
            a.qb_out[o] = fmaf(a.theta, qnew - cur.qv, qnew);
            a.xi_out[o] = dz;
            a.xi_out[a.N + o] = dy;
            a.xi_out[2 * a.N + o] = dx;
        }
        pz = dz;
        qc = cur.qn;
        qlc = cur.qln;
    };
    for (int z = zs; z < z1; z++) step(z, load(z));
}

// Two primal-dual iterations per launch.  One iteration moves 44 bytes per voxel for about 90 instructions; at
// 128x256x256, where the fields do not fit the L2, that was 105 us against 55 us of memory time, and at
// 64x128x128, where they do, 15.7 us of latency between barriers.  Fused, the fields are read and written once
// per two iterations.  A CTA owns rows y0 .. y0 + H - 1 (and 128 columns x of lines longer than that) over a run
// of z planes and marches along z; a thread holds four consecutive x of one row.  At plane z it evaluates
// the first iteration's dual and primal there and the second iteration's for plane z - 1, which needs the first
// one's over-relaxed iterate at z.  What the second iteration reads of neighbouring tiles is evaluated
// redundantly: all H + 3 rows y0 - 2 .. y0 + H in both iterations (of which the second needs two less, and the primals
// one less), and three planes more than a run stores (the second dual two).  At 64x128x128 (H = 8, runs of 8) that is
// 1.8 dual evaluations per voxel and iteration, at 128x256x256 1.68.  Neighbours along x and y come through
// shared memory (two barriers per plane for both iterations), along z through registers; a plane's inputs
// are fetched while the one before is computed.  Per voxel the operations are tv_step_kernel's, in the same
// order, so the results are the same bit for bit.  20 iterations of 128x256x256 2193 -> 1101 us,
// 50 of 64x128x128 829 -> 411 us.
struct TvStep2 {
    const float* qb_in;
    float* qb_out;
    const float* xi_in;  // components z, y, x at offsets 0, N, 2N
    float* xi_out;
    const float* q_in;
    float* q_out;
    const float* p;
    float alpha;
    float sigma[2], tau[2], theta[2], inv[2];  // inv = 1 / (1 + tau)
    int nonneg;
    int nz, ny, nx;
    int ntx, H, split;   // threads per row, rows stored per tile; split: lines longer than a tile
    int zrun, nruns;     // planes per run, runs per image
    long long n, N;      // voxels per image, B * n
};
constexpr int kTv2Cols = 128;     // columns a tile stores when lines are split (one more thread on each side)
constexpr int kTv2Threads = 384;  // most threads of a CTA

struct TvIn4 {
    float4 qn, qy;      // qbar at z + 1, at y + 1
    float qx;           // qbar at the x after the last of this thread's
    float4 xz, xy, xx;  // dual
    float4 q, p;
};

// tv_scale and v / d of the two-iteration kernel, which is bound by its instructions: the IEEE square root and
// divisions were half of an iteration's 253 per voxel.  Here the root and both quotients come from one
// reciprocal square root (and inv = 1 / d from the host) and are rounded through fma corrections: the residual of
// a root or quotient is exact in fma, and one correction by it gives the rounded value (P. Markstein,
// "Computation of elementary functions on the IBM RISC System/6000", 1990).  Compared with sqrtf and the division
// on the device: equal for all 2^24 mantissas and for 2^32 random quotients (12 differ without the step on
// 1 / g, for 2 % of the time).  The bounds on the radius keep the residuals' exponents in range for every norm
// that is scaled.  A numerator v below 2^-102 has a residual below the subnormals' spacing: such quotients (the front of
// an image that spreads into zeros decays through them) are divided after all, four at a time in a branch that is
// rarely taken (50 iterations of 64x128x128 with it 411 us, without 425: the division's loop is also cut in two).
// The norm comes out as NaN where its square is 0, infinite or NaN, of which the infinite one
// scales by 0 and the others by 1, as in tv_scale.
constexpr float kTvRadiusMin = 1e-15f, kTvRadiusMax = 1e15f;  // outside, or NaN: one iteration at a time
__device__ __forceinline__ float tv_scale_fast(float n, float alpha) {
    float r = rsqrtf(n), h = 0.5f * r, g = n * r;
    const float t = fmaf(-g, h, 0.5f);
    g = fmaf(g, t, g);
    h = fmaf(h, t, h);
    g = fmaf(fmaf(-g, g, n), h, g);      // sqrt(n)
    r = h + h;
    r = fmaf(r, fmaf(-g, r, 1.f), r);    // 1 / g
    float s = alpha * r;
    s = fmaf(fmaf(-s, g, alpha), r, s);  // alpha / g
    s = (g > alpha) ? s : 1.f;
    return (n > 3.402823466e38f) ? 0.f : s;
}
__device__ __forceinline__ float tv_divide(float v, float d, float inv) {
    const float q = v * inv, rem = fmaf(-q, d, v);
    return rem == rem ? fmaf(rem, inv, q) : q;  // infinite v
}

constexpr unsigned kTvTiny = 2u * 0x0d800000u;  // twice the bits of 2^-100
__device__ __noinline__ float4 tv_divide4(float4 v, float d) { return make_float4(v.x / d, v.y / d, v.z / d, v.w / d); }

__device__ __forceinline__ float& at4(float4& v, int i) { return reinterpret_cast<float*>(&v)[i]; }
__device__ __forceinline__ float at4(const float4& v, int i) { return reinterpret_cast<const float*>(&v)[i]; }

__global__ void __launch_bounds__(kTv2Threads, 1) tv_step2_kernel(TvStep2 a) {
    extern __shared__ float4 tv_smem[];
    const int rows = a.H + 3, ntx = a.ntx;
    // [row][thread]: y components of both duals, the over-relaxed iterate of two planes, and the x component of
    // each thread's last voxel
    float4* sdy1 = tv_smem;
    float4* sdy2 = sdy1 + rows * ntx;
    float4* sqb = sdy2 + rows * ntx;  // two planes
    float* sdx1 = reinterpret_cast<float*>(sqb + 2 * rows * ntx);
    float* sdx2 = sdx1 + rows * ntx;
    const int rr = threadIdx.x / ntx, tx = threadIdx.x - rr * ntx;
    const int me = threadIdx.x;  // rr * ntx + tx
    const int x = (a.split ? (int)blockIdx.x * kTv2Cols - 4 : 0) + 4 * tx;
    const int y = (int)blockIdx.y * a.H - 2 + rr;
    const int b = blockIdx.z / a.nruns, run = blockIdx.z - b * a.nruns;
    const int z0 = run * a.zrun, z1 = min(z0 + a.zrun, a.nz);
    const bool in = x >= 0 && x < a.nx && y >= 0 && y < a.ny;
    const bool own = in && rr >= 2 && rr < a.H + 2 && (!a.split || (tx > 0 && tx < ntx - 1));
    const bool yn = y + 1 < a.ny, xlast = x + 4 >= a.nx;  // the last of the four has no successor
    const bool seam = (x & 31) == 28;                     // the last of the four ends a piece of the line
    const float inside = a.alpha * a.alpha * 0.99999f;    // squared norms up to here are not scaled
    const bool upy = rr + 1 < rows;                       // row y + 1 is in the tile
    const long long plane = (long long)a.ny * a.nx;
    const long long base = b * a.n + (long long)y * a.nx + x;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    // through L2: written by the launch before, which may still run when this one starts
    auto ld = [](const float* p) { return __ldcg(reinterpret_cast<const float4*>(p)); };
    auto load = [&](int z) {
        TvIn4 v;
        const long long o = base + z * plane;
        const bool on = in && z < a.nz;
        v.qn = (on && z + 1 < a.nz) ? ld(a.qb_in + o + plane) : zero;
        v.qy = (on && yn) ? ld(a.qb_in + o + a.nx) : zero;
        v.qx = (on && !xlast) ? __ldcg(a.qb_in + o + 4) : 0.f;
        v.xz = on ? ld(a.xi_in + o) : zero;
        v.xy = on ? ld(a.xi_in + a.N + o) : zero;
        v.xx = on ? ld(a.xi_in + 2 * a.N + o) : zero;
        v.q = on ? ld(a.q_in + o) : zero;
        v.p = on ? ld(a.p + o) : zero;
        return v;
    };
    // new dual of four voxels from (dz, dy, dx) and qbar at them, at z + 1, y + 1 and the x after the last; dxr is
    // the last one's x component as it enters the voxel after it
    auto dual = [&](float sigma, bool zn, const float4& qc, const float4& qn, const float4& qy, float qx, float4& dz,
                    float4& dy, float4& dx, float& dxr) {
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const float c = at4(qc, i), r = i < 3 ? at4(qc, i + 1) : qx;
            const float gz = zn ? at4(qn, i) - c : 0.f;
            const float gy = yn ? at4(qy, i) - c : 0.f;
            const float gx = (i < 3 || !xlast) ? r - c : 0.f;
            float ez = fmaf(sigma, gz, at4(dz, i)), ey = fmaf(sigma, gy, at4(dy, i)), ex = fmaf(sigma, gx, at4(dx, i));
            const float n = tv_square(ez, ey, ex), s = tv_scale_fast(n, a.alpha);
            at4(dz, i) = ez * s;
            at4(dy, i) = ey * s;
            at4(dx, i) = ex * s;
            if (i == 3) {
                const float ns = tv_square_seam(ez, ey, ex);
                float ss = s;
                if (seam && ns != n && ns > inside) ss = tv_scale_fast(ns, a.alpha);  // else the same
                dxr = ex * ss;
            }
        }
    };
    // new primal and over-relaxed iterate from the new dual, its z component at z - 1, y component at y - 1 and x
    // component at the x before the first
    auto primal = [&](int k, int z, const float4& q, const float4& p, const float4& dz, const float4& pz, const float4& dy,
                      const float4& dyl, const float4& dx, float dxl, float4& qn, float4& qb) {
        const float tau = a.tau[k], theta = a.theta[k];
        const bool zn = z + 1 < a.nz;
        float4 num, quo;
        unsigned least = ~0u;  // twice the least magnitude but 0, less 1
#pragma unroll
        for (int i = 0; i < 4; i++) {
            float gt = 0.f;
            if (zn) gt -= at4(dz, i);
            if (z > 0) gt += at4(pz, i);
            if (yn) gt -= at4(dy, i);
            if (y > 0) gt += at4(dyl, i);
            if (i < 3 || !xlast) gt -= at4(dx, i);
            if (i > 0 || x > 0) gt += i > 0 ? at4(dx, i - 1) : dxl;
            at4(num, i) = fmaf(-tau, gt, fmaf(tau, at4(p, i), at4(q, i)));
            at4(quo, i) = tv_divide(at4(num, i), 1.f + tau, a.inv[k]);
            least = min(least, 2u * __float_as_uint(at4(num, i)) - 1u);
        }
        if (least < kTvTiny) quo = tv_divide4(num, 1.f + tau);
#pragma unroll
        for (int i = 0; i < 4; i++) {
            float v = at4(quo, i);
            if (a.nonneg) v = fmaxf(0.f, v);
            at4(qn, i) = v;
            at4(qb, i) = fmaf(theta, v - at4(q, i), v);
        }
    };
    const int up = me + ntx, down = me - ntx;  // rows y + 1, y - 1
    pdl_wait();     // the launch before, whose results these are, is complete
    pdl_trigger();  // the next one may be set up while this one runs
    const int zs = z0 > 1 ? z0 - 2 : 0;
    float4 qc = in ? ld(a.qb_in + base + zs * plane) : zero;  // qbar at z
    float4 pz1 = zero, pz2 = zero;                            // z component of the duals a plane before
    float4 d1z = zero, d1y = zero, d1x = zero;                // first dual, iterate and input at z - 1
    float4 q1 = zero, qb1 = zero, p1 = zero;
    TvIn4 cur = load(zs);
    for (int z = zs; z <= z1; z++) {
        const TvIn4 nxt = load(z + 1 <= z1 ? z + 1 : a.nz);
        float4 dz = cur.xz, dy = cur.xy, dx = cur.xx;
        dual(a.sigma[0], z + 1 < a.nz, qc, cur.qn, cur.qy, cur.qx, dz, dy, dx, sdx1[me]);
        sdy1[me] = dy;
        __syncthreads();
        // first primal at z
        float4 qn, qb;
        {
            const float4 dyl = rr > 0 ? sdy1[down] : zero;
            const float dxl = tx > 0 ? sdx1[me - 1] : 0.f;
            primal(0, z, cur.q, cur.p, dz, pz1, dy, dyl, dx, dxl, qn, qb);
        }
        float4* sq = sqb + (z & 1) * rows * ntx;
        sq[me] = qb;
        // second dual at z - 1 (from the second plane on; its neighbours were stored a plane ago)
        float4 ez = d1z, ey = d1y, ex = d1x;
        if (z > zs) {
            const float4* so = sqb + ((z - 1) & 1) * rows * ntx;
            const float4 qy = upy ? so[up] : zero;
            const float qx = tx + 1 < ntx ? so[me + 1].x : 0.f;
            dual(a.sigma[1], z < a.nz, qb1, qb, qy, qx, ez, ey, ex, sdx2[me]);
        }
        sdy2[me] = ey;
        __syncthreads();
        // second primal at z - 1
        if (own && z - 1 >= z0) {
            float4 q2, qb2;
            primal(1, z - 1, q1, p1, ez, pz2, ey, sdy2[down], ex, tx > 0 ? sdx2[me - 1] : 0.f, q2, qb2);
            const long long o = base + (z - 1) * plane;
            auto st = [](float* p, const float4& v) { *reinterpret_cast<float4*>(p) = v; };
            st(a.q_out + o, q2);
            st(a.qb_out + o, qb2);
            st(a.xi_out + o, ez);
            st(a.xi_out + a.N + o, ey);
            st(a.xi_out + 2 * a.N + o, ex);
        }
        pz1 = dz;
        pz2 = ez;
        d1z = dz;
        d1y = dy;
        d1x = dx;
        q1 = qn;
        qb1 = qb;
        p1 = cur.p;
        qc = cur.qn;
        cur = nxt;
    }
}

// ------------------------------------------------------------------------------ FP64 reductions

enum RedOp { RED_SUMSQ_DIFF = 0, RED_TV = 1, RED_SUMSQ = 2, RED_ABS_DIFF = 3, RED_DOT = 4, RED_SUMSQ_DIFF_FF = 5 };

struct RedArgs {
    int op;
    const float* a;
    const float* b;    // second float operand (ABS_DIFF, DOT)
    const double* gd;  // FP64 operand (SUMSQ_DIFF: sum (a - gd)^2)
    size_t n;
    TvDims d;          // RED_TV
};

__device__ __forceinline__ double red_term(const RedArgs& r, size_t i) {
    switch (r.op) {
        case RED_SUMSQ_DIFF: {
            const double e = (double)r.a[i] - r.gd[i];
            return e * e;
        }
        case RED_TV: {
            const size_t plane = (size_t)r.d.ny * r.d.nx;
            const unsigned v = (unsigned)(i % r.d.n), nx = (unsigned)r.d.nx, ny = (unsigned)r.d.ny;
            const unsigned t = v / nx;
            const int x = (int)(v - t * nx), y = (int)(t % ny), z = (int)(t / ny);
            const double c = r.a[i];
            const double gz = (z + 1 < r.d.nz) ? (double)r.a[i + plane] - c : 0.0;
            const double gy = (y + 1 < r.d.ny) ? (double)r.a[i + r.d.nx] - c : 0.0;
            const double gx = (x + 1 < r.d.nx) ? (double)r.a[i + 1] - c : 0.0;
            return sqrt(gz * gz + gy * gy + gx * gx);
        }
        case RED_SUMSQ: {
            const double e = r.a[i];
            return e * e;
        }
        case RED_ABS_DIFF: return fabs((double)r.a[i] - (double)r.b[i]);
        case RED_SUMSQ_DIFF_FF: {
            const double e = (double)r.a[i] - (double)r.b[i];
            return e * e;
        }
        default: return (double)r.a[i] * (double)r.b[i];
    }
}

// Up to kRedMost sums at once, one per blockIdx.y (stage 1) or block (stage 2), and one wait of the host for them
// all: what an iteration needs (data term, TV, change) took three pairs of launches, copies and waits, during each of
// which the GPU stood still for about 20 us.  Stage 2 writes the results to pinned host memory itself.
constexpr int kRedMost = 3;
struct RedSet {
    RedArgs r[kRedMost];
    int nb[kRedMost];  // blocks of each sum
};

__global__ void reduce_stage1_kernel(const __grid_constant__ RedSet s, double* partial) {
    __shared__ double sh[kRedThreads / 32];
    const RedArgs& r = s.r[blockIdx.y];
    const int nb = s.nb[blockIdx.y];
    if ((int)blockIdx.x >= nb) return;
    double acc = 0.0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < r.n; i += (size_t)nb * blockDim.x)
        acc += red_term(r, i);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kRedThreads / 32; w++) t += sh[w];
        partial[blockIdx.y * kRedBlocks + blockIdx.x] = t;
    }
}

__global__ void reduce_stage2_kernel(const __grid_constant__ RedSet s, const double* partial, double* out) {
    __shared__ double sh[kRedThreads];
    const double* p = partial + blockIdx.x * kRedBlocks;
    const int np = s.nb[blockIdx.x];
    double acc = 0.0;
    for (int i = threadIdx.x; i < np; i += blockDim.x) acc += p[i];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) sh[threadIdx.x] += sh[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = sh[0];
}

// ------------------------------------------------------------------------------ host helpers

struct Ctx {
    pat_grid* G;
    cudaStream_t st;
    size_t N;   // image elements (B*nz*ny*nx)
    size_t D;   // data elements (B*T*m)
    TvDims td;
};

// n sums; the host waits for them
static pat_status reduce(Ctx& c, const RedArgs* r, int n, double* out) {
    SolverWs& w = c.G->sw;
    RedSet s = {};
    int most = 1;
    for (int k = 0; k < n; k++) {
        s.r[k] = r[k];
        s.nb[k] = (int)std::min<size_t>(kRedBlocks, std::max<size_t>(1, (r[k].n + kRedThreads - 1) / kRedThreads));
        most = std::max(most, s.nb[k]);
    }
    reduce_stage1_kernel<<<dim3((unsigned)most, (unsigned)n), kRedThreads, 0, c.st>>>(s, w.partial);
    reduce_stage2_kernel<<<n, kRedThreads, 0, c.st>>>(s, w.partial, w.host);
    PAT_CUDA(cudaGetLastError(), "reduction launch");
    PAT_CUDA(cudaStreamSynchronize(c.st), "reduction sync");
    for (int k = 0; k < n; k++) out[k] = w.host[k];
    return PAT_OK;
}

// A buffer of the workspace, unless it is there: a call that ran out of memory leaves some of them, and the next one
// goes on from there.
template <class T>
static pat_status ensure(pat_grid* G, T** p, size_t count, const char* what) {
    if (*p) return PAT_OK;
    void* q = nullptr;
    const pat_status st = grid_alloc(G, &q, count * sizeof(T), what);
    if (st == PAT_OK) *p = (T*)q;
    return st;
}

static pat_status ensure_ws(pat_grid* G, bool solver) {
    SolverWs& w = G->sw;
    const size_t N = (size_t)G->g.B * G->g.nreal;
    const size_t D = (size_t)G->g.B * G->g.T * (size_t)G->m;
    pat_status st = PAT_OK;
    if (!w.n_img) {
        st = ensure(G, &w.qbar, N, "prox qbar");
        if (st == PAT_OK) st = ensure(G, &w.qbar2, N, "prox qbar");
        if (st == PAT_OK) st = ensure(G, &w.xi, 3 * N, "prox dual");
        if (st == PAT_OK) st = ensure(G, &w.xi2, 3 * N, "prox dual");
        if (st == PAT_OK) st = ensure(G, &w.z, N, "prox input copy");
        if (st == PAT_OK) st = ensure(G, &w.q2, N, "prox iterate");
        if (st == PAT_OK) st = ensure(G, &w.partial, kRedMost * kRedBlocks, "reduction");
        if (st == PAT_OK && !w.host) {
            cudaError_t e = cudaMallocHost((void**)&w.host, 4 * sizeof(double));
            if (e != cudaSuccess) {
                w.host = nullptr;
                return set_cuda_error(e, "cudaMallocHost(reduction)");
            }
        }
        if (st != PAT_OK) return st;
        w.n_img = N;
    }
    if (solver && !w.n_dat) {
        const size_t data = std::max<size_t>(D, 1);
        st = ensure(G, &w.x, N, "solver x");
        if (st == PAT_OK) st = ensure(G, &w.xp, N, "solver x_prev");
        if (st == PAT_OK) st = ensure(G, &w.y, N, "solver y");
        if (st == PAT_OK) st = ensure(G, &w.grad, N, "solver gradient");
        if (st == PAT_OK) st = ensure(G, &w.ax, data, "solver Ax");
        if (st == PAT_OK) st = ensure(G, &w.axp, data, "solver Ax_prev");
        if (st == PAT_OK) st = ensure(G, &w.ay, data, "solver Ay");
        if (st == PAT_OK) st = ensure(G, &w.r, data, "solver residual");
        if (st == PAT_OK) st = ensure(G, &w.gdat, data, "solver data");
        if (st == PAT_OK) st = ensure(G, &w.bdat, data, "solver Bregman");
        if (st != PAT_OK) return st;
        w.n_dat = data;
    }
    return PAT_OK;
}

// Tiling of tv_step2_kernel: rows per tile so that a CTA has up to kTv2Threads threads, and the z run that
// minimises rounds of CTAs times planes marched (a run evaluates three planes more than it stores).
static void tv2_plan(const TvDims& d, int B, TvStep2* a, dim3* grid, int* threads, size_t* smem) {
    a->split = d.nx > kTv2Cols;
    a->ntx = a->split ? kTv2Cols / 4 + 2 : d.nx / 4;
    int H = 16;
    while (H > 8 && (H + 3) * a->ntx > kTv2Threads) H /= 2;
    if (H > d.ny) H = d.ny;
    // where every plane of every tile of 8 rows can have an SM of its own, no more than one warp a scheduler
    // (50 iterations of 32^3: 135 -> 121 us)
    if (H > 8 && (H + 3) * a->ntx > 128 && (long long)((d.ny + 7) / 8) * d.nz * B <= 152) H = 8;
    a->H = H;
    const int gx = a->split ? (d.nx + kTv2Cols - 1) / kTv2Cols : 1, gy = (d.ny + H - 1) / H;
    const long long tiles = (long long)gx * gy * B;
    *threads = (H + 3) * a->ntx;
    // CTAs resident: 14 warps an SM (of 139 registers a thread).  Counted as 384 threads, which narrow tiles do not reach,
    // 50 iterations of 128x256x16 took 309 us, now 271
    const int resident = 152 * std::max(1, 14 / ((*threads + 31) / 32));
    long long best = 0;
    for (int run = 1; run <= d.nz; run++) {
        const int n = (d.nz + run - 1) / run;
        if ((long long)B * n > 65535) continue;  // grid's z extent
        const long long cost = ((tiles * n + resident - 1) / resident) * (run + 3);
        if (best == 0 || cost < best) {
            best = cost;
            a->zrun = run;
            a->nruns = n;
        }
    }
    *grid = dim3(gx, gy, B * a->nruns);
    *smem = (size_t)*threads * (4 * sizeof(float4) + 2 * sizeof(float));
}

// PDHG for the positivity-constrained TV denoising problem; q (output) must not alias p.
static pat_status tv_prox_run(Ctx& c, const float* p, float* q, double alpha, int iters, int nonneg) {
    SolverWs& w = c.G->sw;
    const int nb = ew_blocks(c.N);
    // iterations two at a time (16-byte accesses; a caller's image may be aligned to less)
    const bool vec = (((uintptr_t)p | (uintptr_t)q) & 15) == 0;
    const int pairs = vec && alpha >= kTvRadiusMin && alpha <= kTvRadiusMax ? iters / 2 : 0;
    // pairs of iterations read one iterate buffer and write the other, the last one q
    float* qbuf[2] = {(pairs & 1) ? w.q2 : q, (pairs & 1) ? q : w.q2};
    clamp_copy_kernel<<<nb, 256, 0, c.st>>>(qbuf[0], w.qbar, p, c.N);
    if (!nonneg) PAT_CUDA(cudaMemcpyAsync(qbuf[0], p, c.N * sizeof(float), cudaMemcpyDeviceToDevice, c.st), "prox init");
    if (!nonneg) PAT_CUDA(cudaMemcpyAsync(w.qbar, p, c.N * sizeof(float), cudaMemcpyDeviceToDevice, c.st), "prox init");
    if (alpha <= 0.0 || iters == 0) {
        PAT_CUDA(cudaGetLastError(), "prox launch");
        return PAT_OK;
    }
    PAT_CUDA(cudaMemsetAsync(w.xi, 0, 3 * c.N * sizeof(float), c.st), "prox init");
    const TvDims& d = c.td;
    const int B = (int)(d.total / d.n);
    float* qb[2] = {w.qbar, w.qbar2};
    float* xi[2] = {w.xi, w.xi2};
    double tau = 1.0 / sqrt(12.0), sigma = 1.0 / (tau * 12.0);
    auto next = [&](float* sg, float* ta, float* th) {
        const double theta = 1.0 / sqrt(1.0 + 2.0 * tau);
        *sg = (float)sigma;
        *ta = (float)tau;
        *th = (float)theta;
        tau *= theta;
        sigma /= theta;
    };
    if (pairs > 0) {
        TvStep2 a = {};
        dim3 grid;
        int threads;
        size_t smem;
        tv2_plan(d, B, &a, &grid, &threads, &smem);
        a.p = p;
        a.alpha = (float)alpha;
        a.nonneg = nonneg;
        a.nz = d.nz;
        a.ny = d.ny;
        a.nx = d.nx;
        a.n = (long long)d.n;
        a.N = (long long)d.total;
        for (int it = 0; it < pairs; it++) {
            const int in = it & 1, out = in ^ 1;
            a.qb_in = qb[in];
            a.qb_out = qb[out];
            a.xi_in = xi[in];
            a.xi_out = xi[out];
            a.q_in = qbuf[in];
            a.q_out = qbuf[out];
            for (int k = 0; k < 2; k++) {
                next(&a.sigma[k], &a.tau[k], &a.theta[k]);
                a.inv[k] = 1.f / (1.f + a.tau[k]);
            }
            PAT_CUDA(launch_pdl(tv_step2_kernel, grid, threads, smem, c.st, a), "prox launch");
        }
    }
    // what is left (an odd iteration; all of them for unaligned images) one at a time, in place on q
    if (2 * pairs < iters) {
        const int gx = (d.nx + 31) / 32, gy = (d.ny + kTvRows - 1) / kTvRows;
        // runs of z planes: about 512 CTAs in all, at least 4 planes per run (each run evaluates one
        // plane more than it stores)
        const long long cols = (long long)gx * gy * B;
        int nruns = (int)std::max<long long>(1, std::min<long long>((512 + cols - 1) / cols, (d.nz + 3) / 4));
        const int zrun = (d.nz + nruns - 1) / nruns;
        nruns = (d.nz + zrun - 1) / zrun;
        TvStep a;
        a.q = q;
        a.p = p;
        a.alpha = (float)alpha;
        a.nonneg = nonneg;
        a.nz = d.nz;
        a.ny = d.ny;
        a.nx = d.nx;
        a.zrun = zrun;
        a.nruns = nruns;
        a.n = (long long)d.n;
        a.N = (long long)d.total;
        for (int it = 2 * pairs; it < iters; it++) {
            const int in = (it - pairs) & 1;  // buffers alternate per launch
            a.qb_in = qb[in];
            a.qb_out = qb[in ^ 1];
            a.xi_in = xi[in];
            a.xi_out = xi[in ^ 1];
            next(&a.sigma, &a.tau, &a.theta);
            tv_step_kernel<<<dim3(gx, gy, B * nruns), 32 * kTvWarps, 0, c.st>>>(a);
        }
    }
    PAT_CUDA(cudaGetLastError(), "prox launch");
    return PAT_OK;
}

// E = 1/2 ||ax - g||^2 + lam TV(x) and, with xp, change = ||x - xp||_1
static pat_status energy(Ctx& c, const float* ax, const float* x, double lam, double* E, const float* xp, double* change) {
    RedArgs r[kRedMost] = {};
    r[0].op = RED_SUMSQ_DIFF;
    r[0].a = ax;
    r[0].gd = c.G->sw.gdat;
    r[0].n = c.D;
    r[1].op = RED_TV;
    r[1].a = x;
    r[1].n = c.N;
    r[1].d = c.td;
    r[2].op = RED_ABS_DIFF;
    r[2].a = x;
    r[2].b = xp;
    r[2].n = c.N;
    double v[kRedMost] = {};
    const pat_status st = reduce(c, r, xp ? 3 : 2, v);
    if (st != PAT_OK) return st;
    *E = 0.5 * v[0] + lam * v[1];
    if (xp) *change = v[2];
    return PAT_OK;
}

static pat_status A_fwd(Ctx& c, const float* x, float* ax) {
    pat_grid* G = c.G;
    cudaError_t e = run_forward(G->g, G->t, G->w, G->s, G->kind, G->m, x, ax, c.st, nullptr);
    if (e != cudaSuccess) return set_cuda_error(e, "solver forward");
    return PAT_OK;
}

static pat_status A_adj(Ctx& c, const float* r, float* out) {
    pat_grid* G = c.G;
    cudaError_t e = run_adjoint(G->g, G->t, G->w, G->s, G->kind, G->m, r, out, c.st, nullptr);
    if (e != cudaSuccess) return set_cuda_error(e, "solver adjoint");
    return PAT_OK;
}

// grad = A^T C^T (ax - g)
static pat_status gradient(Ctx& c, const float* ax, float* grad) {
    SolverWs& w = c.G->sw;
    residual_kernel<<<ew_blocks(c.D), 256, 0, c.st>>>(w.r, ax, w.gdat, c.D);
    PAT_CUDA(cudaGetLastError(), "residual launch");
    return A_adj(c, w.r, grad);
}

// x = prox_{eta lam}(base - eta grad)
static pat_status prox_step(Ctx& c, const float* base, const float* grad, double eta, double lam,
                            int prox_iters, float* x) {
    SolverWs& w = c.G->sw;
    axpby_kernel<<<ew_blocks(c.N), 256, 0, c.st>>>(w.z, base, grad, 1.f, (float)-eta, c.N);
    PAT_CUDA(cudaGetLastError(), "step launch");
    return tv_prox_run(c, w.z, x, eta * lam, prox_iters, 1);
}

// Power iteration for L ~ ||A^T C^T C A||_2 from a seeded Gaussian start (SplitMix64 + Box-Muller).
static pat_status power_iteration(Ctx& c, int iters, uint64_t seed, double* L) {
    SolverWs& w = c.G->sw;
    std::vector<float> h(c.N);
    uint64_t state = seed;
    auto next = [&]() {
        state += 0x9E3779B97F4A7C15ull;
        uint64_t z = state;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        return (double)(z >> 11) * (1.0 / 9007199254740992.0);
    };
    for (size_t i = 0; i < c.N; i++) {
        const double u1 = next(), u2 = next();
        h[i] = (float)(sqrt(-2.0 * log(1.0 - u1)) * cos(2.0 * M_PI * u2));
    }
    PAT_CUDA(cudaMemcpyAsync(w.x, h.data(), c.N * sizeof(float), cudaMemcpyHostToDevice, c.st), "power init");
    double nrm = 0.0;
    RedArgs r = {};
    r.op = RED_SUMSQ;
    r.a = w.x;
    r.n = c.N;
    pat_status st = reduce(c, &r, 1, &nrm);
    if (st != PAT_OK) return st;
    nrm = sqrt(nrm);
    double lam = 0.0;
    for (int it = 0; it < iters; it++) {
        axpby_kernel<<<ew_blocks(c.N), 256, 0, c.st>>>(w.x, w.x, w.x, (float)(1.0 / nrm), 0.f, c.N);
        PAT_CUDA(cudaGetLastError(), "power launch");
        if ((st = A_fwd(c, w.x, w.ax)) != PAT_OK) return st;
        if ((st = A_adj(c, w.ax, w.x)) != PAT_OK) return st;
        r.a = w.x;
        if ((st = reduce(c, &r, 1, &nrm)) != PAT_OK) return st;
        nrm = sqrt(nrm);
        lam = nrm;
        if (!(nrm > 0)) break;
    }
    *L = lam;
    return PAT_OK;
}

struct FistaOut {
    int iterations = 0, restarts = 0;
    double energy = 0.0;
};

// FISTA with restart and backtracking; x_prev holds the start on entry and the result on exit,
// ax_prev its image under C A.  Buffers are swapped by pointer, so results are copied back into
// the solver workspace's canonical xp / axp at the end.
static pat_status fista(Ctx& c, const pat_solve_params& P, double eta, FistaOut* out) {
    SolverWs& w = c.G->sw;
    float *x = w.x, *xp = w.xp, *y = w.y;
    float *ax = w.ax, *axp = w.axp, *ay = w.ay;
    pat_status st;
    if ((st = A_fwd(c, xp, axp)) != PAT_OK) return st;
    double Ep = 0.0;
    if ((st = energy(c, axp, xp, P.lambda, &Ep, nullptr, nullptr)) != PAT_OK) return st;
    PAT_CUDA(cudaMemcpyAsync(y, xp, c.N * sizeof(float), cudaMemcpyDeviceToDevice, c.st), "fista init");
    PAT_CUDA(cudaMemcpyAsync(ay, axp, c.D * sizeof(float), cudaMemcpyDeviceToDevice, c.st), "fista init");
    double t = 1.0, best = Ep;
    int since_best = 0;
    for (int it = 0; it < P.inner; it++) {
        if ((st = gradient(c, ay, w.grad)) != PAT_OK) return st;
        if ((st = prox_step(c, y, w.grad, eta, P.lambda, P.prox_iters, x)) != PAT_OK) return st;
        if ((st = A_fwd(c, x, ax)) != PAT_OK) return st;
        double E = 0.0, change = 0.0;
        if ((st = energy(c, ax, x, P.lambda, &E, xp, &change)) != PAT_OK) return st;
        if (E > Ep) {
            out->restarts++;
            t = 1.0;
            if ((st = gradient(c, axp, w.grad)) != PAT_OK) return st;
            double eta_b = eta;
            for (int b = 0; b <= P.max_backtrack; b++) {
                if ((st = prox_step(c, xp, w.grad, eta_b, P.lambda, P.prox_iters, x)) != PAT_OK) return st;
                if ((st = A_fwd(c, x, ax)) != PAT_OK) return st;
                if ((st = energy(c, ax, x, P.lambda, &E, xp, &change)) != PAT_OK) return st;
                if (E <= Ep) break;
                eta_b *= 0.5;
            }
            if (E > Ep) {  // no descent found: keep the previous iterate
                PAT_CUDA(cudaMemcpyAsync(x, xp, c.N * sizeof(float), cudaMemcpyDeviceToDevice, c.st), "fista keep");
                PAT_CUDA(cudaMemcpyAsync(ax, axp, c.D * sizeof(float), cudaMemcpyDeviceToDevice, c.st), "fista keep");
                E = Ep;
                change = 0.0;
            }
        }
        out->iterations++;
        const double t_next = 0.5 * (1.0 + sqrt(1.0 + 4.0 * t * t));
        const double beta = (t - 1.0) / t_next;
        axpby_kernel<<<ew_blocks(c.N), 256, 0, c.st>>>(y, x, xp, (float)(1.0 + beta), (float)-beta, c.N);
        axpby_kernel<<<ew_blocks(c.D), 256, 0, c.st>>>(ay, ax, axp, (float)(1.0 + beta), (float)-beta, c.D);
        PAT_CUDA(cudaGetLastError(), "momentum launch");
        std::swap(x, xp);
        std::swap(ax, axp);
        Ep = E;
        t = t_next;
        if (E < best) {
            best = E;
            since_best = 0;
        } else {
            since_best++;
        }
        if (change == 0.0 || since_best >= P.stall) break;
    }
    if (xp != w.xp) PAT_CUDA(cudaMemcpyAsync(w.xp, xp, c.N * sizeof(float), cudaMemcpyDeviceToDevice, c.st), "fista out");
    if (axp != w.axp) PAT_CUDA(cudaMemcpyAsync(w.axp, axp, c.D * sizeof(float), cudaMemcpyDeviceToDevice, c.st), "fista out");
    out->energy = Ep;
    return PAT_OK;
}

}  // namespace pat

using namespace pat;

extern "C" pat_status pat_tv_prox(pat_grid* G, const float* in, float* out, double alpha, int32_t iters,
                                  int32_t bc, void* stream) {
    const NvtxRange range("pat_tv_prox");
    set_error(PAT_OK, "");
    if (!G) return set_error(PAT_ERR_INVALID_ARG, "pat_tv_prox: NULL grid");
    if (!in || !out) return set_error(PAT_ERR_INVALID_ARG, "pat_tv_prox: NULL buffer");
    if (!(alpha >= 0) || iters < 0) return set_error(PAT_ERR_INVALID_ARG, "pat_tv_prox: need alpha >= 0, iters >= 0");
    if (bc != 0) return set_error(PAT_ERR_UNSUPPORTED, "pat_tv_prox: only the Neumann boundary (bc = 0) is built");
    pat_status st = check_grid_device(G);
    if (st != PAT_OK) return st;
    if ((st = ensure_ws(G, false)) != PAT_OK) return st;
    Ctx c;
    c.G = G;
    c.st = (cudaStream_t)stream;
    c.N = (size_t)G->g.B * G->g.nreal;
    c.D = 0;
    c.td = TvDims{G->g.nz, G->g.ny, G->g.nx, (size_t)G->g.nreal, c.N};
    const float* p = in;
    if (in == out) {  // the primal step reads the input every iteration
        cudaError_t e = cudaMemcpyAsync(G->sw.z, in, c.N * sizeof(float), cudaMemcpyDeviceToDevice, c.st);
        if (e != cudaSuccess) return set_cuda_error(e, "pat_tv_prox copy");
        p = G->sw.z;
    }
    return tv_prox_run(c, p, out, alpha, iters, 1);
}

extern "C" pat_status pat_bp_tv(pat_grid* G, const float* f, float* p_out, double alpha, int32_t iters,
                                void* stream) {
    const NvtxRange range("pat_bp_tv");
    set_error(PAT_OK, "");
    if (!G) return set_error(PAT_ERR_INVALID_ARG, "pat_bp_tv: NULL grid");
    if (!p_out || (!f && G->m > 0)) return set_error(PAT_ERR_INVALID_ARG, "pat_bp_tv: NULL buffer");
    if (!(alpha >= 0) || iters < 0) return set_error(PAT_ERR_INVALID_ARG, "pat_bp_tv: need alpha >= 0, iters >= 0");
    pat_status st = check_grid_device(G);
    if (st != PAT_OK) return st;
    if ((st = ensure_ws(G, false)) != PAT_OK) return st;
    Ctx c;
    c.G = G;
    c.st = (cudaStream_t)stream;
    c.N = (size_t)G->g.B * G->g.nreal;
    c.D = 0;
    c.td = TvDims{G->g.nz, G->g.ny, G->g.nx, (size_t)G->g.nreal, c.N};
    // back-projection A^T C^T f (Eq. BP) into the prox's input buffer, then its TV+ denoising
    float* bp = G->sw.z;
    cudaError_t e = run_adjoint(G->g, G->t, G->w, G->s, G->kind, G->m, f, bp, c.st, nullptr);
    if (e != cudaSuccess) return set_cuda_error(e, "pat_bp_tv adjoint");
    return tv_prox_run(c, bp, p_out, alpha, iters, 1);
}

extern "C" pat_status pat_bregman_solve(pat_grid* G, const float* f, const float* warm, float* p_out,
                                        const pat_solve_params* params, pat_solve_report* report, void* stream) {
    const NvtxRange range("pat_bregman_solve");
    set_error(PAT_OK, "");
    if (!G || !params) return set_error(PAT_ERR_INVALID_ARG, "pat_bregman_solve: NULL grid or params");
    if (!f || !p_out) return set_error(PAT_ERR_INVALID_ARG, "pat_bregman_solve: NULL buffer");
    if (G->g.B != 1) return set_error(PAT_ERR_UNSUPPORTED, "pat_bregman_solve: batch must be 1");
    const pat_solve_params P = *params;
    if (!(P.lambda >= 0) || P.outer < 1 || P.inner < 1 || P.prox_iters < 1 || P.max_backtrack < 0 ||
        P.stall < 1 || !(P.step_scale > 0) || (P.L <= 0 && P.power_iters < 1))
        return set_error(PAT_ERR_INVALID_ARG, "pat_bregman_solve: invalid parameters");
    pat_status st = check_grid_device(G);
    if (st != PAT_OK) return st;
    if ((st = ensure_ws(G, true)) != PAT_OK) return st;
    Ctx c;
    c.G = G;
    c.st = (cudaStream_t)stream;
    c.N = (size_t)G->g.nreal;
    c.D = (size_t)G->g.T * G->m;
    c.td = TvDims{G->g.nz, G->g.ny, G->g.nx, (size_t)G->g.nreal, c.N};
    SolverWs& w = G->sw;
    pat_solve_report rep = {};
    double L = P.L;
    if (L <= 0) {
        if ((st = power_iteration(c, P.power_iters, P.seed, &L)) != PAT_OK) return st;
        if (!(L > 0)) return set_error(PAT_ERR_NOT_CONVERGED, "pat_bregman_solve: power iteration gave L <= 0");
    }
    rep.L = L;
    const double eta = P.step_scale / L;
    if (warm) PAT_CUDA(cudaMemcpyAsync(w.xp, warm, c.N * sizeof(float), cudaMemcpyDeviceToDevice, c.st), "warm start");
    else PAT_CUDA(cudaMemsetAsync(w.xp, 0, c.N * sizeof(float), c.st), "cold start");
    if (P.b_in) PAT_CUDA(cudaMemcpyAsync(w.bdat, P.b_in, c.D * sizeof(double), cudaMemcpyDeviceToDevice, c.st),
                         "Bregman resume");
    else PAT_CUDA(cudaMemsetAsync(w.bdat, 0, c.D * sizeof(double), c.st), "Bregman init");
    for (int k = 0; k < P.outer; k++) {
        const NvtxRange step("Bregman step");
        data_shift_kernel<<<ew_blocks(c.D), 256, 0, c.st>>>(w.gdat, f, w.bdat, c.D);
        PAT_CUDA(cudaGetLastError(), "data launch");
        FistaOut fo;
        if ((st = fista(c, P, eta, &fo)) != PAT_OK) return st;
        rep.inner_total += fo.iterations;
        rep.restarts += fo.restarts;
        rep.energy = fo.energy;
        bregman_update_kernel<<<ew_blocks(c.D), 256, 0, c.st>>>(w.bdat, f, w.axp, c.D);
        PAT_CUDA(cudaGetLastError(), "Bregman launch");
        // data residual ||C A p^{k+1} - f|| (FP64)
        double res2 = 0.0;
        RedArgs q = {};
        q.op = RED_SUMSQ_DIFF_FF;
        q.a = w.axp;
        q.b = f;
        q.n = c.D;
        if ((st = reduce(c, &q, 1, &res2)) != PAT_OK) return st;
        const double res = sqrt(res2);
        if (k < 64) rep.residual[k] = res;
        rep.n_residual = std::min(k + 1, 64);
    }
    PAT_CUDA(cudaMemcpyAsync(p_out, w.xp, c.N * sizeof(float), cudaMemcpyDeviceToDevice, c.st), "solution copy");
    if (P.b_out)
        PAT_CUDA(cudaMemcpyAsync(P.b_out, w.bdat, c.D * sizeof(double), cudaMemcpyDeviceToDevice, c.st),
                 "Bregman state copy");
    if (report) *report = rep;
    // a time-step kernel whose bounded wait for a bulk copy gave up makes every result since then
    // undefined; the solve has synchronised anyway, so it reads (and clears) the record itself
    return pat_device_status(G, stream);
}
