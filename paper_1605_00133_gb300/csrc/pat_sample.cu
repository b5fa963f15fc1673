// pat_sample.cu - sampling operator C and its transpose per time point (Sec. 3.1, Sec. 4.3):
// rSP row selection (gather) and zero-filled scatter; scrambled-Hadamard patterns through a
// register/shared-memory fast Walsh-Hadamard transform, one CTA per recorded plane.
#include <math.h>

#include "pat_kargs.h"

namespace pat {

#define PAT_TRY(x)                            \
    do {                                      \
        cudaError_t _e = (x);                 \
        if (_e != cudaSuccess) return _e;     \
    } while (0)

// ---------------------------------------------------------------------------------------------
// sampling kernels (Sec. 3.1 / Sec. 4.3)
// ---------------------------------------------------------------------------------------------

// One plane per blockIdx.x, kRspChunk measurements per blockIdx.y: no index division, and the index list
// is read by consecutive threads.  Bound by the random 4-byte reads of the planes.
constexpr int kRspChunk = 2048;
__global__ void __launch_bounds__(256) rsp_gather_kernel(const float* __restrict__ rec, float* __restrict__ f,
                                                         const int32_t* __restrict__ idx, int m, int M) {
    const float* src = rec + (size_t)blockIdx.x * M;
    float* dst = f + (size_t)blockIdx.x * m;
    for (int j0 = blockIdx.y * kRspChunk; j0 < m; j0 += gridDim.y * kRspChunk) {
        const int j1 = min(m, j0 + kRspChunk);
#pragma unroll 8
        for (int j = j0 + threadIdx.x; j < j1; j += 256) dst[j] = src[__ldg(idx + j)];
    }
}

// The zero-filled scatter written as a gather over plane points, so every plane is written once, in
// order: inv[l] is the measurement at point l, or -1.
__global__ void __launch_bounds__(256) rsp_scatter_kernel(const float* __restrict__ f, float* __restrict__ rec,
                                                          const int32_t* __restrict__ inv, int m, int M) {
    const float* src = f + (size_t)blockIdx.x * m;
    float* dst = rec + (size_t)blockIdx.x * M;
    for (int l0 = blockIdx.y * kRspChunk; l0 < M; l0 += gridDim.y * kRspChunk) {
        const int l1 = min(M, l0 + kRspChunk);
#pragma unroll 8
        for (int l = l0 + threadIdx.x; l < l1; l += 256) {
            const int j = __ldg(inv + l);
            dst[l] = j >= 0 ? src[j] : 0.f;
        }
    }
}

// Unnormalised Walsh-Hadamard transform (Sylvester order) of one plane of M = 2^LOGM points by one CTA.
// A thread holds VPT values and does up to log2(VPT) of the butterfly sweeps h = 1, 2, 4, ... in
// registers between two exchanges through shared memory, so a 16384-point plane takes 3 register passes
// and 2 exchanges instead of 14 sweeps over shared memory with a barrier each (the sweeps and their
// order, so the rounding, are the same).  The scramble is a gather in (or scatter into) a plane in
// shared memory, so global memory is read and written in order.  400 planes of 16384 points: 69 ->
// 21 us (forward), 77 -> 19 us (transpose); what is left is shared-memory throughput (about 5000
// wavefronts a plane, the random accesses of the scramble among them).
template <int LOGM>
struct WH {
    static constexpr int M = 1 << LOGM;
    static constexpr int LV = (LOGM >= 10) ? 5 : LOGM - 5;  // log2 of the values per thread
    static constexpr int VPT = 1 << LV;
    static constexpr int NT = M / VPT;                      // 32 .. 1024 threads
    static constexpr int NPASS = (LOGM + LV - 1) / LV;
    static constexpr int MINB = (NT >= 1024) ? 1 : (NT >= 512) ? 2 : 4;
    // sweeps of pass p: bits [p LV, p LV + width(p))
    __host__ __device__ static constexpr int width(int p) { return (p + 1) * LV <= LOGM ? LV : LOGM - p * LV; }
};
// Shared-memory word of element l.  A thread of pass 0 owns consecutive elements and one of a later
// pass elements 2^s apart; the flip of the low five bits by the next five keeps a warp's accesses of
// both kinds in different banks.
__device__ __forceinline__ int wh_word(int l) { return l ^ ((l >> 5) & 31); }
// element i of group g of pass P: bits [s, s + w) are i, the others count threads, then groups
template <int LOGM, int P>
__device__ __forceinline__ int wh_elem(int g, int i) {
    constexpr int s = P * WH<LOGM>::LV, w = WH<LOGM>::width(P);
    const int r = threadIdx.x + WH<LOGM>::NT * g;
    return (r & ((1 << s) - 1)) | (i << s) | ((r >> s) << (s + w));
}
// the sweeps of pass P on v[group][element] (groups of 2^w values)
template <int LOGM, int P>
__device__ __forceinline__ void wh_sweeps(float* v) {
    constexpr int w = WH<LOGM>::width(P), VPT = WH<LOGM>::VPT;
#pragma unroll
    for (int h = 1; h < (1 << w); h <<= 1)
#pragma unroll
        for (int i = 0; i < VPT; i++)
            if (!(i & h)) {
                const float x = v[i], y = v[i + h];
                v[i] = x + y;
                v[i + h] = x - y;
            }
}
// passes P .. NPASS-1 on v (pass P's layout on entry, the last pass's on exit) through sm
template <int LOGM, int P>
__device__ __forceinline__ void wh_passes(float* v, float* sm) {
    using W = WH<LOGM>;
    wh_sweeps<LOGM, P>(v);
    if constexpr (P + 1 < W::NPASS) {
        constexpr int w = W::width(P), w2 = W::width(P + 1);
        __syncthreads();  // whatever was read from sm before
#pragma unroll
        for (int i = 0; i < W::VPT; i++) sm[wh_word(wh_elem<LOGM, P>(i >> w, i & ((1 << w) - 1)))] = v[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < W::VPT; i++) v[i] = sm[wh_word(wh_elem<LOGM, P + 1>(i >> w2, i & ((1 << w2) - 1)))];
        wh_passes<LOGM, P + 1>(v, sm);
    }
}

// one CTA per plane (batch entry, time step): scramble, transform, select rows.  permt: the scramble of
// the thread's pass-0 elements, two to a word: perm[thread * VPT + i] at 2 (i/2 * NT + thread) + i%2
template <int LOGM>
__global__ void __launch_bounds__(WH<LOGM>::NT, WH<LOGM>::MINB)
    shd_forward_kernel(const float* __restrict__ rec, float* __restrict__ f, const uint16_t* __restrict__ permt,
                       const int32_t* __restrict__ rows, int m, int pm1, float inv_sqrt_m, int vec) {
    using W = WH<LOGM>;
    extern __shared__ float4 smem_raw[];
    float* sm = reinterpret_cast<float*>(smem_raw);
    const size_t p = blockIdx.x;
    const float* src = rec + p * W::M;
    if (vec) {
        for (int l = threadIdx.x; l < W::M / 4; l += W::NT) smem_raw[l] = __ldcs(reinterpret_cast<const float4*>(src) + l);
    } else {
        for (int l = threadIdx.x; l < W::M; l += W::NT) sm[l] = src[l];
    }
    // the scramble's indices are fetched while the plane is in flight, two to a register
    uint32_t at[W::VPT / 2];
#pragma unroll
    for (int i = 0; i < W::VPT / 2; i++)
        at[i] = __ldg(reinterpret_cast<const uint32_t*>(permt) + i * W::NT + threadIdx.x);
    __syncthreads();
    float v[W::VPT];
#pragma unroll
    for (int i = 0; i < W::VPT; i++) v[i] = sm[(at[i / 2] >> (16 * (i & 1))) & 0xffff];
    wh_passes<LOGM, 0>(v, sm);
    constexpr int P = W::NPASS - 1, w = W::width(P);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < W::VPT; i++) sm[wh_word(wh_elem<LOGM, P>(i >> w, i & ((1 << w) - 1)))] = v[i];
    __syncthreads();
    const float w0 = sm[0];
    for (int j = threadIdx.x; j < m; j += W::NT) {
        const float t = sm[wh_word(__ldg(rows + j))];
        f[p * m + j] = pm1 ? t * inv_sqrt_m : 0.5f * (w0 + t);
    }
}

template <int LOGM>
__global__ void __launch_bounds__(WH<LOGM>::NT, WH<LOGM>::MINB)
    shd_adjoint_kernel(const float* __restrict__ f, float* __restrict__ rec, const int32_t* __restrict__ perm,
                       const int32_t* __restrict__ rows, int m, int pm1, float inv_sqrt_m, int vec) {
    using W = WH<LOGM>;
    extern __shared__ float4 smem_raw[];
    float* sm = reinterpret_cast<float*>(smem_raw);
    __shared__ float red[32];
    const size_t p = blockIdx.x;
    for (int l = threadIdx.x; l < W::M / 4; l += W::NT) smem_raw[l] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    // scatter the data, and sum them (the constant half of the 0/1 patterns) as 1024 strided partial
    // sums and a tree over them, whatever the number of threads
    for (int t0 = 0; t0 < 1024; t0 += W::NT) {
        float sum = 0.f;
        for (int j = t0 + threadIdx.x; j < m; j += 1024) {
            const float y = f[p * m + j];
            sm[wh_word(__ldg(rows + j))] = y;
            sum += y;
        }
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if ((threadIdx.x & 31) == 0) red[(t0 + threadIdx.x) >> 5] = sum;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        float t = red[threadIdx.x];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) red[0] = t;
    }
    float v[W::VPT];
    constexpr int w0 = W::width(0);
#pragma unroll
    for (int i = 0; i < W::VPT; i++) v[i] = sm[wh_word(wh_elem<LOGM, 0>(i >> w0, i & ((1 << w0) - 1)))];
    wh_passes<LOGM, 0>(v, sm);
    constexpr int P = W::NPASS - 1, w = W::width(P);
    __syncthreads();
    const float total = red[0];
#pragma unroll
    for (int i = 0; i < W::VPT; i++)
        sm[__ldg(perm + wh_elem<LOGM, P>(i >> w, i & ((1 << w) - 1)))] =
            pm1 ? v[i] * inv_sqrt_m : 0.5f * (total + v[i]);
    __syncthreads();
    float* dst = rec + p * W::M;
    if (vec) {
        for (int l = threadIdx.x; l < W::M / 4; l += W::NT) reinterpret_cast<float4*>(dst)[l] = smem_raw[l];
    } else {
        for (int l = threadIdx.x; l < W::M; l += W::NT) dst[l] = sm[l];
    }
}

struct ShdKernels {
    decltype(&shd_forward_kernel<10>) fwd = nullptr;
    decltype(&shd_adjoint_kernel<10>) adj = nullptr;
    int nt = 0;
};
template <int LOGM>
static ShdKernels make_shd() {
    ShdKernels k;
    k.fwd = shd_forward_kernel<LOGM>;
    k.adj = shd_adjoint_kernel<LOGM>;
    k.nt = WH<LOGM>::NT;
    return k;
}
static ShdKernels shd_kernels_for(int M) {  // planes of 8 x 8 up to the limit of pat_create_grid
    switch (M) {
        case 64: return make_shd<6>();
        case 128: return make_shd<7>();
        case 256: return make_shd<8>();
        case 512: return make_shd<9>();
        case 1024: return make_shd<10>();
        case 2048: return make_shd<11>();
        case 4096: return make_shd<12>();
        case 8192: return make_shd<13>();
        case 16384: return make_shd<14>();
        case 32768: return make_shd<15>();
        default: return ShdKernels{};
    }
}
int shd_threads(int M) { return shd_kernels_for(M).nt; }

// adjoint with T = 1: p = 0 except the detection plane, which takes the injected plane
__global__ void inject_plane_kernel(const float* __restrict__ inj, float* __restrict__ p, Geom g) {
    const long long total = (long long)g.B * g.nreal;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const long long b = i / g.nreal;
        const long long v = i - b * g.nreal;
        const long long z = v / g.m_plane;
        p[i] = (z == g.sensor_z) ? inj[b * (long long)g.T * g.m_plane + (v - z * g.m_plane)] : 0.f;
    }
}

static dim3 rsp_grid(long long planes, int n) {
    const int chunks = (n + kRspChunk - 1) / kRspChunk;
    return dim3((unsigned)planes, (unsigned)(chunks < 32 ? chunks : 32));
}

static int aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

cudaError_t run_sample(const Geom& g, const Workspace& w, int kind, int m, const float* pbar,
                       float* f, int nt, cudaStream_t st) {
    const long long planes = (long long)g.B * nt;
    if (kind == PAT_SAMPLE_FULL) {
        return cudaMemcpyAsync(f, pbar, sizeof(float) * planes * g.m_plane, cudaMemcpyDeviceToDevice, st);
    }
    if (kind == PAT_SAMPLE_POINTS) {
        if (planes * m == 0) return cudaSuccess;
        rsp_gather_kernel<<<rsp_grid(planes, m), 256, 0, st>>>(pbar, f, w.idx, m, g.m_plane);
        return cudaGetLastError();
    }
    const ShdKernels k = shd_kernels_for(g.m_plane);
    if (!k.fwd) return cudaErrorInvalidValue;
    k.fwd<<<(unsigned)planes, k.nt, g.m_plane * sizeof(float), st>>>(
        pbar, f, w.permt, w.rows, m, kind == PAT_SAMPLE_HADAMARDPM, (float)(1.0 / sqrt((double)g.m_plane)),
        aligned16(pbar));
    return cudaGetLastError();
}

cudaError_t run_sample_adjoint(const Geom& g, const Workspace& w, int kind, int m, const float* f,
                               float* pbar, int nt, cudaStream_t st) {
    const long long planes = (long long)g.B * nt;
    if (kind == PAT_SAMPLE_FULL) {
        return cudaMemcpyAsync(pbar, f, sizeof(float) * planes * g.m_plane, cudaMemcpyDeviceToDevice, st);
    }
    if (kind == PAT_SAMPLE_POINTS) {
        rsp_scatter_kernel<<<rsp_grid(planes, g.m_plane), 256, 0, st>>>(f, pbar, w.inv, m, g.m_plane);
        return cudaGetLastError();
    }
    const ShdKernels k = shd_kernels_for(g.m_plane);
    if (!k.adj) return cudaErrorInvalidValue;
    k.adj<<<(unsigned)planes, k.nt, g.m_plane * sizeof(float), st>>>(
        f, pbar, w.perm, w.rows, m, kind == PAT_SAMPLE_HADAMARDPM, (float)(1.0 / sqrt((double)g.m_plane)),
        aligned16(pbar));
    return cudaGetLastError();
}

cudaError_t configure_sampling(const Geom& g, int kind) {
    const size_t shd_bytes = (size_t)g.m_plane * sizeof(float);
    if ((kind != PAT_SAMPLE_HADAMARD01 && kind != PAT_SAMPLE_HADAMARDPM) || shd_bytes <= 48 * 1024) return cudaSuccess;
    const ShdKernels k = shd_kernels_for(g.m_plane);
    if (!k.fwd) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(k.fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shd_bytes);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k.adj, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shd_bytes);
}

cudaError_t run_inject_only(const Geom& g, const float* inj, float* p, cudaStream_t st) {
    const long long total = (long long)g.B * g.nreal;
    const int blocks = (int)((total + 255) / 256 < 152 * 32 ? (total + 255) / 256 : 152 * 32);
    inject_plane_kernel<<<blocks, 256, 0, st>>>(inj, p, g);
    return cudaGetLastError();
}

}  // namespace pat
