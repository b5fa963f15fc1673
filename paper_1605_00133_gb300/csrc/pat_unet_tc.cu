// pat_unet_tc.cu - 3x3x3 convolution of the learned warm start on the fifth-generation tensor cores
// (tcgen05): BF16 operands staged by the TMA unit, FP32 accumulators in tensor memory.
//
// Implicit GEMM, D[m][n] = sum_k A[m][k] B[n][k] with M = voxels, N = output channels, K = 27 taps x
// input channels, accumulated in the order taps, then channels by 16 (whatever the kernel and its tiles: the
// result of a layer does not depend on them).  What bounds it, measured:
//   the MMA, M = 128, K = 16: 46 cycles for N <= 32, 49 at 64, 65 at 128, 129 at 256 -- if the issuing warp
//     is converged (elect_one);
//   the TMA unit: one box row (one voxel's channels, up to 64 bytes; 128 bytes in 1.2 cycles) per cycle and
//     SM, whatever the row's width: so a row of 48 (or 96, ...) channels is fetched as one (two) rows of 64
//     channels, the missing ones zero-filled, not in 16-channel pieces.
// conv3_ring_kernel (few channels, large volumes) fetches every line a few times and serves three taps with one
// MMA; conv3_tc_kernel serves every other shape, one shifted box per tap.
// conv3_tc_kernel: a CTA owns one tile of M = 128 voxels, a bx x by x bz box of the volume (x fastest), and
// BN output channels.  One K step is one tap and CK input channels:
//   A: the voxel box shifted by the tap, loaded by a 4D tensor map over (channel, x, y, z); parts of
//      the box outside the volume come back as zeros, which is the convolution's zero padding;
//   B: the tap's weights w[t][n0 .. n0+BN)[c0 .. c0+CK), a 3D tensor map over (cin, cout, tap).
// Both land K-major in shared memory, CK BF16 per row with the swizzle of that row width (32, 64 or
// 128 bytes), the layout the MMA's shared-memory descriptors read.  Warp roles (192 threads):
//   warp 0   one thread issues the TMA copies of a ring of stages (full/empty mbarriers);
//   warp 1   allocates the tensor-memory accumulator (128 lanes x BN FP32 columns) and issues tcgen05.mma
//            (M = 128, N = BN, K = 16 per instruction), committing each stage's MMAs to that stage's
//            empty barrier and the last to the done barrier;
//   warps 2-5 the epilogue: tcgen05.ld of the accumulator rows (warp w reads lanes 32 (w % 4) ..),
//            optional ReLU or mask, BF16 rounding, one voxel row per thread to global memory.
// Launch overlap: all kernels here, and the layers between them, are launched with programmatic stream
// serialisation, so that a CTA sets up its barriers and tensor memory while the grid before it drains; every thread
// then waits for that grid before touching global memory.  A pass is some 77 launches of 5 .. 115 us:
// forward and backward at 64x128x128 voxels 1454 -> 1328 us, a gradient and its sum at 32x64x64 20.7 -> 15.7.
// Every mbarrier wait is bounded.  A wait that gives up records bit 0 of a device word (read and
// cleared by pat_unet_device_status), and the CTA stops issuing work, waits (bounded) for the copies
// it issued, frees its tensor memory and exits; its outputs are then invalid.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <climits>
#include <mutex>
#include <type_traits>

#include "pat_fft.cuh"

namespace pat {

__device__ int g_unet_err;  // bit 0: a tensor-core convolution gave up waiting (outputs invalid)

namespace {

constexpr int kNStage = 4;
constexpr int kBM = 128;
constexpr int kThreads = 192;
constexpr int kPolls = 1 << 20;  // bounded waits: each poll suspends for at most about a microsecond

// test hook of the kernels' failure paths (pat_unet_debug_copy_fault): process-wide
int g_stop_after = -1;
int g_polls = kPolls;
struct CopyFault {
    int stop_after;  // the producer issues only stages (of conv3_ring_kernel: input planes) < stop_after (< 0: all)
    int polls;       // poll limit of the waits for what the hook leaves out
    // ON: whether the kernel reads the hook.  The ring and the gradient by lines have a form that does not: limits that
    // vary cost them up to 5 % (16 -> 16 channels at 64x128x128 30.7 -> 32.1 us).
    template <bool ON = true>
    __device__ __forceinline__ bool out(int s) const {
        return ON && stop_after >= 0 && s >= stop_after;
    }
    template <bool ON = true>
    __device__ __forceinline__ int limit(int s) const {
        return out<ON>(s) ? polls : kPolls;
    }
};

struct ConvTcArgs {
    __nv_bfloat16* y;
    const __nv_bfloat16* mask;  // NULL: none
    int ldm;
    int ldy, cin, cout, bn;
    int D, H, W;
    int bx, by, bz;     // voxel box of a tile
    int tx, ty;         // tiles along x and y
    int relu;
    uint32_t tmem_cols;
    CopyFault fault;
};

// shared-memory matrix descriptor of a K-major operand tile: rows of `row_bytes` (= the swizzle
// width: 32, 64 or 128 bytes), 8-row groups `8 * row_bytes` apart (stride byte offset); the leading
// byte offset is unused for swizzled K-major tiles; descriptor version 1; layout type 6 / 4 / 2 for
// the 32 / 64 / 128-byte swizzle
__device__ __forceinline__ uint64_t kmajor_desc(uint32_t saddr, uint32_t row_bytes) {
    const uint64_t layout = (row_bytes == 128) ? 2 : (row_bytes == 64) ? 4 : 6;
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(((8 * row_bytes) >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    d |= layout << 61;
    return d;
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major, M = 128, N = n
__device__ __forceinline__ uint32_t mma_idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
}

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_addr(bar))
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int c0, int c1, int c2,
                                            unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::
            "r"(smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_addr(bar))
        : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// One lane of a converged warp.  The MMA warp runs its loop with all lanes, and only this lane issues: the
// descriptors are then warp-uniform values.  Issued from inside a one-lane branch an instruction took
// about 145 cycles (operands moved to uniform registers one by one behind their own arithmetic), three
// times what the MMA itself takes at N = 48.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
// a descriptor's low word (address field; the descriptors below differ in nothing else within a kernel) and
// high word are passed separately
__device__ __forceinline__ uint32_t lo32(uint64_t d) { return (uint32_t)d; }
__device__ __forceinline__ uint32_t hi32(uint64_t d) { return (uint32_t)(d >> 32); }
__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint32_t alo, uint32_t ahi, uint32_t blo, uint32_t bhi,
                                       uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tmov.b64 da, {%1, %2};\n\tmov.b64 db, {%3, %4};\n\t"
        "setp.ne.b32 p, %6, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}" ::"r"(tmem_d),
        "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(acc)
        : "memory");
}
// the same from one lane of a converged warp without a branch around it, for loops that are not unrolled
__device__ __forceinline__ void tc_mma_if(bool issue, uint32_t tmem_d, uint32_t alo, uint32_t ahi, uint32_t blo,
                                          uint32_t bhi, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\tmov.b64 da, {%1, %2};\n\tmov.b64 db, {%3, %4};\n\t"
        "setp.ne.b32 p, %6, 0;\n\tsetp.ne.b32 q, %7, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}" ::"r"(tmem_d),
        "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(acc), "r"((uint32_t)issue)
        : "memory");
}
// arrive on `bar` once every tcgen05 operation this thread issued before has completed
__device__ __forceinline__ void tc_commit(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
                 : "memory");
}

// 16 consecutive FP32 columns of this thread's tensor-memory lane
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float* v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
        "[%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = __uint_as_float(r[i]);
}

// the same of two groups of columns, in flight together
__device__ __forceinline__ void tc_ld16x2(uint32_t ta, uint32_t tb, float* v, float* u) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
        "[%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, "
        "%31}, [%33];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(ta), "r"(tb));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; i++) {
        v[i] = __uint_as_float(r[i]);
        u[i] = __uint_as_float(r[16 + i]);
    }
}

// zeros into 16 consecutive FP32 columns of this thread's tensor-memory lane (tc_wait_st() before they are relied on)
__device__ __forceinline__ void tc_zero16(uint32_t taddr) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(
            taddr),
        "r"(0u)
        : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Rounds 16 channels of a voxel to BF16 and stores them.  With a mask (the activation a gradient is taken
// through) channels where it is not positive are stored as zero.
__device__ __forceinline__ void conv_store16(const float* v, int relu, const __nv_bfloat16* mask, __nv_bfloat16* out) {
    uint4 pk[2], mk[2];
    uint32_t* w32 = reinterpret_cast<uint32_t*>(pk);
    if (mask) {
        mk[0] = reinterpret_cast<const uint4*>(mask)[0];
        mk[1] = reinterpret_cast<const uint4*>(mask)[1];
    }
    const __nv_bfloat162* m2 = reinterpret_cast<const __nv_bfloat162*>(mk);
#pragma unroll
    for (int i = 0; i < 8; i++) {
        float p = v[2 * i], q = v[2 * i + 1];
        if (relu) {
            p = fmaxf(p, 0.f);
            q = fmaxf(q, 0.f);
        }
        if (mask) {
            const float2 mv = __bfloat1622float2(m2[i]);
            p = mv.x > 0.f ? p : 0.f;
            q = mv.y > 0.f ? q : 0.f;
        }
        const __nv_bfloat162 h = __floats2bfloat162_rn(p, q);
        w32[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    uint4* dst = reinterpret_cast<uint4*>(out);
    dst[0] = pk[0];
    dst[1] = pk[1];
}

template <int CK>
__global__ void __launch_bounds__(kThreads, 1) conv3_tc_kernel(const __grid_constant__ CUtensorMap tmx,
                                                                const __grid_constant__ CUtensorMap tmw,
                                                                ConvTcArgs a) {
    extern __shared__ uint8_t smem_raw[];
    // 1024-byte alignment of every operand tile (the 128-byte swizzle repeats every 1024 bytes)
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    constexpr uint32_t RB = CK * 2;            // bytes per operand row = swizzle width
    constexpr uint32_t A_BYTES = kBM * RB;     // 4, 8 or 16 KB: a multiple of 1024
    const uint32_t b_bytes = (uint32_t)a.bn * RB;
    const uint32_t stage_bytes = (A_BYTES + b_bytes + 1023) & ~1023u;
    constexpr int nstage = kNStage;
    unsigned long long* full = reinterpret_cast<unsigned long long*>(smem + nstage * stage_bytes);
    unsigned long long* empty = full + nstage;
    unsigned long long* done = empty + nstage;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    int* counts = reinterpret_cast<int*>(tmem_slot + 1);  // [0] stages issued, [1] consumed, [2] failed

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tile = blockIdx.x;
    const int x0 = (tile % a.tx) * a.bx;
    const int y0 = ((tile / a.tx) % a.ty) * a.by;
    const int z0 = (tile / (a.tx * a.ty)) * a.bz;
    const int n0 = blockIdx.y * a.bn;
    const int nc = (a.cin + CK - 1) / CK;
    const int S = 27 * nc;
    // bytes a stage's two copies deliver: the voxel box (at most 128 rows; rows of the tile beyond it
    // are never stored) and the weight tile
    const uint32_t tx_bytes = RB * (uint32_t)(a.bx * a.by * a.bz) + b_bytes;

    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"(a.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < nstage; s++) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, 1);
        }
        mbar_init(done, 1);
        mbar_fence_init();
        counts[0] = counts[1] = counts[2] = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();
    pdl_trigger();  // now that this CTA has its tensor memory: the next grid's cannot take it first

    if (warp == 0 && lane == 0) {
        // producer
        int s = 0, st = 0, c0 = 0, t = 0, dx = -1, dy = -1, dz = -1;
        uint32_t phase = 1;  // a fresh empty barrier's preceding phase counts as complete
        for (; s < S; s++) {
            if (a.fault.out(s)) break;  // test hook: nothing more is issued
            if (!mbar_wait(empty + st, phase, kPolls)) {
                counts[2] = 1;
                break;
            }
            uint8_t* sa = smem + st * stage_bytes;
            mbar_arrive_expect_tx(full + st, tx_bytes);
            tma_load_4d(sa, &tmx, c0, x0 + dx, y0 + dy, z0 + dz, full + st);
            tma_load_3d(sa + A_BYTES, &tmw, c0, n0, t, full + st);
            if ((c0 += CK) >= a.cin) {
                c0 = 0;
                t++;
                if (++dx > 1) {
                    dx = -1;
                    if (++dy > 1) {
                        dy = -1;
                        dz++;
                    }
                }
            }
            if (++st == nstage) {
                st = 0;
                phase ^= 1;
            }
        }
        counts[0] = s;
    } else if (warp == 1) {
        // MMA issuer (all lanes run the loop, one issues)
        const bool leader = elect_one();
        const uint32_t idesc = mma_idesc(a.bn);
        const uint64_t d0 = kmajor_desc(smem_addr(smem), RB);
        const uint32_t hi = hi32(d0), lo0 = lo32(d0), stage16 = stage_bytes >> 4;
        int s = 0, st = 0, c0 = 0;
        uint32_t phase = 0, lo = lo0;
        for (; s < S; s++) {
            if (!__all_sync(0xffffffffu, mbar_wait(full + st, phase, a.fault.limit(s)))) {
                if (leader) counts[2] = 1;
                break;
            }
            tc_fence_after();
            if (leader) {
#pragma unroll
                for (int k = 0; k < CK / 16; k++)  // 32 bytes along K; channels past cin are zeros, left out
                    if (c0 + 16 * k < a.cin)
                        tc_mma(tmem, lo + 2 * k, hi, lo + A_BYTES / 16 + 2 * k, hi, idesc, (s > 0 || k > 0) ? 1u : 0u);
                tc_commit(empty + st);
            }
            __syncwarp();
            if ((c0 += CK) >= a.cin) c0 = 0;
            lo += stage16;
            if (++st == nstage) {
                st = 0;
                phase ^= 1;
                lo = lo0;
            }
        }
        if (leader) {
            counts[1] = s;
            tc_commit(done);
        }
    } else if (warp >= 2) {
        // epilogue
        const bool ok = mbar_wait(done, 0, kPolls);
        if (!ok) counts[2] = 1;
        __syncwarp();  // the tensor-memory loads below are warp-wide
        tc_fence_after();
        const int m = 32 * (warp & 3) + lane;  // tensor-memory lane = tile row
        const uint32_t trow = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
        const int xx = m % a.bx, yy = (m / a.bx) % a.by, zz = m / (a.bx * a.by);
        const int x = x0 + xx, y = y0 + yy, z = z0 + zz;
        const bool valid = ok && m < a.bx * a.by * a.bz && x < a.W && y < a.H && z < a.D;
        const size_t vox = ((size_t)z * a.H + y) * a.W + x;  // used only where valid
        __nv_bfloat16* out = a.y + vox * a.ldy + n0;
        const __nv_bfloat16* mask = a.mask + vox * a.ldm + n0;
        for (int c = 0; c < a.bn; c += 16) {
            float v[16];
            tc_ld16(trow + (uint32_t)c, v);  // every thread of the warp takes part
            if (valid) conv_store16(v, a.relu, a.mask ? mask + c : nullptr, out + c);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (counts[2]) {
        if (threadIdx.x == 0) {
            atomicOr(&g_unet_err, 1);
            // copies issued but never consumed may still be in flight: let them land (bounded)
            for (int s = counts[1]; s < counts[0]; s++) mbar_wait(full + s % nstage, (s / nstage) & 1, kPolls);
            mbar_wait(done, 0, kPolls);
        }
        __syncthreads();
    }
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.tmem_cols) : "memory");
    }
}

// ---------------------------------------------------------------------------------------------
// The same convolution for few channels on large volumes (lines up to 128 voxels, weights that fit shared
// memory): a persistent kernel.  A CTA keeps its weights in shared memory and walks along z through a
// column of one M tile (by lines of W voxels), with a ring of input planes of by + 2 lines; steps
// (column, z) are numbered column by column and each CTA takes an equal contiguous range.  A tap's operand
// is 128 rows of a plane from another start: dy lines and dx voxels on.
//   Lines over 64 voxels (by = 1): a plane's lines are W + 2 voxels (x = -1 .. W), in parts of 16 channels
//     (32-byte rows), up to four; the operand starts dy (W + 2) + dx rows on.  The 32-byte swizzle is applied
//     to shared-memory address bits by the TMA unit and the tensor core alike, so any row may be the first.
//   Shorter lines (16 or 32 channels): every plane is held three times, shifted by dx, its lines bx voxels (W
//     rounded up to 8), so that operands start at multiples of 8 rows and by lines fill the 128 rows.
// A plane enters three outputs, z + 1, z and z - 1, through the taps dz = -1, 0, 1.  Their accumulators lie side by
// side in a ring of tensor-memory columns, and the three dz of a (dy, dx) in the weights, so one MMA of 3 bn columns
// serves all three: 9 MMAs a plane of 16 channels instead of 27 of a third the width, which take no less (see
// above).  An output still sums its taps in order: all of plane z - 1, then z, then z + 1.  Since one instruction
// covers outputs that begin and outputs that go on, the epilogue leaves zeros in the accumulators it has read.
// The epilogue is two groups of four warps taking alternate outputs.  64x128x128 voxels, one box per tap and MMAs
// issued from one lane -> 27 MMAs -> 9 MMAs: 16 -> 16 channels 137 -> 50 -> 30 us, 48 -> 16 371 -> 114 -> 59, 16 -> 48
// 379 -> 54 -> 44.  What bounds it now: per plane about 60 cycles an MMA and 350 of waits and issue (16 -> 16; the TMA
// unit alone takes 21 us), the MMAs (48 -> 16), the epilogue's stores (16 -> 48: 37 us without).
// Other shapes use the kernel above: longer lines, more channels (weights and planes do not fit, and its K
// steps are bound less by the TMA unit), and volumes of less than four tiles an SM (the weights would be
// fetched for too little work).
// ---------------------------------------------------------------------------------------------

constexpr int kRingThreads = 320;  // producer, MMA issuer, 2 x 4 epilogue warps
constexpr int kMaxPlanes = 8, kMaxAcc = 16;

struct ConvRingArgs {
    __nv_bfloat16* y;
    const __nv_bfloat16* mask;  // NULL: none
    int ldm;
    int ldy, cin, bn;
    int D, H, W;
    int pitch, by, lines;     // rows from line to line; a tile is by lines, a plane of the ring by + 2
    int ncopies;              // copies of a plane shifted by dx (1: the lines have a halo), from x = -1
    int steps_per_cta, steps; // (column, z) steps
    int relu;
    int nplanes, nacc;        // ring of input planes, of accumulators (bn columns each)
    uint32_t box_bytes;       // one part of one copy of a plane
    uint32_t dxstep;          // from tap dx to dx + 1, in 16-byte units: a copy or a row
    CopyFault fault;
};

template <int CK, int NP, bool FAULT>  // NP parts of CK input channels; FAULT: with the test hook
__global__ void __launch_bounds__(kRingThreads, 1)
    conv3_ring_kernel(const __grid_constant__ CUtensorMap tmx, const __grid_constant__ CUtensorMap tmw, ConvRingArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    __shared__ unsigned long long pfull[kMaxPlanes], pempty[kMaxPlanes], tfull[kMaxAcc], tempty[kMaxAcc], wfull, done;
    __shared__ uint32_t tmem_slot;
    __shared__ int failed;
    constexpr uint32_t RB = CK * 2;  // bytes per operand row = swizzle width
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t plane_bytes = a.ncopies * NP * a.box_bytes;
    uint8_t* planes = smem;
    uint8_t* wts = smem + a.nplanes * plane_bytes;
    const int n0 = blockIdx.y * a.bn;
    const int u0 = blockIdx.x * a.steps_per_cta, u1 = min(a.steps, u0 + a.steps_per_cta);

    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_slot)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int i = 0; i < a.nplanes; i++) {
            mbar_init(pfull + i, 1);
            mbar_init(pempty + i, 1);
        }
        for (int i = 0; i < a.nacc; i++) {
            mbar_init(tfull + i, 1);
            mbar_init(tempty + i, 4);  // one arrival per epilogue warp
        }
        mbar_init(&wfull, 1);
        mbar_init(&done, 1);
        mbar_fence_init();
        failed = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    pdl_wait();
    pdl_trigger();  // now that this CTA has its tensor memory: the next grid's cannot take it first

    if (warp == 0 && lane == 0) {
        // producer: the weights, then the planes z-1 .. z+1 of every step in order, each once per run of z
        mbar_arrive_expect_tx(&wfull, 27u * NP * a.bn * RB);
        // the weights of (dy, dx): those of dz = 1, 0, -1 behind one another
        for (int q = 0; q < NP; q++)
            for (int t = 0; t < 27; t++)
                tma_load_3d(wts + ((q * 9 + t % 9) * 3 + 2 - t / 9) * a.bn * RB, &tmw, q * CK, n0, t, &wfull);
        const uint32_t tx_bytes = (uint32_t)(a.ncopies * NP * a.pitch * a.lines) * RB;
        int p = 0, slot = 0;
        uint32_t phase = 1;  // a fresh empty barrier's preceding phase counts as complete
        bool ok = true;
        for (int u = u0; u < u1 && ok && !a.fault.out<FAULT>(p);) {
            const int col = u / a.D, z0 = u - col * a.D, n = min(u1 - u, a.D - z0);
            for (int z = z0 - 1; z <= z0 + n && !a.fault.out<FAULT>(p); z++, p++) {
                if (!mbar_wait(pempty + slot, phase, kPolls)) {
                    ok = false;
                    break;
                }
                uint8_t* d = planes + slot * plane_bytes;
                mbar_arrive_expect_tx(pfull + slot, tx_bytes);
                for (int k = 0; k < a.ncopies; k++)
                    for (int q = 0; q < NP; q++, d += a.box_bytes)
                        tma_load_4d(d, &tmx, q * CK, k - 1, col * a.by - 1, z, pfull + slot);
                if (++slot == a.nplanes) {
                    slot = 0;
                    phase ^= 1;
                }
            }
            u += n;
        }
        if (!ok) atomicOr(&failed, 1);
        // let every copy issued land before this CTA's shared memory can go to another (bounded)
        mbar_wait(&wfull, 0, kPolls);
        for (int k = max(0, p - a.nplanes); k < p; k++) mbar_wait(pfull + k % a.nplanes, (k / a.nplanes) & 1, kPolls);
    } else if (warp == 1) {
        // MMA issuer (all lanes run the loop, one issues)
        const bool leader = elect_one();
        const uint64_t da = kmajor_desc(smem_addr(planes), RB), db = kmajor_desc(smem_addr(wts), RB);
        const uint32_t hi = hi32(da);
        // address steps in 16-byte units: a plane, a part, dx, a line, one tap's weights, a part's
        const uint32_t pstep = plane_bytes >> 4, qstep = a.box_bytes >> 4, dxstep = a.dxstep;
        const uint32_t lstep = a.pitch * (RB / 16), wstep = a.bn * (RB / 16), wqstep = 27 * wstep;
        // the nine (dy, dx) of the plane at x for n outputs, from accumulator acc and weight block b on
        auto plane_mmas = [&](uint32_t x0, int acc, int b, int n) {
            const uint32_t td = tmem + acc * a.bn, idesc = mma_idesc(n * a.bn), w0 = lo32(db) + b * wstep;
#pragma unroll
            for (int r = 0; r < 9; r++) {
                const uint32_t x = x0 + (r % 3) * dxstep + (r / 3) * lstep, w = w0 + r * 3 * wstep;
#pragma unroll
                for (int q = 0; q < NP; q++) {
                    tc_mma(td, x + q * qstep, hi, w + q * wqstep, hi, idesc, 1u);
                    if (CK == 32) tc_mma(td, x + 2, hi, w + 2, hi, idesc, 1u);
                }
            }
        };
        bool ok = mbar_wait(&wfull, 0, kPolls);
        int slot = 0, acc = 0;  // ring slots of the plane and of its first output
        int p = 0;              // planes so far
        uint32_t pphase = 0, acc_phase = 0;
        int fresh = 0;          // accumulator of the next output to begin
        for (int u = u0; u < u1 && ok;) {
            const int col = u / a.D, z0 = u - col * a.D, n = min(u1 - u, a.D - z0);
            for (int i = -1; i <= n; i++, p++) {
                // plane z0 + i: outputs i - 1 .. i + 1 of this run, of which i + 1 begins and i - 1 is complete
                const int lo = max(i - 1, 0), cnt = min(i + 1, n - 1) - lo + 1;
                ok = mbar_wait(pfull + slot, pphase, a.fault.limit<FAULT>(p));
                if (i + 1 < n) {
                    ok = ok && mbar_wait(tempty + fresh, acc_phase, kPolls);
                    if (++fresh == a.nacc) {
                        fresh = 0;
                        acc_phase ^= 1;
                    }
                }
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                const uint32_t x0 = lo32(da) + slot * pstep;
                const int b = lo - (i - 1), c1 = min(cnt, a.nacc - acc);  // accumulators before the ring wraps
                if (leader) {
                    plane_mmas(x0, acc, b, c1);
                    if (c1 < cnt) plane_mmas(x0, 0, b + c1, cnt - c1);
                    tc_commit(pempty + slot);
                    if (i > 0) tc_commit(tfull + acc);
                }
                __syncwarp();
                if (i > 0 && ++acc == a.nacc) acc = 0;
                if (++slot == a.nplanes) {
                    slot = 0;
                    pphase ^= 1;
                }
            }
            u += n;
        }
        if (leader) {
            if (!ok) atomicOr(&failed, 1);
            tc_commit(&done);
        }
        __syncwarp();
        mbar_wait(&done, 0, kPolls);  // every MMA has finished before the tensor memory is freed
    } else if (warp >= 2) {
        const int grp = (warp - 2) >> 2, m = 32 * (warp & 3) + lane;
        const uint32_t trow = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
        const int xx = m % a.pitch, yy = m / a.pitch;
        int acc = 0, turn = 0, col = u0 / a.D, z = u0 - col * a.D;
        int last = 2;  // the plane that completes the output
        uint32_t acc_phase = 0;
        bool ok = true;
        // every accumulator starts from zero (an instruction covers one that begins and two that go on)
        auto give = [&](int i) {
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(tempty + i)) : "memory");
        };
        for (int i = grp; i < a.nacc; i += 2) {
            for (int c = 0; c < a.bn; c += 16) tc_zero16(trow + i * a.bn + c);
            give(i);
        }
        for (int u = u0; u < u1 && ok; u++) {
            if (turn == grp) {
                ok = __all_sync(0xffffffffu, mbar_wait(tfull + acc, acc_phase, a.fault.limit<FAULT>(last)));
                tc_fence_after();
                const int y = col * a.by + yy;
                const bool valid = ok && yy < a.by && xx < a.W && y < a.H;
                const size_t vox = ((size_t)z * a.H + y) * a.W + xx;  // used only where valid
                __nv_bfloat16* out = a.y + vox * a.ldy + n0;
                const __nv_bfloat16* mask = a.mask + vox * a.ldm + n0;
                const uint32_t td = trow + acc * a.bn;
                for (int c = 0; c < a.bn; c += 16) {
                    float v[16];
                    tc_ld16(td + c, v);
                    tc_zero16(td + c);
                    if (c + 16 >= a.bn) give(acc);  // the accumulator is in registers
                    if (valid) conv_store16(v, a.relu, a.mask ? mask + c : nullptr, out + c);
                }
            }
            turn ^= 1;
            last++;
            if (++z == a.D) {
                z = 0;
                col++;
                last += 2;
            }
            if (++acc == a.nacc) {
                acc = 0;
                acc_phase ^= 1;
            }
        }
        if (!ok) atomicOr(&failed, 1);
    }
    tc_fence_before();
    __syncthreads();
    if (failed && threadIdx.x == 0) atomicOr(&g_unet_err, 1);
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// ---------------------------------------------------------------------------------------------
// Weight gradient, general form: dW[t][co][ci] = sum_v dY[v][co] X[v + off_t][ci]
// = sum_u dY[u - dx][co] X[u + (dz,dy)][ci], all 27 taps in one GEMM: M = (dz, dy) x input channels, N = dx x
// output channels, K = voxels, split
// over chunks of voxel blocks with a fixed-order sum afterwards.  With the tap's shift shared between
// the operands a block is fetched as 9 shifted boxes of X and 3 of dY, where 27 shifted boxes of X (and dY
// once per M tile) took 27 box rows a voxel of the TMA unit's one per cycle (see the file comment).
// A K block is a box of 64 voxels.  Both operands arrive channel-contiguous, i.e. MN-major: a
// swizzle atom is 8 voxel rows x WA channels of one (dz, dy) (A) or 8 voxel rows x WB output channels of
// one dx (B), WA, WB in {16, 32, 64}, zero-filled past cin; an M tile's 128 rows are 128 / WA atoms side by
// side (one TMA box each, zero outside the volume), the N columns 3 BN / WB atoms.  In a descriptor the
// leading byte offset steps from one atom to the next along M or N, the stride byte offset from one
// 8-row group of voxels to the next.  A CTA accumulates several M tiles (as many as fit the tensor
// memory with their N columns and three stages of shared memory), so one fetch of a block serves them all.
// The boxes of a stage are issued by the lanes of the producer warp together, each its own (coordinates and
// destinations are fixed per lane but for the block).
// Accuracy: one accumulator sums a CTA's share of the voxels, truncating, so the error grows with the volume: 64 -> 64
// and 192 -> 64 channels at 16x32x32 voxels 1.9e-7 and 5.0e-7 with ReLU'd operands, 64 -> 64 at 64x128x128 3.4e-5.
// ---------------------------------------------------------------------------------------------

constexpr int kKB = 64;  // voxels per K block

struct WgradArgs {
    float4* partial;    // [chunk][M tile][4 columns of 3 cout][128 rows]
    int cin, cout, bn, wa, wb;
    int mtiles, mt;     // M tiles in all, per CTA
    int D, H, W;
    int bx, by, bz, tx, ty, nkb;   // voxel box of a K block, blocks along x and y, blocks in all
    int kb_per_cta;
    int nstage;
    uint32_t tmem_cols;
    CopyFault fault;
};

// MN-major descriptor: atoms of 8 rows x `row_bytes`, `lbo` bytes apart along M/N, 8-row groups
// 8 * row_bytes apart along K
__device__ __forceinline__ uint64_t mnmajor_desc(uint32_t saddr, uint32_t row_bytes, uint32_t lbo) {
    const uint64_t layout = (row_bytes == 128) ? 2 : (row_bytes == 64) ? 4 : 6;
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)(((8 * row_bytes) >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    d |= layout << 61;
    return d;
}

// this thread's row of an accumulator, N columns four at a time: a warp writes 512 bytes in a row
__device__ __forceinline__ void wgrad_store(uint32_t taddr, int N, float4* out) {
    for (int c = 0; c < N; c += 16) {
        float v[16];
        tc_ld16(taddr + (uint32_t)c, v);
#pragma unroll
        for (int i = 0; i < 4; i++)
            out[(size_t)(c / 4 + i) * kBM] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
}

__global__ void __launch_bounds__(kThreads, 1) wgrad_tc_kernel(const __grid_constant__ CUtensorMap tmx,
                                                               const __grid_constant__ CUtensorMap tmd,
                                                               WgradArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t ra = 2u * a.wa, rb = 2u * a.wb;       // row bytes = swizzle widths
    const uint32_t atom_a = kKB * ra, atom_b = kKB * rb; // one atom column over the K block
    constexpr uint32_t tile_bytes = kBM * kKB * 2;       // one M tile: 16 KB
    const uint32_t a_bytes = a.mt * tile_bytes;
    const int N = 3 * a.bn;
    const int ncols = (N + 31) & ~31;                    // tensor-memory columns of an M tile
    const uint32_t b_bytes = (uint32_t)N * kKB * 2;
    const uint32_t stage_bytes = (a_bytes + b_bytes + 1023) & ~1023u;
    const int nstage = a.nstage;
    unsigned long long* full = reinterpret_cast<unsigned long long*>(smem + nstage * stage_bytes);
    unsigned long long* empty = full + nstage;
    unsigned long long* done = empty + nstage;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    int* counts = reinterpret_cast<int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int mgroups = (a.mtiles + a.mt - 1) / a.mt;
    const int mtile0 = (blockIdx.x % mgroups) * a.mt, ng = blockIdx.x / mgroups;  // M tiles, output channels
    const int mt = min(a.mt, a.mtiles - mtile0);
    const int chunk = blockIdx.y;
    const int kb0 = chunk * a.kb_per_cta;
    const int nkb = min(a.kb_per_cta, a.nkb - kb0);
    const int per_tile = kBM / a.wa;                 // atoms (dz dy, channel block) of an M tile
    const int cblocks = (a.cin + a.wa - 1) / a.wa;
    const int atom0 = mtile0 * per_tile;
    const int na = min(mt * per_tile, 9 * cblocks - atom0);  // atoms of this CTA that exist
    const int nbb = a.bn / a.wb;                     // atoms per dx
    const int nbox = na + 3 * nbb;
    const uint32_t tx_bytes = (uint32_t)na * atom_a + b_bytes;

    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"(a.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < nstage; s++) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, 1);
        }
        mbar_init(done, 1);
        mbar_fence_init();
        counts[0] = counts[1] = counts[2] = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();
    pdl_trigger();  // now that this CTA has its tensor memory: the next grid's cannot take it first

    if (warp == 0) {
        // this lane's box of every stage (nbox <= 32, checked by the launch)
        const CUtensorMap* map = &tmx;
        int c0 = 0, dx = 0, dy = 0, dz = 0;
        uint32_t dst = 0;
        if (lane < na) {
            const int atom = atom0 + lane, row = atom / cblocks;
            c0 = (atom - row * cblocks) * a.wa;
            dy = row % 3 - 1;
            dz = row / 3 - 1;
            dst = lane * atom_a;
        } else {
            const int e = lane - na, d = e / nbb;
            map = &tmd;
            c0 = ng * a.bn + (e - d * nbb) * a.wb;
            dx = 1 - d;  // tap dx = d - 1 reads dY at u - dx
            dst = a_bytes + e * atom_b;
        }
        int tx = kb0 % a.tx, ty = (kb0 / a.tx) % a.ty, tz = kb0 / (a.tx * a.ty);
        int s = 0, st = 0;
        uint32_t phase = 1;  // a fresh empty barrier's preceding phase counts as complete
        for (; s < nkb && !a.fault.out(s); s++) {
            if (!__all_sync(0xffffffffu, mbar_wait(empty + st, phase, kPolls))) {
                if (lane == 0) counts[2] = 1;
                break;
            }
            if (lane == 0) mbar_arrive_expect_tx(full + st, tx_bytes);
            __syncwarp();
            if (lane < nbox)
                tma_load_4d(smem + st * stage_bytes + dst, map, c0, tx * a.bx + dx, ty * a.by + dy, tz * a.bz + dz,
                            full + st);
            if (++tx == a.tx) {
                tx = 0;
                if (++ty == a.ty) {
                    ty = 0;
                    tz++;
                }
            }
            if (++st == nstage) {
                st = 0;
                phase ^= 1;
            }
        }
        if (lane == 0) counts[0] = s;
    } else if (warp == 1) {
        // A and B MN-major (bits 15, 16), FP32 accumulator, BF16 operands, M = 128; all lanes run the loop,
        // one issues
        const bool leader = elect_one();
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                               ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
        const uint64_t ad = mnmajor_desc(smem_addr(smem), ra, atom_a);
        const uint64_t bd = mnmajor_desc(smem_addr(smem) + a_bytes, rb, atom_b);
        const uint32_t ahi = hi32(ad), bhi = hi32(bd), stage16 = stage_bytes >> 4, tile16 = tile_bytes >> 4;
        int s = 0, st = 0;
        uint32_t phase = 0, off = 0;
        for (; s < nkb; s++) {
            if (!__all_sync(0xffffffffu, mbar_wait(full + st, phase, a.fault.limit(s)))) {
                if (leader) counts[2] = 1;
                break;
            }
            tc_fence_after();
            if (leader) {
                // 16 voxel rows = two 8-row groups: the start moves by 16 rows of each operand
                const uint32_t blo = lo32(bd) + off;
                uint32_t alo = lo32(ad) + off, td = tmem;
                const uint32_t on = s > 0 ? 1u : 0u;
                for (int t = 0; t < mt; t++, alo += tile16, td += ncols) {
#pragma unroll
                    for (int k = 0; k < kKB / 16; k++)
                        tc_mma(td, alo + k * ra, ahi, blo + k * rb, bhi, idesc, k ? 1u : on);
                }
                tc_commit(empty + st);
            }
            __syncwarp();
            off += stage16;
            if (++st == nstage) {
                st = 0;
                phase ^= 1;
                off = 0;
            }
        }
        if (leader) {
            counts[1] = s;
            tc_commit(done);
        }
    } else if (warp >= 2) {
        const bool ok = mbar_wait(done, 0, kPolls);
        if (!ok) counts[2] = 1;
        __syncwarp();
        tc_fence_after();
        const int m = 32 * (warp & 3) + lane;
        const uint32_t trow = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
        for (int t = 0; t < mt; t++) {
            float4* out = a.partial + (((size_t)chunk * a.mtiles + mtile0 + t) * (3 * a.cout / 4) + ng * N / 4) * kBM + m;
            wgrad_store(trow + (uint32_t)(t * ncols), N, out);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (counts[2]) {
        if (threadIdx.x == 0) {
            atomicOr(&g_unet_err, 1);
            for (int s = counts[1]; s < counts[0]; s++) mbar_wait(full + s % nstage, (s / nstage) & 1, kPolls);
            mbar_wait(done, 0, kPolls);
        }
        __syncthreads();
    }
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.tmem_cols) : "memory");
    }
}

// The same product for few channels: lines along x are fetched once for the three dy.  A K block is R lines of bx
// voxels (bx = 16 .. 64).  Of X a stage holds R + 2 lines y0 - 1 .., each as 3 dz x channel blocks atoms of bx voxel
// rows x WA channels (one box of a tensor map with y outermost): the atoms (dy, dz, block) of line r follow each other
// from atom 3 r blocks on, so the M rows of a tap are there under one leading byte offset, whatever dy.
// Of dY it holds R lines of bx + 2 voxels; the three dx are operand starts one voxel row apart (leading byte
// offset = one row, column block j being dx = 1 - j).  The TMA unit fetches 3 blocks (R + 2) / R + (bx + 2) / bx box
// rows a voxel instead of 9 blocks + 3.  An M group that needs two of the three dy fetches R + 1 lines.
// Rows of the last M tile beyond the 9 blocks atoms multiply whatever follows in shared memory and are not used.
// What bounds it: the MMAs with few channels (two M tiles of N = 48 for 16 -> 16: 49 cycles each), the TMA unit with
// more.  The whole gradient took with wgrad_tc_kernel (its partial products written 16 bytes a lane, 192 or more apart) ->
// now: 64x128x128 voxels 16 -> 16 channels 69.9 -> 31 us, 48 -> 16 145 -> 62; 32x64x64 voxels 32 -> 32 31.5 -> 16,
// 96 -> 32 49.5 -> 27.
// Accuracy: the tensor core truncates as it adds, so a sum of n voxels of one sign comes out low by about 1.3e-9 n of
// its value (7168 voxels 9.1e-6, 14144 2.0e-5).  So K blocks go to two accumulators in turn where tensor memory holds
// two, and after kChain voxels in each, or at the end, the epilogue adds them up, rounding to nearest, and to what
// earlier segments left in the partial product.  Relative error against FP64 with one accumulator to the end, 48
// channels in two groups of tiles -> now: ReLU'd normal numbers at 64x128x128 voxels 16 -> 16 channels 9.1e-6 -> 3.8e-6,
// 48 -> 16 2.0e-5 -> 8.9e-6; at 32x64x64 16 -> 32 9.5e-7 -> 4.1e-7; at 128x256x256 16 -> 16 1.0e-4 -> 9e-6 (200 -> 218 us).
// In the network at 64x128x128, whose operands are large in few places (eight of them): d1a (48 -> 16) 1.0e-5 .. 4.6e-5
// -> 5.6e-6 .. 2.1e-5, d1b 5e-6 .. 2.4e-5 -> 2.6e-6 .. 1.1e-5, e1a 7e-6 -> 3.6e-6, the others below 4e-6.
constexpr int kChain = 7424;  // most voxels summed by one accumulator: 464 MMAs

struct WlineArgs {
    float4* partial;    // as above; rows in the order (dy, dz, channel), columns (1 - dx, output channel)
    int cb, wa, bn;     // channel blocks, their channels; output channels
    int mtiles, mt;     // M tiles in all, per CTA
    int bx, R, lines;   // voxels per line, lines of a block, lines of X fetched for it
    int tx, ty, nkb;    // blocks along x and y, in all
    int kb_per_cta;
    int nset, seg;      // accumulators (1 or 2) taking K blocks in turn; K blocks after which they are added up
    int nstage;
    uint32_t stage_bytes, x_bytes, bar_off;
    uint32_t tmem_cols;
    CopyFault fault;
};

__device__ __forceinline__ void tma_load_5d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, int c4,
                                            unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], "
        "[%7];" ::"r"(smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_addr(bar))
        : "memory");
}

// wgrad_store of the sum of nset <= 2 accumulators set_cols columns apart, N a multiple of 48.  more: added to what is
// there (this thread's own, of the segment before), 12 loads in flight.
__device__ __forceinline__ void wgrad_store_sum(uint32_t taddr, int nset, int set_cols, int N, bool more, float4* out) {
    for (int c0 = 0; c0 < N; c0 += 48) {
        float4* p = out + (size_t)(c0 / 4) * kBM;
        float4 o[12];
        if (more) {
#pragma unroll
            for (int i = 0; i < 12; i++) o[i] = p[i * kBM];
        }
#pragma unroll
        for (int h = 0; h < 3; h++) {
            float v[16];
            if (nset > 1) {
                float u[16];
                tc_ld16x2(taddr + (uint32_t)(c0 + 16 * h), taddr + (uint32_t)(set_cols + c0 + 16 * h), v, u);
#pragma unroll
                for (int i = 0; i < 16; i++) v[i] += u[i];
            } else {
                tc_ld16(taddr + (uint32_t)(c0 + 16 * h), v);
            }
#pragma unroll
            for (int i = 0; i < 4; i++) {
                float4 t = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                if (more) {
                    const float4 w = o[4 * h + i];
                    t = make_float4(w.x + t.x, w.y + t.y, w.z + t.z, w.w + t.w);
                }
                p[(4 * h + i) * kBM] = t;
            }
        }
    }
}

template <int KS, bool FAULT>  // bx / 16; FAULT: with the test hook
__global__ void __launch_bounds__(kThreads, 1) wgrad_line_kernel(const __grid_constant__ CUtensorMap tmx,
                                                                 const __grid_constant__ CUtensorMap tmd,
                                                                 WlineArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t ra = 2u * a.wa, rb = 2u * a.bn;  // row bytes = swizzle widths
    const uint32_t unit = a.bx * ra;                // one atom
    const int N = 3 * a.bn, ncols = (N + 31) & ~31, set_cols = a.mt * ncols, nstage = a.nstage;
    const uint32_t d_bytes = a.R * (a.bx + 2) * rb;
    unsigned long long* full = reinterpret_cast<unsigned long long*>(smem + a.bar_off);
    unsigned long long* empty = full + nstage;
    unsigned long long* done = empty + nstage;
    unsigned long long* drained = done + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drained + 1);
    int* counts = reinterpret_cast<int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int mtile0 = blockIdx.x * a.mt, mt = min(a.mt, a.mtiles - mtile0);
    const int chunk = blockIdx.y, kb0 = chunk * a.kb_per_cta, nkb = min(a.kb_per_cta, a.nkb - kb0);
    const int atom0 = mtile0 * (kBM / a.wa), dy0 = atom0 / (3 * a.cb);  // first atom and dy of this group

    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"(a.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < nstage; s++) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, 1);
        }
        mbar_init(done, 1);
        mbar_init(drained, 4);  // one arrival per epilogue warp
        mbar_fence_init();
        counts[0] = counts[1] = counts[2] = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();
    pdl_trigger();  // now that this CTA has its tensor memory: the next grid's cannot take it first

    if (warp == 0) {
        if (lane == 0) {
            int tx = kb0 % a.tx, ty = (kb0 / a.tx) % a.ty, z = kb0 / (a.tx * a.ty);
            int s = 0, st = 0;
            uint32_t phase = 1;  // a fresh empty barrier's preceding phase counts as complete
            for (; s < nkb && !a.fault.out<FAULT>(s); s++) {
                if (!mbar_wait(empty + st, phase, kPolls)) {
                    counts[2] = 1;
                    break;
                }
                uint8_t* dst = smem + st * a.stage_bytes;
                mbar_arrive_expect_tx(full + st, (uint32_t)a.lines * 3 * a.cb * unit + d_bytes);
                tma_load_5d(dst, &tmx, 0, tx * a.bx, 0, z - 1, ty * a.R - 1 + dy0, full + st);
                tma_load_4d(dst + a.x_bytes, &tmd, 0, tx * a.bx - 1, ty * a.R, z, full + st);
                if (++tx == a.tx) {
                    tx = 0;
                    if (++ty == a.ty) {
                        ty = 0;
                        z++;
                    }
                }
                if (++st == nstage) {
                    st = 0;
                    phase ^= 1;
                }
            }
            counts[0] = s;
        }
    } else if (warp == 1) {
        // A and B MN-major (bits 15, 16), FP32 accumulator, BF16 operands, M = 128; all lanes run the loop,
        // one issues
        const bool leader = elect_one();
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                               ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
        const uint64_t ad = mnmajor_desc(smem_addr(smem) + (atom0 - 3 * a.cb * dy0) * unit, ra, unit);
        const uint64_t bd = mnmajor_desc(smem_addr(smem) + a.x_bytes, rb, rb);
        const uint32_t ahi = hi32(ad), bhi = hi32(bd), stage16 = a.stage_bytes >> 4;
        const uint32_t tile16 = (kBM / a.wa) * unit >> 4, aline16 = 3 * a.cb * unit >> 4, bline16 = (a.bx + 2) * rb >> 4;
        int s = 0, st = 0, segment = 0;
        uint32_t phase = 0, off = 0;
        for (bool ok = true; ok && s < nkb; segment++) {
            // accumulators handed back by the epilogue of the segment before
            if (segment > 0) ok = __all_sync(0xffffffffu, mbar_wait(drained, (segment - 1) & 1, kPolls));
            const int end = min(nkb, s + a.seg);
            for (int i = 0; ok && s < end; i++, s++) {
                ok = __all_sync(0xffffffffu, mbar_wait(full + st, phase, a.fault.limit<FAULT>(s)));
                if (!ok) break;
                tc_fence_after();
                uint32_t al = lo32(ad) + off, td = tmem + ((i & (a.nset - 1)) ? set_cols : 0);
                const uint32_t bl = lo32(bd) + off;
                for (int t = 0; t < mt; t++, al += tile16, td += ncols) {
                    uint32_t alo = al, blo = bl, on = i >= a.nset ? 1u : 0u;
                    for (int r = 0; r < a.R; r++, alo += aline16, blo += bline16) {
                        // 16 voxel rows: the starts move by 16 rows of each operand
#pragma unroll
                        for (int k = 0; k < KS; k++)
                            tc_mma_if(leader, td, alo + k * ra, ahi, blo + k * rb, bhi, idesc, k ? 1u : on);
                        on = 1u;
                    }
                }
                if (leader) tc_commit(empty + st);
                __syncwarp();
                off += stage16;
                if (++st == nstage) {
                    st = 0;
                    phase ^= 1;
                    off = 0;
                }
            }
            if (leader) {
                if (!ok) counts[2] = 1;
                counts[1] = s;
                tc_commit(done);
            }
        }
        __syncwarp();
        mbar_wait(done, (segment - 1) & 1, kPolls);  // every MMA has finished before the tensor memory is freed
    } else if (warp >= 2) {
        // epilogue: adds up the accumulators of each segment once it is done, and hands them back
        const uint32_t trow = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
        float4* out = a.partial + ((size_t)chunk * a.mtiles + mtile0) * (N / 4) * kBM + 32 * (warp & 3) + lane;
        for (int j = 0; j * a.seg < nkb; j++) {
            bool ok = mbar_wait(done, j & 1, kPolls);
            if (!ok) counts[2] = 1;
            ok = ok && !*const_cast<volatile int*>(counts + 2);  // set before `done` if the issuer gave up
            if (!__all_sync(0xffffffffu, ok)) break;
            tc_fence_after();
            const int ns = min(a.nset, min(a.seg, nkb - j * a.seg));
            for (int t = 0; t < mt; t++)
                if (ns > 1 || j > 0)
                    wgrad_store_sum(trow + t * ncols, ns, set_cols, N, j > 0, out + (size_t)t * (N / 4) * kBM);
                else
                    wgrad_store(trow + t * ncols, N, out + (size_t)t * (N / 4) * kBM);
            tc_fence_before();
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(drained)) : "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    if (counts[2]) {
        if (threadIdx.x == 0) {
            atomicOr(&g_unet_err, 1);
            for (int s = counts[1]; s < counts[0]; s++) mbar_wait(full + s % nstage, (s / nstage) & 1, kPolls);
        }
        __syncthreads();
    }
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.tmem_cols) : "memory");
    }
}

// dw[tap][co][ci] = sum over chunks of the partial products.  A row is (dz, dy, ci), its dz and dy the other way
// round if `lines`; a column is (co / bn, dx, co % bn), its dx descending if `lines`.  A warp takes 32
// consecutive rows of four columns, 512 bytes a chunk, and S warps share the chunks (a serial loop over 152
// chunks is a chain of memory latencies); their parts are added in a fixed order.  Gradient and sum of 64 -> 64
// channels at 16x32x32 voxels: 26.8 -> 17.2 us with this layout of the partial products, 192 -> 64 33.0 -> 22.7.
template <int S>
__global__ void __launch_bounds__(32 * S) wgrad_sum_kernel(const float4* __restrict__ partial, int nchunk, int mtiles,
                                                           int cin, int cout, int bn, int wa, int lines,
                                                           float* __restrict__ dw) {
    __shared__ float4 sh[S][32];
    const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
    const int c4 = blockIdx.x, m = blockIdx.y * 32 + lane, n4 = 3 * cout / 4;
    pdl_wait();
    pdl_trigger();
    const float4* p = partial + ((size_t)(m / kBM) * n4 + c4) * kBM + m % kBM;
    const size_t cs = (size_t)mtiles * n4 * kBM;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 10
    for (int c = sl; c < nchunk; c += S) {
        const float4 v = __ldcg(p + c * cs);
        s.x += v.x;
        s.y += v.y;
        s.z += v.z;
        s.w += v.w;
    }
    sh[sl][lane] = s;
    __syncthreads();
    if (sl >= 4) return;
    // warp i: column i of the four
    const int cblocks = (cin + wa - 1) / wa, atom = m / wa, row = atom / cblocks;
    const int ci = (atom - row * cblocks) * wa + m % wa;
    if (row >= 9 || ci >= cin) return;  // rows past the product, zero-filled channels
    const int tap_row = lines ? (row % 3) * 3 + row / 3 : row;
    const float* q = &reinterpret_cast<const float*>(&sh[0][lane])[sl];
    float t = q[0];
#pragma unroll
    for (int k = 1; k < S; k++) t += q[k * 128];
    const int c = 4 * c4 + sl, g = c / (3 * bn), r = c - g * 3 * bn, j = r / bn, d = lines ? 2 - j : j;
    dw[((size_t)(3 * tap_row + d) * cout + g * bn + r - j * bn) * cin + ci] = t;
}

// A kernel's cap on dynamic shared memory is one for all host threads: always set to the most any shape takes (all of an
// SM's but for what the kernel declares itself), so that no thread lowers it between another's call and its launch.
constexpr size_t kSmemCap = 227 * 1024, kRingSmemCap = 226 * 1024;
template <typename... P>
cudaError_t raise_smem(void (*kernel)(P...), size_t cap, size_t smem) {
    if (smem > cap) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cap);
}

template <typename... P, typename... A>
cudaError_t launch(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A... args) {
    const cudaError_t e = launch_pdl(kernel, grid, threads, smem, st, args...);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

typedef CUresult (*EncodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encoder() {
    static std::once_flag once;
    static EncodeTiled fn = nullptr;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiled>(p);
    });
    // a map is encoded in the thread's current context, which a thread that has none yet gets here (also under capture)
    thread_local bool bound = false;
    int device;
    if (!bound) bound = cudaGetDevice(&device) == cudaSuccess && cudaSetDevice(device) == cudaSuccess;
    return fn;
}

template <int CK>
cudaError_t launch_ck(const CUtensorMap& mx, const CUtensorMap& mw, const ConvTcArgs& a, unsigned tiles,
                      cudaStream_t st) {
    const uint32_t stage = (kBM * CK * 2 + a.bn * CK * 2 + 1023) & ~1023u;
    size_t smem = 1024 + kNStage * (size_t)stage + (2 * kNStage + 1) * 8 + 4 + 16;
    // at most 512 / tmem_cols CTAs on an SM, so that every CTA's tensor-memory allocation succeeds at
    // once: request enough shared memory (228 KB per SM, 1 KB reserved per CTA) to keep out one more
    const size_t max_ctas = 512 / a.tmem_cols;
    const size_t floor_smem = 233472 / (max_ctas + 1) + 1;
    if (smem < floor_smem) smem = floor_smem;
    cudaError_t e = raise_smem(conv3_tc_kernel<CK>, kSmemCap, smem);
    if (e != cudaSuccess) return e;
    return launch(conv3_tc_kernel<CK>, dim3(tiles, (unsigned)(a.cout / a.bn)), kThreads, smem, st, mx, mw, a);
}

}  // namespace

// a K-major operand map: channels c of a (channel, x, y, z) or (cin, cout, tap) tensor in boxes of ck of them
static CUresult kmajor_map(CUtensorMap* m, int rank, const void* p, const cuuint64_t* dims, const cuuint64_t* strides,
                           const cuuint32_t* box) {
    const cuuint32_t es[4] = {1, 1, 1, 1};
    const CUtensorMapSwizzle swz = box[0] == 64   ? CU_TENSOR_MAP_SWIZZLE_128B
                                   : box[0] == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
                                                  : CU_TENSOR_MAP_SWIZZLE_32B;
    return encoder()(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(p), dims, strides, box, es,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

// Geometry of conv3_ring_kernel; ctas = 0 where the other kernel serves the shape.
struct RingGeom {
    ConvRingArgs a;
    int ctas, groups, ck;  // ck: channels of a part
    size_t smem;
};
static RingGeom ring_geom(int cin, int cout, int D, int H, int W) {
    RingGeom g = {};
    ConvRingArgs& a = g.a;
    const bool halo = W > 64;
    if (W > kBM || cin > (halo ? 64 : 32)) return g;
    a.cin = cin;
    a.D = D;
    a.H = H;
    a.W = W;
    g.ck = halo ? 16 : cin;
    a.pitch = halo ? W + 2 : (W + 7) & ~7;
    a.by = halo ? 1 : std::min(H, kBM / a.pitch);
    a.lines = a.by + 2;
    a.ncopies = halo ? 1 : 3;
    a.box_bytes = (uint32_t)(a.lines * a.pitch * g.ck * 2 + 1023) & ~1023u;
    a.dxstep = halo ? (uint32_t)g.ck / 8 : a.box_bytes >> 4;
    const size_t plane = (size_t)a.ncopies * (cin / g.ck) * a.box_bytes;
    // the largest share of the output channels whose weights fit beside three planes; an operand reads up to
    // 128 rows past its box: 8 KB of pad follow the weights
    constexpr size_t kRoom = 227 * 1024 - 1024 - 1024 - 8192;
    for (int n = 1; n <= 8 && !a.bn; n++)
        if (cout % (16 * n) == 0 && 3 * (cout / n) <= 256 && (size_t)27 * (cout / n) * cin * 2 + 3 * plane <= kRoom) {
            g.groups = n;
            a.bn = cout / n;
        }
    if (!a.bn) return g;
    const size_t wbytes = (size_t)27 * a.bn * cin * 2;
    const int ytiles = (H + a.by - 1) / a.by, sms = 152 / g.groups;
    a.steps = ytiles * D;
    if ((long long)ytiles * D < 4LL * sms) return g;
    a.steps_per_cta = (a.steps + sms - 1) / sms;
    a.nacc = std::min(kMaxAcc, 512 / a.bn);
    a.nplanes = (int)std::min<size_t>(kMaxPlanes, (kRoom - wbytes) / plane);
    g.ctas = (a.steps + a.steps_per_cta - 1) / a.steps_per_cta;
    g.smem = 1024 + a.nplanes * plane + wbytes + 8192;
    // one CTA per SM (it holds all of the tensor memory): more than half of the shared memory
    g.smem = std::max(g.smem, (size_t)(120 * 1024));
    return g;
}

static cudaError_t launch_ring(RingGeom& g, const void* x, int ldx, const void* w, int cout, cudaStream_t st) {
    const ConvRingArgs& a = g.a;
    alignas(64) CUtensorMap mx, mw;
    const cuuint64_t xd[4] = {(cuuint64_t)a.cin, (cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)a.D};
    const cuuint64_t xs[3] = {(cuuint64_t)ldx * 2, (cuuint64_t)ldx * 2 * a.W, (cuuint64_t)ldx * 2 * a.W * a.H};
    const cuuint32_t xb[4] = {(cuuint32_t)g.ck, (cuuint32_t)a.pitch, (cuuint32_t)a.lines, 1};
    const cuuint64_t wd[3] = {(cuuint64_t)a.cin, (cuuint64_t)cout, 27};
    const cuuint64_t ws[2] = {(cuuint64_t)a.cin * 2, (cuuint64_t)a.cin * 2 * cout};
    const cuuint32_t wb[3] = {(cuuint32_t)g.ck, (cuuint32_t)a.bn, 1};
    if (kmajor_map(&mx, 4, x, xd, xs, xb) != CUDA_SUCCESS || kmajor_map(&mw, 3, w, wd, ws, wb) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    const int np = a.cin / g.ck;
    const auto pick = [&](auto fault) {
        constexpr bool F = decltype(fault)::value;
        return g.ck == 32 ? conv3_ring_kernel<32, 1, F>
               : np == 1  ? conv3_ring_kernel<16, 1, F>
               : np == 2  ? conv3_ring_kernel<16, 2, F>
               : np == 3  ? conv3_ring_kernel<16, 3, F>
                          : conv3_ring_kernel<16, 4, F>;
    };
    const auto kernel = a.fault.stop_after < 0 ? pick(std::false_type()) : pick(std::true_type());
    cudaError_t e = raise_smem(kernel, kRingSmemCap, g.smem);
    if (e != cudaSuccess) return e;
    return launch(kernel, dim3((unsigned)g.ctas, (unsigned)g.groups), kRingThreads, g.smem, st, mx, mw, a);
}

// y[v][n] = act(sum_t sum_c x[v + off_t][c] w[t][n][c]) on the tensor cores (see the file comment).
// Channel counts multiples of 16, strides multiples of 16 elements, pointers 16-byte aligned (checked
// by the caller).
cudaError_t conv3_tc(const void* x, int ldx, int cin, const void* w, int cout, void* y, int ldy, int D, int H,
                     int W, int relu, const void* mask, int ldm, cudaStream_t st) {
    EncodeTiled enc = encoder();
    if (!enc) return cudaErrorNotSupported;
    RingGeom ring = ring_geom(cin, cout, D, H, W);
    if (ring.ctas > 0) {
        ring.a.y = reinterpret_cast<__nv_bfloat16*>(y);
        ring.a.ldy = ldy;
        ring.a.relu = relu;
        ring.a.mask = reinterpret_cast<const __nv_bfloat16*>(mask);
        ring.a.ldm = ldm;
        ring.a.fault = {g_stop_after, g_polls};
        return launch_ring(ring, x, ldx, w, cout, st);
    }
    ConvTcArgs a = {};
    a.y = reinterpret_cast<__nv_bfloat16*>(y);
    a.ldy = ldy;
    a.cin = cin;
    a.cout = cout;
    // output channels per CTA: the largest divisor up to 128, so that a tile's voxels are fetched for as many
    // channels as fit; fewer while all CTAs still have an SM of their own.  Beyond that the same voxels are fetched
    // twice by an SM: 128 tiles (16x32x32 voxels) with halves 192 -> 64 channels 23.8, 128 -> 32 20.7, 64 -> 64 10.4
    // us, without 18.2, 12.7, 8.3; 72 tiles 64 -> 64 7.8 and 8.1
    for (int n = 1; !a.bn; n++)
        if (cout % (16 * n) == 0 && cout / n <= 128) a.bn = cout / n;
    a.D = D;
    a.H = H;
    a.W = W;
    a.bx = W < kBM ? W : kBM;
    a.by = H < kBM / a.bx ? H : kBM / a.bx;
    a.bz = kBM / (a.bx * a.by);
    a.tx = (W + a.bx - 1) / a.bx;
    a.ty = (H + a.by - 1) / a.by;
    const long long tz = (D + a.bz - 1) / a.bz;
    const long long tiles = (long long)a.tx * a.ty * tz;
    if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
    a.relu = relu;
    a.mask = reinterpret_cast<const __nv_bfloat16*>(mask);
    a.ldm = ldm;
    while (a.bn > 16 && 2 * tiles * (cout / a.bn) <= 152 && cout % (a.bn / 2) == 0 && (a.bn / 2) % 16 == 0) a.bn /= 2;
    a.tmem_cols = a.bn <= 32 ? 32 : a.bn <= 64 ? 64 : 128;
    a.fault = {g_stop_after, g_polls};
    // channels per operand row: one row where cin fits in it (16, 32), else pieces of 64, the last one zero-filled past
    // cin.  But 96 and 160 channels in whole pieces of 32, of which more CTAs fit an SM, where more than one has to:
    // 96 -> 32 at 32x64x64 voxels 54.4 us, in pieces of 64 69.2, 160 -> 32 86.6 and 97.5.  With a CTA an SM at most
    // the fewer steps of 64 win: 96 -> 32 at 16x32x32 12.7 us, in pieces of 32 16.1; with 224 channels and more too
    // (32x64x64, 128 outputs: 188 and 192)
    const int ck = cin == 16 ? 16 : cin == 32 || ((cin == 96 || cin == 160) && tiles * (cout / a.bn) > 152) ? 32 : 64;
    alignas(64) CUtensorMap mx, mw;
    const cuuint64_t xd[4] = {(cuuint64_t)cin, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)D};
    const cuuint64_t xs[3] = {(cuuint64_t)ldx * 2, (cuuint64_t)ldx * 2 * W, (cuuint64_t)ldx * 2 * W * H};
    const cuuint32_t xb[4] = {(cuuint32_t)ck, (cuuint32_t)a.bx, (cuuint32_t)a.by, (cuuint32_t)a.bz};
    const cuuint64_t wd[3] = {(cuuint64_t)cin, (cuuint64_t)cout, 27};
    const cuuint64_t ws[2] = {(cuuint64_t)cin * 2, (cuuint64_t)cin * 2 * cout};
    const cuuint32_t wb[3] = {(cuuint32_t)ck, (cuuint32_t)a.bn, 1};
    if (kmajor_map(&mx, 4, x, xd, xs, xb) != CUDA_SUCCESS || kmajor_map(&mw, 3, w, wd, ws, wb) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    if (ck == 64) return launch_ck<64>(mx, mw, a, (unsigned)tiles, st);
    if (ck == 32) return launch_ck<32>(mx, mw, a, (unsigned)tiles, st);
    return launch_ck<16>(mx, mw, a, (unsigned)tiles, st);
}

// Geometry of the weight-gradient GEMM (shared by the scratch-size query and the launch).
struct WgradGeom {
    int wa, wb, bn, bx, by, bz, tx, ty, nkb, mtiles, mt, mgroups, ngroups, nstage, kb_per_cta, nchunk;
    uint32_t tmem_cols;
    size_t smem;
};

static WgradGeom wgrad_geom(int cin, int cout, int D, int H, int W) {
    WgradGeom g;
    g.wa = cin == 16 ? 16 : cin == 32 ? 32 : 64;
    g.bn = 16;  // output channels per CTA, N = 3 bn <= 256
    for (int b : {80, 64, 48, 32})
        if (cout % b == 0) {
            g.bn = b;
            break;
        }
    g.wb = (g.bn % 64 == 0) ? 64 : (g.bn % 32 == 0) ? 32 : 16;
    g.ngroups = cout / g.bn;
    const int atoms = 9 * ((cin + g.wa - 1) / g.wa), N = 3 * g.bn;
    g.mtiles = (atoms * g.wa + kBM - 1) / kBM;
    // M tiles per CTA: as many as the 512 tensor-memory columns and three stages of shared memory hold,
    // spread evenly over the groups
    auto stage_bytes = [&](int mt) { return (size_t)((mt * kBM + N) * kKB * 2 + 1023) & ~(size_t)1023; };
    constexpr size_t kSmem = 227 * 1024 - 1024 - 256;
    const int ncols = (N + 31) & ~31;
    int mt = std::min(g.mtiles, 512 / ncols);
    while (mt > 1 && 3 * stage_bytes(mt) > kSmem) mt--;
    g.mgroups = (g.mtiles + mt - 1) / mt;
    g.mt = (g.mtiles + g.mgroups - 1) / g.mgroups;
    g.mgroups = (g.mtiles + g.mt - 1) / g.mt;
    g.nstage = (int)std::min<size_t>(6, kSmem / stage_bytes(g.mt));
    g.smem = 1024 + g.nstage * stage_bytes(g.mt) + (2 * g.nstage + 1) * 8 + 4 + 16;
    const int cols = g.mt * ncols;
    g.tmem_cols = cols <= 64 ? 64 : cols <= 128 ? 128 : cols <= 256 ? 256 : 512;
    // no more CTAs on an SM than tensor memory serves at once (228 KB per SM, 1 KB reserved per CTA)
    g.smem = std::max(g.smem, (size_t)(233472 / (512 / g.tmem_cols + 1) + 1));
    // a K block is exactly kKB voxels (the MMA reads all its rows): powers of two, the box reaching
    // past the volume where a side is shorter (those voxels read as zeros)
    auto pow2_at_least = [](int v) {
        int p = 1;
        while (p < v) p <<= 1;
        return p;
    };
    g.bx = std::min(kKB, pow2_at_least(W));
    g.by = std::min(kKB / g.bx, pow2_at_least(H));
    g.bz = kKB / (g.bx * g.by);
    g.tx = (W + g.bx - 1) / g.bx;
    g.ty = (H + g.by - 1) / g.by;
    const long long tz = (D + g.bz - 1) / g.bz;
    g.nkb = (int)((long long)g.tx * g.ty * tz);
    // one round of CTAs over the SMs (as many as fit each), at least 4 K blocks each
    const int per_sm = std::max(1, std::min((int)(512 / g.tmem_cols), (int)(233472 / (g.smem + 1024))));
    const long long want = std::max(1LL, 152LL * per_sm / (g.mgroups * g.ngroups));
    long long per = (g.nkb + want - 1) / want;
    if (per < 4) per = 4;
    g.kb_per_cta = (int)per;
    g.nchunk = (g.nkb + g.kb_per_cta - 1) / g.kb_per_cta;
    return g;
}

// Geometry of wgrad_line_kernel; nchunk = 0 where wgrad_tc_kernel serves the shape: output channels that are not one
// atom of dY (16 or 32), whose N columns would have no single leading byte offset, or over 96 input channels, of which
// three stages hold too few lines.
struct WlineGeom {
    int wa, cb, mtiles, mt, mgroups, span, bx, R, tx, ty, nkb, nset, seg, nstage, kb_per_cta, nchunk;
    uint32_t tmem_cols, x_bytes, stage_bytes, bar_off;
    size_t smem;
};

static WlineGeom wline_geom(int cin, int cout, int D, int H, int W) {
    WlineGeom g = {};
    if ((cout != 16 && cout != 32) || cin > 96) return g;
    g.wa = cin % 32 ? 16 : 32;
    g.cb = cin / g.wa;
    const int per_tile = kBM / g.wa, N = 3 * cout, ncols = (N + 31) & ~31;
    g.mtiles = (9 * cin + kBM - 1) / kBM;
    // Up to four M tiles a CTA, so that 48 channels are one group, whose lines are fetched once: 48 -> 16 channels at
    // 64x128x128 62 us, in two groups of two tiles 87 (and the chains of a tile are half as long).
    g.mgroups = (g.mtiles + 3) / 4;
    g.mt = (g.mtiles + g.mgroups - 1) / g.mgroups;
    for (int i = 0; i < g.mgroups; i++) {
        const int a0 = i * g.mt * per_tile, a1 = std::min((i + 1) * g.mt * per_tile, 9 * g.cb) - 1;
        g.span = std::max(g.span, a1 / (3 * g.cb) - a0 / (3 * g.cb));
    }
    // One CTA an SM: all of its tensor memory.  But four tiles take one accumulator each: with two, at no cost, d1a came
    // out at 3e-6 .. 9e-6 in the network, which moved 3 % of the whole gradients by more than 2e-5, the most that results
    // in FP32 may move from one version to the next.
    g.nset = g.mt == 4 ? 1 : std::min(2, 512 / (g.mt * ncols));
    g.tmem_cols = 64;
    while ((int)g.tmem_cols < g.nset * g.mt * ncols) g.tmem_cols *= 2;
    // The block shape with the least time of TMA unit (a box row a cycle) or MMAs, over the volume padded to whole
    // blocks; 200 cycles for what a stage costs besides.  48 -> 16 channels at 64x128x128, in two groups of tiles:
    // 16 voxels x 13 lines 92 us, 32 x 4 100, 64 x 2 117.
    constexpr int kSmem = 227 * 1024 - 1024 - 256;
    double best = 0;
    for (int bx = 16; bx <= 64 && bx < W + 16; bx += 16)
        for (int R = 1; R <= 16 && R <= H; R++) {
            const int unit = 2 * bx * g.wa, x_bytes = (((R + g.span) * 3 * g.cb * unit) + 1023) & ~1023;
            const int stage = (x_bytes + R * (bx + 2) * 2 * cout + 1023) & ~1023;
            // how far the last M tile of the last line reads past the stage
            int over = 0;
            for (int i = 0; i < g.mgroups; i++) {
                const int a0 = i * g.mt * per_tile, lines0 = a0 / (3 * g.cb);
                const int end = (R - 1 - lines0) * 3 * g.cb + a0 + std::min(g.mt, g.mtiles - i * g.mt) * per_tile;
                over = std::max(over, end * unit - stage);
            }
            const int nstage = std::min(6, (kSmem - over) / stage);
            if (nstage < 3) continue;
            const int tx = (W + bx - 1) / bx, ty = (H + R - 1) / R;
            const double tma = (R + g.span) * 3 * g.cb * bx + R * (bx + 2), mma = R * (bx / 16) * g.mt * (N > 48 ? 57 : 48);
            const double cost = (double)tx * ty * (std::max(tma, mma) + 200);
            if (best == 0 || cost < best) {
                best = cost;
                g.bx = bx;
                g.R = R;
                g.tx = tx;
                g.ty = ty;
                g.nstage = nstage;
                g.x_bytes = x_bytes;
                g.stage_bytes = stage;
                g.bar_off = nstage * stage + ((over + 15) & ~15);
            }
        }
    if (best == 0) return g;
    const long long nkb = (long long)g.tx * g.ty * D;
    if (nkb > INT_MAX) return g;
    g.nkb = (int)nkb;
    g.seg = g.nset * (kChain / (g.bx * g.R));
    // one CTA an SM: more than half of its shared memory
    g.smem = std::max<size_t>(1024 + g.bar_off + (2 * g.nstage + 2) * 8 + 4 + 16, 233472 / 2);
    const int want = std::max(1, 152 / g.mgroups), least = std::max(1, 256 / (g.bx * g.R));
    g.kb_per_cta = std::max((g.nkb + want - 1) / want, least);
    g.nchunk = (g.nkb + g.kb_per_cta - 1) / g.kb_per_cta;
    return g;
}

int64_t wgrad_tc_scratch(int cin, int cout, int D, int H, int W) {
    const WlineGeom l = wline_geom(cin, cout, D, H, W);
    if (l.nchunk) return (int64_t)l.nchunk * l.mtiles * kBM * 3 * cout;
    const WgradGeom g = wgrad_geom(cin, cout, D, H, W);
    return (int64_t)g.nchunk * g.mtiles * kBM * 3 * cout;
}

static cudaError_t wgrad_sum(const float4* partial, int nchunk, int mtiles, int cin, int cout, int bn, int wa, int lines,
                             float* dw, cudaStream_t st) {
    const dim3 grid((unsigned)(3 * cout / 4), (unsigned)((9 * ((cin + wa - 1) / wa) * wa + 31) / 32));
    if (nchunk > 32)
        return launch(wgrad_sum_kernel<16>, grid, 512, 0, st, partial, nchunk, mtiles, cin, cout, bn, wa, lines, dw);
    return launch(wgrad_sum_kernel<4>, grid, 128, 0, st, partial, nchunk, mtiles, cin, cout, bn, wa, lines, dw);
}

static cudaError_t wgrad_line(EncodeTiled enc, const WlineGeom& g, const void* x, int ldx, int cin, const void* dy, int ldy,
                              int cout, int D, int H, int W, float* partial, float* dw, cudaStream_t st) {
    alignas(64) CUtensorMap mx, md;
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    const cuuint64_t xrow = (cuuint64_t)ldx * 2, drow = (cuuint64_t)ldy * 2;
    {
        const cuuint64_t dims[5] = {(cuuint64_t)g.wa, (cuuint64_t)W, (cuuint64_t)g.cb, (cuuint64_t)D, (cuuint64_t)H};
        const cuuint64_t strides[4] = {xrow, (cuuint64_t)g.wa * 2, xrow * W * H, xrow * W};
        const cuuint32_t box[5] = {(cuuint32_t)g.wa, (cuuint32_t)g.bx, (cuuint32_t)g.cb, 3, (cuuint32_t)(g.R + g.span)};
        if (enc(&mx, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(x), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, g.wa == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    {
        const cuuint64_t dims[4] = {(cuuint64_t)cout, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)D};
        const cuuint64_t strides[3] = {drow, drow * W, drow * W * H};
        const cuuint32_t box[4] = {(cuuint32_t)cout, (cuuint32_t)(g.bx + 2), (cuuint32_t)g.R, 1};
        if (enc(&md, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(dy), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, cout == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    WlineArgs a = {};
    a.partial = reinterpret_cast<float4*>(partial);
    a.cb = g.cb;
    a.wa = g.wa;
    a.bn = cout;
    a.mtiles = g.mtiles;
    a.mt = g.mt;
    a.bx = g.bx;
    a.R = g.R;
    a.lines = g.R + g.span;
    a.tx = g.tx;
    a.ty = g.ty;
    a.nkb = g.nkb;
    a.kb_per_cta = g.kb_per_cta;
    a.nset = g.nset;
    a.seg = g.seg;
    a.nstage = g.nstage;
    a.stage_bytes = g.stage_bytes;
    a.x_bytes = g.x_bytes;
    a.bar_off = g.bar_off;
    a.tmem_cols = g.tmem_cols;
    a.fault = {g_stop_after, g_polls};
    const auto pick = [&](auto fault) {
        constexpr bool F = decltype(fault)::value;
        return g.bx == 64   ? wgrad_line_kernel<4, F>
               : g.bx == 48 ? wgrad_line_kernel<3, F>
               : g.bx == 32 ? wgrad_line_kernel<2, F>
                            : wgrad_line_kernel<1, F>;
    };
    const auto kernel = a.fault.stop_after < 0 ? pick(std::false_type()) : pick(std::true_type());
    cudaError_t e = raise_smem(kernel, kSmemCap, g.smem);
    if (e != cudaSuccess) return e;
    e = launch(kernel, dim3((unsigned)g.mgroups, (unsigned)g.nchunk), kThreads, g.smem, st, mx, md, a);
    if (e != cudaSuccess) return e;
    return wgrad_sum(a.partial, g.nchunk, g.mtiles, cin, cout, cout, g.wa, 1, dw, st);
}

// dw[t][co][ci] = sum_v dy[v][co] x[v + off_t][ci] on the tensor cores; partial: wgrad_tc_scratch
// floats.  cin multiple of 16 (<= 512), cout in {16, 32, 48, ..., 256} with cout % 16 == 0.
cudaError_t wgrad_tc(const void* x, int ldx, int cin, const void* dy, int ldy, int cout, int D, int H, int W,
                     float* partial, float* dw, cudaStream_t st) {
    EncodeTiled enc = encoder();
    if (!enc) return cudaErrorNotSupported;
    const WlineGeom l = wline_geom(cin, cout, D, H, W);
    if (l.nchunk) return wgrad_line(enc, l, x, ldx, cin, dy, ldy, cout, D, H, W, partial, dw, st);
    const WgradGeom g = wgrad_geom(cin, cout, D, H, W);
    if (g.mt * (kBM / g.wa) + 3 * (g.bn / g.wb) > 32) return cudaErrorInvalidValue;  // boxes a stage: one a lane
    const CUtensorMapSwizzle sa = g.wa == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : g.wa == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
                                                                                      : CU_TENSOR_MAP_SWIZZLE_32B;
    const CUtensorMapSwizzle sb = g.wb == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : g.wb == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
                                                                                      : CU_TENSOR_MAP_SWIZZLE_32B;
    alignas(64) CUtensorMap mx, md;
    const cuuint32_t es[4] = {1, 1, 1, 1};
    {
        const cuuint64_t dims[4] = {(cuuint64_t)cin, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)D};
        const cuuint64_t strides[3] = {(cuuint64_t)ldx * 2, (cuuint64_t)ldx * 2 * W, (cuuint64_t)ldx * 2 * W * H};
        const cuuint32_t box[4] = {(cuuint32_t)g.wa, (cuuint32_t)g.bx, (cuuint32_t)g.by, (cuuint32_t)g.bz};
        if (enc(&mx, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(x), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, sa, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    {
        const cuuint64_t dims[4] = {(cuuint64_t)cout, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)D};
        const cuuint64_t strides[3] = {(cuuint64_t)ldy * 2, (cuuint64_t)ldy * 2 * W, (cuuint64_t)ldy * 2 * W * H};
        const cuuint32_t box[4] = {(cuuint32_t)g.wb, (cuuint32_t)g.bx, (cuuint32_t)g.by, (cuuint32_t)g.bz};
        if (enc(&md, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(dy), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, sb, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    WgradArgs a = {};
    a.partial = reinterpret_cast<float4*>(partial);
    a.cin = cin;
    a.cout = cout;
    a.bn = g.bn;
    a.wa = g.wa;
    a.wb = g.wb;
    a.mtiles = g.mtiles;
    a.mt = g.mt;
    a.D = D;
    a.H = H;
    a.W = W;
    a.bx = g.bx;
    a.by = g.by;
    a.bz = g.bz;
    a.tx = g.tx;
    a.ty = g.ty;
    a.nkb = g.nkb;
    a.kb_per_cta = g.kb_per_cta;
    a.nstage = g.nstage;
    a.tmem_cols = g.tmem_cols;
    a.fault = {g_stop_after, g_polls};
    cudaError_t e = raise_smem(wgrad_tc_kernel, kSmemCap, g.smem);
    if (e != cudaSuccess) return e;
    e = launch(wgrad_tc_kernel, dim3((unsigned)(g.mgroups * g.ngroups), (unsigned)g.nchunk), kThreads, g.smem, st, mx,
                   md, a);
    if (e != cudaSuccess) return e;
    return wgrad_sum(a.partial, g.nchunk, g.mtiles, cin, cout, g.bn, g.wa, 0, dw, st);
}

// test hook: later convolutions and weight gradients issue only their first stop_after stages or planes (< 0: normal
// operation) and give up waiting for the others after `polls` polls (<= 0: the default)
void unet_set_copy_fault(int stop_after, int polls) {
    g_stop_after = stop_after;
    g_polls = polls > 0 ? polls : kPolls;
}

// reads and clears the device word of the tensor-core convolutions
cudaError_t unet_take_status(int* word, cudaStream_t st) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_unet_err);
    if (e == cudaSuccess) e = cudaMemcpyAsync(word, p, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess && *word) e = cudaMemsetAsync(p, 0, sizeof(int), st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return e;
}

}  // namespace pat
