// pat_step.cuh - a whole time step of a small grid in one launch.
//
// The three line passes of a step (pat_line.cuh) read the same spectrum and states of their own, and depend on one
// another only through the new spectrum, which the y and z passes add to.  On a small grid a pass is 30 to 400 CTAs, a
// fraction of the chip, and takes as long as its chain of loads, four transforms and stores; three of them after one
// another, their second halves serialised by the additions, made a step (8.9 us at 32^3).  Here each pass writes a
// spectrum of its own and the next step reads the sum of the three, added in the order in which the passes added them
// ((x + y) + z), so the results are the same bit for bit.  The passes then run side by side in one grid, and a step
// waits for its predecessor once.  The recorded plane is taken from the spectrum when the next step reads it.
//
// Every tile of every axis is a CTA, and the line lengths are a switch inside the kernel (18 inlined passes: a kernel
// per combination of three lengths would be 216).  RES is the number of CTAs an SM the registers are kept for:
// 3 (168 registers) or 4 (128, a few spilled).
#pragma once
#include "pat_line.cuh"

namespace pat {

template <int L, int AX>
__device__ __forceinline__ void step_pass(const LineArgs& a, int tile) {
    static_assert(LS<L>::NT <= kStepThreads, "threads of a pass");
    if (LS<L>::NT < kStepThreads && (int)threadIdx.x >= LS<L>::NT) return;
    line_pass<L, AX, false, true>(a, tile);
}

template <int AX>
__device__ __forceinline__ void step_axis(const LineArgs& a, int tile) {
    switch (a.g.len[AX]) {
        case 8: step_pass<8, AX>(a, tile); break;
        case 16: step_pass<16, AX>(a, tile); break;
        case 32: step_pass<32, AX>(a, tile); break;
        case 64: step_pass<64, AX>(a, tile); break;
        case 128: step_pass<128, AX>(a, tile); break;
        case 256: step_pass<256, AX>(a, tile); break;
    }
}

template <int RES>
__global__ void __launch_bounds__(kStepThreads, RES) step_kernel(const __grid_constant__ StepArgs s) {
    const int i = blockIdx.x;
    if (i >= s.first[0]) step_axis<0>(s.a[0], i - s.first[0]);
    else if (i >= s.first[1]) step_axis<1>(s.a[1], i - s.first[1]);
    else step_axis<2>(s.a[2], i);
}

}  // namespace pat
