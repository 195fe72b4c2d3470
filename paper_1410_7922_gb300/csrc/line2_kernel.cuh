// line2_kernel.cuh -- the split line kernel of one build.
#pragma once
#include "line2_builds.h"

namespace edp {

using line2::Build;
using line2::Cut;
using line2::Fixed2;
using line2::Fixed3;
using line2::NoCut;

// FUSED: the pair cost computed from the images instead of read from C
template <class B, bool FUSED>
__global__ void __launch_bounds__(B::threads, 1) edp_pass_line2_kernel(const __grid_constant__ TeamArgs A) {
    extern __shared__ __align__(128) int smem_i[];
    __shared__ int s_item;
    __shared__ volatile int s_abort;
    if (threadIdx.x == 0) s_abort = (*(volatile int *)A.status != 0);
    __syncthreads();
    if (s_abort) return;
    const int items = A.nbands * (A.pair ? 2 : 1);
    while (true) {
        if (threadIdx.x == 0) s_item = (int)atomicAdd(A.band_counter, 1u);
        __syncthreads();
        const int item = s_item;
        if (item >= items) break;
        const int h = item >= A.nbands;
        if (!line2_item<B, FUSED>(A, h, item - h * A.nbands, smem_i, &s_abort)) return;
    }
}

template <class B, bool WITH_FUSED>
void *line2_kernel(bool fused) {
    if constexpr (WITH_FUSED)
        if (fused) return reinterpret_cast<void *>(edp_pass_line2_kernel<B, true>);
    return fused ? nullptr : reinterpret_cast<void *>(edp_pass_line2_kernel<B, false>);
}

}  // namespace edp
