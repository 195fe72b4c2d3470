// edp_pass_axis1.cu -- the scan-pass kernel for one label axis in the split line
// kernel's frame; the row body is in pass_axis1.cuh.
#include "line2_kernel.cuh"
#include "pass_axis1.cuh"

namespace edp {

// labels per lane: 16 lanes hold a vector
static int axis1_labels(int Q) { return Q <= 32 ? 2 : Q <= 64 ? 4 : Q <= 128 ? 8 : 16; }

template <int E>
static void *axis1_kernel_e(bool quad, bool vc) {
    using line2::Axis1Build;
    if (quad)
        return vc ? line2_kernel<Axis1Build<E, true, true>, false>(false) : line2_kernel<Axis1Build<E, true, false>, false>(false);
    return vc ? line2_kernel<Axis1Build<E, false, true>, false>(false) : line2_kernel<Axis1Build<E, false, false>, false>(false);
}
static void *axis1_kernel_for(int Q, int l1) {
    const bool quad = l1 == 2, vc = Q % 4 == 0;
    switch (axis1_labels(Q)) {
    case 2: return axis1_kernel_e<2>(quad, vc);
    case 4: return axis1_kernel_e<4>(quad, vc);
    case 8: return axis1_kernel_e<8>(quad, vc);
    default: return axis1_kernel_e<16>(quad, vc);
    }
}

int pass_axis1_carry(int Q, int g) {
    const int E = axis1_labels(Q);
    return g <= 1 ? 0 : (int)((g - 1LL + E - 1) / E < 15 ? (g - 1LL + E - 1) / E : 15);
}
size_t pass_axis1_smem(int NT, int Qm, int nst, int l1) {
    return ((size_t)Qm + 64 + NT * line2::team_ints(Qm, nst, l1 == 2 ? 2 : 0)) * 4;
}

int edp_pass_axis1_occupancy(int Q, int l1, int threads, size_t smem) {
    void *k = axis1_kernel_for(Q, l1);
    if (smem > 32 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, threads, smem);
    return occ;
}

int launch_edp_pass_axis1(const TeamArgs &a, int threads, size_t smem, cudaStream_t st) {
    void *k = axis1_kernel_for(a.Q, a.l1);
    if (smem > 32 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    void *args[] = {const_cast<TeamArgs *>(&a)};
    return cudaLaunchKernel(k, dim3(a.grid), dim3(threads), args, smem, st) == cudaSuccess ? 0 : -2;
}

}  // namespace edp
