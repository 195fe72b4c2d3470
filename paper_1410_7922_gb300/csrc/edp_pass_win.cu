// edp_pass_win.cu -- the scan-pass kernel on per-pixel label boxes (two axes,
// linear prior); the row body is in pass_win.cuh, the work item's frame in
// pass_line2.cuh.
#include "line2_kernel.cuh"
#include "pass_win.cuh"

namespace edp {

// one build per box side: segments per line so that a warp's lanes hold a box
static void *win_kernel_for(int n) {
    using line2::WinBuild;
    switch (n) {
    case 3: return line2_kernel<WinBuild<3, 1>, false>(false);
    case 5: return line2_kernel<WinBuild<5, 2>, false>(false);
    case 7: return line2_kernel<WinBuild<7, 3>, false>(false);
    case 9: return line2_kernel<WinBuild<9, 3>, false>(false);
    case 11: return line2_kernel<WinBuild<11, 2>, false>(false);
    case 13: return line2_kernel<WinBuild<13, 2>, false>(false);
    case 15: return line2_kernel<WinBuild<15, 2>, false>(false);
    default: return nullptr;
    }
}

bool pass_win_built(int n) { return win_kernel_for(n) != nullptr; }

size_t pass_win_smem(int NT, int Qm, int nst) { return ((size_t)Qm + NT * line2::team_ints(Qm, nst, 2)) * 4; }

int edp_pass_win_occupancy(int n, int threads, size_t smem) {
    void *k = win_kernel_for(n);
    if (!k) return 0;
    if (smem > 32 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, threads, smem);
    return occ;
}

int launch_edp_pass_win(const TeamArgs &a, int threads, size_t smem, cudaStream_t st) {
    void *k = win_kernel_for(a.win);
    if (!k) return -1;
    if (smem > 32 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    void *args[] = {const_cast<TeamArgs *>(&a)};
    return cudaLaunchKernel(k, dim3(a.grid), dim3(threads), args, smem, st) == cudaSuccess ? 0 : -2;
}

}  // namespace edp
