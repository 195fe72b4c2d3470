// edp_pass_line2.cu -- the scan-pass kernel for two- and three-axis label
// spaces with each label line shared by several lanes: its builds' table and
// launches.  The work item's body is in pass_line2.cuh, the builds in
// edp_pass_line2_*.cu.
#include "line2_builds.h"

namespace edp {

static const Line2Build kBuilds[] = {
    // exact cuts (segments, labels per lane of each axis): the repository's
    // label spaces -- 65 x 65, 33 x 33, 27 x 15, 25 x 25, 17 x 17, 9 x 9,
    // 17 x 17 x 9, 9 x 9 x 9
    {{8, 8, 0}, {9, 9, 0}, true, 672, line2_k0},
    {{8, 4, 0}, {5, 9, 0}, true, line2::kMaxThreads, line2_k1},
    {{8, 4, 0}, {4, 4, 0}, true, line2::kMaxThreads, line2_k2},
    {{8, 4, 0}, {4, 7, 0}, true, line2::kMaxThreads, line2_k3},
    {{8, 4, 0}, {3, 5, 0}, true, line2::kMaxThreads, line2_k4},
    {{4, 4, 0}, {3, 3, 0}, true, line2::kMaxThreads, line2_k5},
    {{4, 2, 1}, {5, 9, 9}, true, line2::kMaxThreads, line2_k6},
    {{4, 2, 2}, {3, 5, 5}, true, line2::kMaxThreads, line2_k7},
    // any line lengths up to segments x labels
    {{4, 4, 0}, {4, 4, 0}, false, line2::kMaxThreads, line2_k8},
    {{8, 4, 0}, {4, 4, 0}, false, line2::kMaxThreads, line2_k9},
    {{8, 4, 0}, {4, 8, 0}, false, line2::kMaxThreads, line2_k10},
    {{8, 8, 0}, {9, 9, 0}, false, 672, line2_k11},
    {{4, 4, 4}, {4, 4, 4}, false, line2::kMaxThreads, line2_k12},
};

int pass_line2_max_lambda() { return line2::kMaxLambda; }
int pass_line2_builds() { return (int)(sizeof kBuilds / sizeof kBuilds[0]); }
const Line2Build &pass_line2_build(int b) { return kBuilds[b]; }
int pass_line2_max_warps() { return line2::kMaxT; }
int pass_line2_threads(int NT, int T) { return 32 * NT * (T + line2::kCopyWarps); }

size_t pass_line2_smem(int NT, int Qm, int nst) { return ((size_t)Qm + NT * line2::team_ints(Qm, nst, 0)) * 4; }

int edp_pass_line2_occupancy(int build, int threads, size_t smem) {
    void *k = kBuilds[build].kernel(false);
    if (smem > 48 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, threads, smem);
    return occ;
}

int launch_edp_pass_line2(const TeamArgs &a, int build, int threads, size_t smem, cudaStream_t st) {
    void *k = kBuilds[build].kernel(a.fI1 != nullptr);
    if (!k) return -1;
    if (smem > 48 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    void *args[] = {const_cast<TeamArgs *>(&a)};
    return cudaLaunchKernel(k, dim3(a.grid), dim3(threads), args, smem, st) == cudaSuccess ? 0 : -2;
}

}  // namespace edp
