// edp_pass_line2.cu -- the scan-pass kernel for two- and three-axis label
// spaces with each label line shared by several lanes: its builds' table and
// launches.  The work item's body is in pass_line2.cuh, the builds in
// edp_pass_line2_*.cu.
#include "line2_builds.h"

namespace edp {

static const Line2Build kBuilds[] = {
    // the label spaces of the repository's workloads and tests
    {{65, 65, 1}, {5, 5, 0}, {13, 13, 0}, 480, line2_k0},
    {{33, 33, 1}, {3, 3, 0}, {11, 11, 0}, 512, line2_k1},
    {{27, 15, 1}, {3, 3, 0}, {9, 5, 0}, 512, line2_k2},
    {{25, 25, 1}, {3, 3, 0}, {9, 9, 0}, 512, line2_k3},
    {{17, 17, 1}, {1, 1, 0}, {17, 17, 0}, 512, line2_k4},
    {{9, 9, 1}, {3, 3, 0}, {3, 3, 0}, 640, line2_k5},
    {{17, 17, 9}, {1, 1, 1}, {17, 17, 9}, 384, line2_k6},
    {{9, 9, 9}, {1, 1, 1}, {9, 9, 9}, 512, line2_k7},
    // any line lengths up to segments x labels.  A column step of the first band,
    // rows coupled (320x265): 21 x 13 labels 1.48 us, 31 x 19 1.72, against 1.13 with
    // 27 x 15 above.  No build takes lines above 72 labels, a short axis beside a
    // long one (40 x 5, 3 x 20), or three axes with lines above 16 (but 17 x 17 x 9):
    // those stay on the multi-axis kernel
    {{0, 0, 0}, {2, 2, 0}, {8, 8, 0}, 512, line2_k8},
    {{0, 0, 0}, {4, 2, 0}, {8, 8, 0}, 512, line2_k9},
    {{0, 0, 0}, {4, 4, 0}, {8, 8, 0}, 512, line2_k10},
    {{0, 0, 0}, {8, 8, 0}, {9, 9, 0}, 512, line2_k11},
    {{0, 0, 0}, {2, 2, 2}, {8, 8, 8}, 512, line2_k12},
};

int pass_line2_max_lambda() { return line2::kMaxLambda; }
int pass_line2_builds() { return (int)(sizeof kBuilds / sizeof kBuilds[0]); }
const Line2Build &pass_line2_build(int b) { return kBuilds[b]; }
int pass_line2_max_rec_labels() { return line2::kMaxRecQ; }
int pass_line2_max_warps() { return line2::kMaxT; }
int pass_line2_max_rows() { return line2::kMaxRows; }
int pass_line2_threads(int NT, int T) { return 32 * NT * (T + line2::kCopyWarps); }

size_t pass_line2_smem(int NT, int Qm, int nst) { return ((size_t)Qm + NT * line2::team_ints(Qm, nst, 0)) * 4; }

// (dynamic shared memory beyond 48 KB with the static part needs the attribute)
int edp_pass_line2_occupancy(int build, int threads, size_t smem) {
    void *k = kBuilds[build].kernel(false);
    if (smem > 32 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, threads, smem);
    return occ;
}

int launch_edp_pass_line2(const TeamArgs &a, int build, int threads, size_t smem, cudaStream_t st) {
    void *k = kBuilds[build].kernel(a.fI1 != nullptr);
    if (!k) return -1;
    if (smem > 32 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    void *args[] = {const_cast<TeamArgs *>(&a)};
    return cudaLaunchKernel(k, dim3(a.grid), dim3(threads), args, smem, st) == cudaSuccess ? 0 : -2;
}

}  // namespace edp
