// line2_builds.h -- the builds of the split line kernel, one function each that
// returns the kernel (fused: with the pair cost computed from the images, null
// where that is not built).
#pragma once
#include "pass_line2.cuh"

namespace edp {
void *line2_k0(bool fused);
void *line2_k1(bool fused);
void *line2_k2(bool fused);
void *line2_k3(bool fused);
void *line2_k4(bool fused);
void *line2_k5(bool fused);
void *line2_k6(bool fused);
void *line2_k7(bool fused);
void *line2_k8(bool fused);
void *line2_k9(bool fused);
void *line2_k10(bool fused);
void *line2_k11(bool fused);
void *line2_k12(bool fused);

}  // namespace edp
