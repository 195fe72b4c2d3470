// edp_pass_line2_a.cu -- builds of the split line kernel (see edp_pass_line2.cu).
#include "line2_kernel.cuh"

namespace edp {

void *line2_k0(bool fused) { return line2_kernel<Build<Cut<8, 9>, Cut<8, 9>, Cut<0, 0>, true, 672>, true>(fused); }

}  // namespace edp
