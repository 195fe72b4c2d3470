// edp_pass_line2_c.cu -- builds of the split line kernel (see edp_pass_line2.cu).
#include "line2_kernel.cuh"

namespace edp {

void *line2_k4(bool fused) { return line2_kernel<Build<Cut<8, 3>, Cut<4, 5>, Cut<0, 0>, true>, false>(fused); }
void *line2_k5(bool fused) { return line2_kernel<Build<Cut<4, 3>, Cut<4, 3>, Cut<0, 0>, true>, false>(fused); }
void *line2_k8(bool fused) { return line2_kernel<Build<Cut<4, 4>, Cut<4, 4>, Cut<0, 0>, false>, false>(fused); }

}  // namespace edp
