// edp_pass_line2_d.cu -- builds of the split line kernel (see edp_pass_line2.cu).
#include "line2_kernel.cuh"

namespace edp {

void *line2_k6(bool fused) { return line2_kernel<Build<Cut<4, 5>, Cut<2, 9>, Cut<1, 9>, true>, false>(fused); }
void *line2_k7(bool fused) { return line2_kernel<Build<Cut<4, 3>, Cut<2, 5>, Cut<2, 5>, true>, false>(fused); }

}  // namespace edp
