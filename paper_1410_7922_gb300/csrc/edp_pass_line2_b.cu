// edp_pass_line2_b.cu -- builds of the split line kernel (see edp_pass_line2.cu).
#include "line2_kernel.cuh"

namespace edp {

void *line2_k1(bool fused) { return line2_kernel<Build<Cut<8, 5>, Cut<4, 9>, Cut<0, 0>, true>, false>(fused); }
void *line2_k2(bool fused) { return line2_kernel<Build<Cut<8, 4>, Cut<4, 4>, Cut<0, 0>, true>, false>(fused); }
void *line2_k3(bool fused) { return line2_kernel<Build<Cut<8, 4>, Cut<4, 7>, Cut<0, 0>, true>, false>(fused); }

}  // namespace edp
