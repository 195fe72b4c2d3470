// edp_pass_line2_f.cu -- builds of the split line kernel (see edp_pass_line2.cu).
#include "line2_kernel.cuh"

namespace edp {

void *line2_k11(bool fused) { return line2_kernel<Build<Cut<8, 9>, Cut<8, 9>, Cut<0, 0>, false, 672>, false>(fused); }
void *line2_k12(bool fused) { return line2_kernel<Build<Cut<4, 4>, Cut<4, 4>, Cut<4, 4>, false>, false>(fused); }

}  // namespace edp
