// edp_pass_line2_e.cu -- builds of the split line kernel (see edp_pass_line2.cu).
#include "line2_kernel.cuh"

namespace edp {

void *line2_k9(bool fused) { return line2_kernel<Build<Cut<4, 8>, Cut<2, 8>, NoCut, 512>, false>(fused); }
void *line2_k10(bool fused) { return line2_kernel<Build<Cut<4, 8>, Cut<4, 8>, NoCut, 512>, false>(fused); }

}  // namespace edp
