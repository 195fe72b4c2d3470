// edp_pass_line2_f.cu -- builds of the split line kernel (see edp_pass_line2.cu).
#include "line2_kernel.cuh"

namespace edp {

void *line2_k11(bool fused) { return line2_kernel<Build<Cut<8, 9>, Cut<8, 9>, NoCut, 512>, false>(fused); }
void *line2_k12(bool fused) { return line2_kernel<Build<Cut<2, 8>, Cut<2, 8>, Cut<2, 8>, 512>, false>(fused); }

}  // namespace edp
