// edp_pass_line2_c.cu -- builds of the split line kernel (see edp_pass_line2.cu).
#include "line2_kernel.cuh"

namespace edp {

void *line2_k3(bool fused) { return line2_kernel<Fixed2<25, 25, 3, 9, 3, 9, 512>, false>(fused); }
void *line2_k4(bool fused) { return line2_kernel<Fixed2<17, 17, 1, 17, 1, 17, 512>, false>(fused); }
void *line2_k8(bool fused) { return line2_kernel<Build<Cut<2, 8>, Cut<2, 8>, NoCut, 512>, false>(fused); }

}  // namespace edp
