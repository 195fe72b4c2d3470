// edp_pass_line2_d.cu -- builds of the split line kernel (see edp_pass_line2.cu).
#include "line2_kernel.cuh"

namespace edp {

void *line2_k6(bool fused) { return line2_kernel<Fixed3<17, 17, 9, 1, 17, 1, 17, 1, 9, 384>, false>(fused); }
void *line2_k7(bool fused) { return line2_kernel<Fixed3<9, 9, 9, 1, 9, 1, 9, 1, 9, 512>, false>(fused); }

}  // namespace edp
