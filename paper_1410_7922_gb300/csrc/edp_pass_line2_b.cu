// edp_pass_line2_b.cu -- builds of the split line kernel (see edp_pass_line2.cu).
#include "line2_kernel.cuh"

namespace edp {

void *line2_k1(bool fused) { return line2_kernel<Fixed2<33, 33, 3, 11, 3, 11, 512>, false>(fused); }
void *line2_k2(bool fused) { return line2_kernel<Fixed2<27, 15, 3, 9, 3, 5, 512>, false>(fused); }

}  // namespace edp
