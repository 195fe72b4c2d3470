// edp_pass_line2_a.cu -- builds of the split line kernel (see edp_pass_line2.cu).
#include "line2_kernel.cuh"

namespace edp {

void *line2_k0(bool fused) { return line2_kernel<Fixed2<65, 65, 5, 13, 5, 13, 480>, true>(fused); }
void *line2_k5(bool fused) { return line2_kernel<Fixed2<9, 9, 3, 3, 3, 3, 640>, false>(fused); }

}  // namespace edp
