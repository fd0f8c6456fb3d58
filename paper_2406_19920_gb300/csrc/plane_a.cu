// plane_a.cu -- FP32 plane transform kernels for planes of x length 8, 12 and 16.
#define IBM_PLANE_DEFINE
#include "plane.cuh"

namespace ibm {
IBM_PLANE_INSTANCE(8)
IBM_PLANE_INSTANCE(12)
IBM_PLANE_INSTANCE(16)
}  // namespace ibm
