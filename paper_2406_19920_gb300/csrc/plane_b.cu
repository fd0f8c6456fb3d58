// plane_b.cu -- FP32 plane transform kernels for planes of x length 24 and 32.
#define IBM_PLANE_DEFINE
#include "plane.cuh"

namespace ibm {
IBM_PLANE_INSTANCE(24)
IBM_PLANE_INSTANCE(32)
}  // namespace ibm
