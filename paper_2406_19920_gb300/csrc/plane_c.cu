// plane_c.cu -- FP32 plane transform kernels for planes of x length 48 and 64.
#define IBM_PLANE_DEFINE
#include "plane.cuh"

namespace ibm {
IBM_PLANE_INSTANCE(48)
IBM_PLANE_INSTANCE(64)
}  // namespace ibm
