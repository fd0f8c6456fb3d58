// plane_d.cu -- FP32 plane transform kernels for planes of x length 96 and 128.
#define IBM_PLANE_DEFINE
#include "plane.cuh"

namespace ibm {
IBM_PLANE_INSTANCE(96)
IBM_PLANE_INSTANCE(128)
}  // namespace ibm
