// plane_e.cu -- FP32 plane transform kernels for planes of x length 192, 256, 384 and 512.
#define IBM_PLANE_DEFINE
#include "plane.cuh"

namespace ibm {
IBM_PLANE_INSTANCE(192)
IBM_PLANE_INSTANCE(256)
IBM_PLANE_INSTANCE(384)
IBM_PLANE_INSTANCE(512)
}  // namespace ibm
