// Multi-step kernels of small domains with FP64 storage.
#include "resident_ops.cuh"

namespace axl {
const ResidentOps resident_fp64 = make_resident_ops<double>();
}  // namespace axl
