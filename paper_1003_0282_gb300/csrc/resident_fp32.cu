// Multi-step kernels of small domains and batches with FP32 storage.
#include "resident_ops.cuh"

namespace axl {
const ResidentOps resident_fp32 = make_resident_ops<float>();
}  // namespace axl
