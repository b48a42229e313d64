// Multi-step kernels of small domains and batches with FP16 storage.
#include "resident_ops.cuh"

namespace axl {
const ResidentOps resident_fp16 = make_resident_ops<__half>();
}  // namespace axl
