// Multi-step kernels of small domains with BF16 storage.
#include "resident_ops.cuh"

namespace axl {
const ResidentOps resident_bf16 = make_resident_ops<__nv_bfloat16>();
}  // namespace axl
