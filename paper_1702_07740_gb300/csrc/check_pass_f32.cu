// Check-node pass kernels with FP32 message storage.
#include "check_pass.cuh"
#include "check_direct.cuh"

namespace qc {
void *cn_kernel_f32(int maxdeg, int nt, bool soft) { return cn_kernel_select<float>(maxdeg, nt, soft); }
void *cn_direct_f32(int slots, bool soft) { return cn_direct_select<float>(slots, soft); }
void cn_smem_cap_f32(int cap) { cn_raise_smem_cap<float>(cap); }
}  // namespace qc
