// Check-node pass kernels with FP16 message storage.
#include "check_pass.cuh"
#include "check_direct.cuh"

namespace qc {
void *cn_kernel_f16(int maxdeg, int nt, bool soft) { return cn_kernel_select<__half>(maxdeg, nt, soft); }
void *cn_direct_f16(int slots, bool soft) { return cn_direct_select<__half>(slots, soft); }
void cn_smem_cap_f16(int cap) { cn_raise_smem_cap<__half>(cap); }
}  // namespace qc
