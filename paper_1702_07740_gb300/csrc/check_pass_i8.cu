// Check-node pass kernels with int8 message storage.
#include "check_pass.cuh"
#include "check_direct.cuh"

namespace qc {
void *cn_kernel_i8(int maxdeg, int nt, bool soft) { return cn_kernel_select<int8_t>(maxdeg, nt, soft); }
void *cn_direct_i8(int slots, bool soft) { return cn_direct_select<int8_t>(slots, soft); }
void cn_smem_cap_i8(int cap) { cn_raise_smem_cap<int8_t>(cap); }
}  // namespace qc
