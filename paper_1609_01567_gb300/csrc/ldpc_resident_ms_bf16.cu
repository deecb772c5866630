// The resident decode's min-sum kernels with check-to-bit messages stored as bfloat16.
#include "ldpc_resident_kernel.cuh"

LDPC_INSTANTIATE_RESIDENT(__nv_bfloat16, 1)
