// The resident decode's min-sum kernels with check-to-bit messages stored as int8 levels.
#include "ldpc_resident_kernel.cuh"

LDPC_INSTANTIATE_RESIDENT(int8_t, 1)
