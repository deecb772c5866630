// The resident decode's min-sum kernels with check-to-bit messages stored as half.
#include "ldpc_resident_kernel.cuh"

LDPC_INSTANTIATE_RESIDENT(__half, 1)
