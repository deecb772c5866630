// The resident decode's sum-product kernels with check-to-bit messages stored as float.
#include "ldpc_resident_kernel.cuh"

LDPC_INSTANTIATE_RESIDENT(float, 0)
