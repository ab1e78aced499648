// The work space of the digit products of afqmc_local_energy_noalloc, in a translation unit (a module) of its
// own: where a GPU has no room left for it, loading it fails by itself and the call runs the FP64 kernel.
#include "kernels.cuh"

namespace afq {

// the digits of h and L take 16 MB at 50 orbitals and 250 vectors, 200 MB at 120 and 600
static __device__ __align__(256) unsigned char g_noalloc_work[NOALLOC_WORK_BYTES];

cudaError_t noalloc_work(void** address) { return cudaGetSymbolAddress(address, g_noalloc_work); }

}  // namespace afq
