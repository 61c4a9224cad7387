// The array alone, in a translation unit of its own: what a .cu file defines reaches a GPU as one module, which the driver loads when
// something of it is first asked for (unless CUDA_MODULE_LOADING=EAGER).  So a program that never makes the allocation-free call
// does not hold these bytes: with the array beside the kernels, every context on a GPU cost 38 MB more.
#include "noalloc_scratch.h"

static __device__ __align__(256) unsigned char g_noalloc_scratch[hc::NOALLOC_SCRATCH_BYTES];

// (the array's name is only a host-side handle, a kernel needs its address on the device it runs on)
cudaError_t hc::noalloc_scratch_address(void** ptr) { return cudaGetSymbolAddress(ptr, g_noalloc_scratch); }
