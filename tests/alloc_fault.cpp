// cudaMalloc that finds no memory for sizes in [lo, hi): the library's host
// code, compiled with cudaMalloc renamed to this, runs its fallbacks on a GPU.
#include <cuda_runtime.h>

static size_t lo = 0, hi = 0;
static int refused = 0;

extern "C" void fault_between(size_t a, size_t b) {
    lo = a;
    hi = b;
}
extern "C" int fault_count() { return refused; }
extern "C" cudaError_t faulty_cudaMalloc(void **p, size_t n) {
    if (n >= lo && n < hi) {
        ++refused;
        *p = nullptr;
        return cudaErrorMemoryAllocation;
    }
    return cudaMalloc(p, n);
}
