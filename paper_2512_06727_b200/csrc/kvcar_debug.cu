// Test hook of the bounded waits.
#include "kvcar_internal.h"
#include "kvcar_ptx.cuh"

namespace kvcar {

using namespace ptx;

namespace {

// A wait that nothing completes: one warp waits on a fresh barrier with the given limit, records its code in the
// status word and returns.  Exercises the path every bounded wait of the library takes when it runs out.
__global__ void expire_wait_kernel(int32_t *status, uint64_t limit_ns) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) mbar_init(smem_u32(&bar), 1);
    __syncwarp();
    const uint32_t b = smem_u32(&bar);
    const uint64_t t0 = global_ns();
    while (!mbar_try(b, 0)) {
        __nanosleep(200);
        if (global_ns() - t0 > limit_ns) {
            atomicCAS(status, 0, 0x7e57);
            break;
        }
    }
}

}  // namespace

cudaError_t launch_expire_wait(int32_t *status, uint64_t limit_ns, cudaStream_t st) {
    expire_wait_kernel<<<1, 32, 0, st>>>(status, limit_ns);
    return cudaGetLastError();
}

}  // namespace kvcar
