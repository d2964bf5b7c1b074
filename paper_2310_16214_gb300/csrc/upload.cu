// Tables made on the host, copied to the device once.
#include "internal.h"

namespace bplg {

// cudaMemcpy from pageable memory may return once the bytes are staged, before
// they are on the device, and orders only the legacy default stream behind
// them: a kernel launched next on a non-blocking stream (torch's side streams
// are) could read a table that is not filled yet.  So the copy runs on a stream
// of its own, which is waited for.
int upload(void *dst, const void *src, size_t bytes, const char *what) {
    cudaStream_t st;
    cudaError_t e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    if (e != cudaSuccess) return cuda_error(e, what);
    e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st);
    const cudaError_t done = cudaStreamSynchronize(st);
    cudaStreamDestroy(st);
    if (e == cudaSuccess) e = done;
    return e == cudaSuccess ? BPLG_OK : cuda_error(e, what);
}

}  // namespace bplg
