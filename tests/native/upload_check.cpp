// Host-side check of upload() (csrc/upload.cu) against a stand-in for the CUDA
// runtime that does as little as CUDA promises: a copy only stages its bytes,
// and they land when the stream of the copy is waited for.  The bytes must be in
// place when upload() returns, the stream given back, and each failing call
// reported.  Prints "OK" or the first failure.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "internal.h"

namespace bplg {
int cuda_error(cudaError_t, const char *) { return BPLG_ERR_CUDA; }
}  // namespace bplg

namespace {
struct Pending {
    void *dst;
    std::vector<char> bytes;
    cudaStream_t st;
};
std::vector<Pending> g_pending;
int g_streams = 0;
std::string g_fail;  // the runtime call that fails
cudaStream_t const kStream = reinterpret_cast<cudaStream_t>(0x100);

cudaError_t result(const char *name) { return g_fail == name ? cudaErrorUnknown : cudaSuccess; }
void stage(void *dst, const void *src, size_t n, cudaStream_t st) {
    const char *p = static_cast<const char *>(src);
    g_pending.push_back(Pending{dst, std::vector<char>(p, p + n), st});
}
}  // namespace

extern "C" {
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    if (result("create") != cudaSuccess) return result("create");
    ++g_streams;
    *s = kStream;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) {
    --g_streams;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind, cudaStream_t st) {
    if (result("copy") != cudaSuccess) return result("copy");
    stage(dst, src, n, st);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *dst, const void *src, size_t n, cudaMemcpyKind) {
    stage(dst, src, n, nullptr);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t st) {
    for (auto it = g_pending.begin(); it != g_pending.end();)
        if (it->st == st) {
            std::memcpy(it->dst, it->bytes.data(), it->bytes.size());
            it = g_pending.erase(it);
        } else {
            ++it;
        }
    return result("wait");
}
}

int main() {
    std::vector<char> src(1000), dst(1000, 0);
    for (size_t i = 0; i < src.size(); ++i) src[i] = static_cast<char>(i * 7 + 1);
    if (bplg::upload(dst.data(), src.data(), src.size(), "table") != BPLG_OK) return printf("FAIL: error\n"), 1;
    if (dst != src) return printf("FAIL: returned before the bytes were in place\n"), 1;
    if (g_streams != 0) return printf("FAIL: %d streams left\n", g_streams), 1;
    for (const char *call : {"create", "copy", "wait"}) {
        g_fail = call;
        if (bplg::upload(dst.data(), src.data(), src.size(), "table") != BPLG_ERR_CUDA || g_streams != 0)
            return printf("FAIL: %s failing\n", call), 1;
    }
    printf("OK\n");
    return 0;
}
