// plan_upload_host.cpp -- the library's host code on a stand-in for the CUDA runtime whose asynchronous copies
// read their source as late as they may: when the stream is waited for.  Freed memory is overwritten, so
// a source that did not outlive its copy shows.  Built and run by test_plan_upload_cpu.py.
#include <cuda_runtime.h>
#include <malloc.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "qs_internal.h"

static void poison_free(void *p)
{
    if (p) memset(p, 0xdd, malloc_usable_size(p));
    free(p);
}
void operator delete(void *p) noexcept { poison_free(p); }
void operator delete[](void *p) noexcept { poison_free(p); }
void operator delete(void *p, size_t) noexcept { poison_free(p); }
void operator delete[](void *p, size_t) noexcept { poison_free(p); }

static struct Copy {
    void *dst;
    const void *src;
    size_t n;
    unsigned long long sum;
} queue[1024];
static int queued = 0, copies = 0, wrong = 0, launches = 0;

static unsigned long long checksum(const void *p, size_t n)
{
    unsigned long long h = 1469598103934665603ull;
    for (size_t i = 0; i < n; ++i) h = (h ^ static_cast<const unsigned char *>(p)[i]) * 1099511628211ull;
    return h;
}

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) { return *p = malloc(n), cudaSuccess; }
cudaError_t cudaFree(void *p) { return free(p), cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { return memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    queue[queued++] = Copy{d, s, n, checksum(s, n)};
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t)
{
    for (int i = 0; i < queued; ++i, ++copies) {
        wrong += checksum(queue[i].src, queue[i].n) != queue[i].sum;
        memcpy(queue[i].dst, queue[i].src, queue[i].n);
    }
    queued = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaStreamSynchronize(nullptr); }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s)
{
    return *s = cudaStreamCaptureStatusNone, cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return ""; }
}

namespace qs {
int max_slab_bits(qs_dtype dt) { return dt == QS_C64 ? 13 : 12; }
int launch_pass(const LaunchCtx &, const PassArgs &, const DevPass &, char *, size_t) { return ++launches, QS_OK; }
int launch_lean_pass(const LaunchCtx &, const LeanPassArgs &, const DevPass &, char *, size_t) { return ++launches, QS_OK; }
int launch_unblocked(const LaunchCtx &, const DevOp *, const DevOp &, const void *, char *, size_t) { return ++launches, QS_OK; }
int read_device_status(void *, int *v) { return *v = 0, QS_OK; }
}  // namespace qs

int main()
{
    alignas(256) static unsigned char amp[16 << 10];
    for (qs_dtype dt : {QS_C64, QS_C128}) {
        qs_state *s = nullptr;
        const int n = 10;
        if (qs_create_from_buffer(n, dt, amp, nullptr, &s)) return 2;
        for (int ng : {3, 40, 12}) {
            std::vector<qs_gate> g(ng);
            for (int i = 0; i < ng; ++i) {
                g[i] = qs_gate{};
                g[i].kind = i % 2 ? QS_RY : QS_CP;
                g[i].nt = i % 2 ? 1 : 2;
                g[i].t[0] = i % n;
                g[i].t[1] = (i + 3) % n;
                g[i].p[0] = 0.1 + i;
            }
            const int A[2] = {0, 2}, B[2] = {n - 1, 7};
            if (qs_apply_circuit(s, g.data(), g.size(), nullptr)) return 3;
            if (qs_remap(s, 2, A, B)) return 4;
            if (qs_canonicalize(s)) return 5;
        }
        qs_destroy(s);
    }
    printf("%d copies, %d wrong, %d unread, %d launches\n", copies, wrong, queued, launches);
    return wrong || queued || !copies || !launches;
}
