// rtc_master_create on a stand-in for the CUDA runtime (linked with --wrap) whose
// asynchronous copies read their source only when the stream is synchronised, as a
// runtime that reads pageable memory in place may.  Checks that no host memory is freed
// while a copy from it is queued, also where a later call fails, and that P arrives, rows
// padded with zeros, before it is put in lane order.  Prints what is wrong.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "rtc_internal.h"

namespace {
struct Copy {
    void* dst;
    const char* src;
    size_t n;
};
Copy queued[16];
int nqueued = 0;
bool freed_early = false;
const void* ordered_matrix = nullptr;      // launch_lane_order's argument, once its turn comes
bool order_queued = false;
std::vector<unsigned char> seen;           // the matrix as that launch finds it
size_t seen_bytes = 0;
bool fail_order = false, fail_product = false;

void run_queue() {
    for (int k = 0; k < nqueued; ++k) std::memcpy(queued[k].dst, queued[k].src, queued[k].n);
    nqueued = 0;
    if (order_queued) {
        order_queued = false;
        const auto* p = static_cast<const unsigned char*>(ordered_matrix);
        seen.assign(p, p + seen_bytes);
    }
}
void check_free(void* p) {
    for (int k = 0; k < nqueued; ++k)
        if (queued[k].src == p) {
            freed_early = true;
            queued[k] = queued[--nqueued];
            return;
        }
}
}  // namespace

void operator delete(void* p) noexcept { check_free(p); std::free(p); }
void operator delete(void* p, size_t) noexcept { check_free(p); std::free(p); }

extern "C" {
cudaError_t __wrap_cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t __wrap_cudaSetDevice(int) { return cudaSuccess; }
cudaError_t __wrap_cudaGetLastError() { return cudaSuccess; }
cudaError_t __wrap_cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) {
    *s = reinterpret_cast<cudaStream_t>(&nqueued);
    return cudaSuccess;
}
cudaError_t __wrap_cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t __wrap_cudaStreamSynchronize(cudaStream_t) { run_queue(); return cudaSuccess; }
cudaError_t __wrap_cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
    *e = reinterpret_cast<cudaEvent_t>(&nqueued);
    return cudaSuccess;
}
cudaError_t __wrap_cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t __wrap_cudaMalloc(void** p, size_t n) { *p = std::malloc(n); return *p ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t __wrap_cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t __wrap_cudaHostAlloc(void** p, size_t n, unsigned) { return __wrap_cudaMalloc(p, n); }
cudaError_t __wrap_cudaFreeHost(void* p) { return __wrap_cudaFree(p); }
cudaError_t __wrap_cudaMemset(void* p, int v, size_t n) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t __wrap_cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t __wrap_cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    if (nqueued == 16) return cudaErrorInvalidValue;
    queued[nqueued++] = Copy{d, static_cast<const char*>(s), n};
    return cudaSuccess;
}
}

namespace rtc {
size_t dtype_size(int dtype) { return dtype == RTC_F32 ? 4 : dtype == RTC_BF16 ? 2 : 1; }
int elems_per_16B(int dtype) { return int(16 / dtype_size(dtype)); }
cudaError_t launch_lane_order(int, void* M, const BlockDev*, int, int, int, int, cudaStream_t) {
    if (fail_order) return cudaErrorLaunchOutOfResources;
    ordered_matrix = M;
    order_queued = true;
    return cudaSuccess;
}
cudaError_t launch_gemv(int, const void*, const BlockDev*, int, int, int, const float*, const float*, float*, long long,
                        const FinaliseArgs*, long long, bool, cudaStream_t, const int*) {
    return fail_product ? cudaErrorLaunchOutOfResources : cudaSuccess;
}
}  // namespace rtc

int main() {
    int bad = 0;
    const int na = 37;
    const int types[3] = {RTC_F32, RTC_BF16, RTC_E4M3};
    for (int dtype : types)
        for (int fail = 0; fail < 3; ++fail) {
            fail_order = fail == 1;
            fail_product = fail == 2;
            freed_early = false;
            nqueued = 0;
            order_queued = false;
            seen.clear();
            const size_t row = na * rtc::dtype_size(dtype), pitch = (row + 15) / 16 * 16;
            seen_bytes = na * pitch;
            std::vector<unsigned char> p(na * row);
            for (size_t i = 0; i < p.size(); ++i) p[i] = (unsigned char)(1 + i % 61);     // finite in every format
            std::vector<float> scale(na, 1.f);
            rtc_polc polc{};
            polc.mode = RTC_POLC_IMPLICIT;
            polc.P = p.data();
            polc.dtype = dtype;
            polc.row_scale = dtype == RTC_F32 ? nullptr : scale.data();
            polc.gain = 0.5f;
            rtc_master_desc desc{};
            desc.na = na;
            desc.nshards = 2;
            desc.polc = &polc;
            rtc_master* m = nullptr;
            const int rc = rtc_master_create(&desc, &m);
            if (freed_early) { std::printf("type %d, failure %d: host memory freed under a queued copy\n", dtype, fail); ++bad; }
            if ((rc == RTC_OK) != (fail == 0)) { std::printf("type %d, failure %d: status %d\n", dtype, fail, rc); ++bad; }
            if (rc == RTC_OK) {
                bool same = seen.size() == seen_bytes;
                for (int r = 0; same && r < na; ++r)
                    for (size_t i = 0; i < pitch; ++i)
                        same = same && seen[r * pitch + i] == (i < row ? p[r * row + i] : 0);
                if (!same) { std::printf("type %d: P not uploaded before it is reordered\n", dtype); ++bad; }
                rtc_master_destroy(m);
            }
        }
    return bad ? 1 : 0;
}
