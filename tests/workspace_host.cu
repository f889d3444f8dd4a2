// The workspace's allocations against a device memory of a given size: the
// CUDA runtime calls that it makes are played on the host (nothing here runs on
// a GPU).
#include <cuda_runtime.h>

#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <map>

static size_t g_room = 0, g_used = 0;
static std::map<void*, size_t> g_live;

static cudaError_t played_malloc(void** p, size_t bytes, cudaStream_t) {
    if (g_used + bytes > g_room) return cudaErrorMemoryAllocation;
    static uintptr_t next = 4096;
    *p = reinterpret_cast<void*>(next);
    next += 4096;
    g_live[*p] = bytes;
    g_used += bytes;
    return cudaSuccess;
}
static cudaError_t played_free(void* p, cudaStream_t) {
    const auto it = g_live.find(p);
    if (it == g_live.end()) abort();
    g_used -= it->second;
    g_live.erase(it);
    return cudaSuccess;
}
template <class... A>
static cudaError_t played_ok(A...) { return cudaSuccess; }
#define cudaMallocAsync played_malloc
#define cudaFreeAsync played_free
#define cudaMemsetAsync played_ok
#define cudaStreamSynchronize played_ok
#define cudaGetLastError played_ok
#include "psf_internal.h"

namespace psf {
cudaError_t launch_reset(Ctl*, unsigned long long, unsigned long long, unsigned, cudaStream_t) { return cudaSuccess; }
size_t scan_scratch_len(int n) { return (size_t)n / 1024 + 3; }
namespace host {
std::atomic<int> g_row_bitmaps{1};
std::pair<void*, void*> mailbox_take() { return {nullptr, nullptr}; }
void mailbox_give(std::pair<void*, void*>) {}
int fail(int code, const char* fmt, ...) {
    va_list a;
    va_start(a, fmt);
    vprintf(fmt, a);
    va_end(a);
    printf("\n");
    return code;
}
}  // namespace host
}  // namespace psf

#define CHECK(x)                                                 \
    do {                                                         \
        if (!(x)) {                                              \
            printf("line %d: %s\n", __LINE__, #x);               \
            return 1;                                            \
        }                                                        \
    } while (0)

int main() {
    using namespace psf;
    using namespace psf::host;
    const int n = 1 << 16;
    const unsigned long long entries = 1ull << 24;
    const size_t lists = sizeof(uint2) * entries;
    g_room = ~(size_t)0 >> 1;
    {
        Work w;
        CHECK(w.init(n, nullptr, 10) == PSF_OK && w.init_products() == PSF_OK && w.reset_pool(entries) == PSF_OK);
        CHECK(w.lists() != nullptr && w.lists_cap == entries);
        g_room = g_used;  // the lists took the last of the memory
        Rows r;
        CHECK(w.rows_for(0, &r) == PSF_OK);  // a step's row arrays are not refused for them
        CHECK(g_used + (lists >> 1) < g_room);
        CHECK(w.lists() == nullptr);  // (the wide window from here on)
        // nor the room that a call without lists had at its end
        CHECK(w.rows_for(9, &r) == PSF_OK);
        const size_t before = g_used;
        CHECK(w.lists() == nullptr && g_used == before);
    }
    CHECK(g_used == 0);
    {
        Work w;
        g_room = ~(size_t)0 >> 1;
        CHECK(w.init(n, nullptr, 1) == PSF_OK && w.reset_pool(entries) == PSF_OK);
        const size_t base = g_used;
        CHECK(w.lists() != nullptr);
        // a phase's second pool has as much room as it had without lists
        g_room = base + base / 4 + 4096;
        CHECK(w.reset_pool(entries + entries / 4) == PSF_OK);
        CHECK(w.lists_cap == 0 && g_used > base + base / 8);
        // and the result
        g_room = ~(size_t)0 >> 1;
        w.no_lists = false;
        CHECK(w.lists() != nullptr);
        g_room = g_used;
        void* p = nullptr;
        CHECK(w.take(&p, lists / 2) == cudaSuccess && p != nullptr);
        CHECK(played_free(p, nullptr) == cudaSuccess);
    }
    CHECK(g_used == 0);
    printf("ok\n");
    return 0;
}
