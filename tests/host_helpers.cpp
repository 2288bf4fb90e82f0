// Host-side helpers of the library with C names, for tests/test_host_helpers.py.
#include <cstdlib>
#include <new>

#include "../paper_2508_07424_gb300/csrc/pff_host.cuh"

extern "C" void map_pages(void *p, size_t bytes) { pff::map_pages(p, bytes); }

// The two CUDA calls of smem_raise, and an allocator that can be told to fail.
static bool g_no_memory = false;
static int g_calls = 0;
static size_t g_set = 0;
void *operator new(size_t n) {
    void *p = g_no_memory ? nullptr : std::malloc(n);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }
extern "C" cudaError_t cudaGetDevice(int *dev) {
    *dev = 0;
    return cudaSuccess;
}
extern "C" cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int bytes) {
    ++g_calls;
    g_set = (size_t)bytes;
    return bytes > 227 * 1024 ? cudaErrorInvalidValue : cudaSuccess;
}

extern "C" int smem_raise(size_t kernel, size_t bytes, int no_memory, int *calls, size_t *set) {
    g_no_memory = no_memory != 0;
    const int e = (int)pff::smem_raise((const void *)kernel, bytes);
    g_no_memory = false;
    *calls = g_calls;
    *set = g_set;
    return e;
}
