// Host code of the library that has no entry point of its own, without a GPU: linked with the library's objects, the runtime
// calls that need a device replaced (-Wl,--wrap).  Usage: host_checks NAME; exit status 0 and a line of figures, or 1.
#include "conv_pipe.h"

#include <cstdio>
#include <cstring>
#include <map>
#include <thread>
#include <vector>

using namespace hpf;

static thread_local int g_device = 0;
static std::mutex g_lock;
static std::map<int, int> g_attributes;      // device -> attributes set on it
static int g_fail_on = -1;

extern "C" {
cudaError_t __wrap_cudaGetDevice(int* dev) { *dev = g_device; return cudaSuccess; }
cudaError_t __wrap_cudaFuncSetAttribute(const void*, cudaFuncAttribute, int)
{
    std::lock_guard<std::mutex> hold(g_lock);
    if (g_device == g_fail_on) return cudaErrorInvalidDevice;
    ++g_attributes[g_device];
    return cudaSuccess;
}
cudaError_t __wrap_cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* q)
{
    *fn = reinterpret_cast<void*>(&g_attributes);
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
}

#define CHECK(x) do { if (!(x)) { printf("%s:%d: %s\n", __FILE__, __LINE__, #x); return 1; } } while (0)

// Kernel attributes belong to a device: each device a process drives gets its own, once, whichever thread comes first.
static int attributes_per_device()
{
    CHECK(conv_tc_init() == cudaSuccess && conv_pipe_init() == cudaSuccess);
    const int n = g_attributes[0];
    CHECK(n > 0);
    g_device = 1;
    CHECK(conv_tc_init() == cudaSuccess && conv_pipe_init() == cudaSuccess);
    CHECK(g_attributes[1] == n);
    g_device = 2; g_fail_on = 2;
    CHECK(conv_pipe_init() != cudaSuccess);      // a failure is not remembered as done
    g_fail_on = -1;
    CHECK(conv_tc_init() == cudaSuccess && conv_pipe_init() == cudaSuccess);
    CHECK(g_attributes[2] == n);
    std::vector<std::thread> all;
    for (int t = 0; t < 16; ++t)
        all.emplace_back([t] { g_device = 3 + t % 4; (void)conv_tc_init(); (void)conv_pipe_init(); });
    for (auto& t : all) t.join();
    for (int d = 0; d < 7; ++d) CHECK(g_attributes[d] == n);
    printf("%d attributes on each of 7 devices\n", n);
    return 0;
}

int main(int argc, char** argv)
{
    if (argc > 1 && !strcmp(argv[1], "attributes_per_device")) return attributes_per_device();
    printf("unknown check\n");
    return 1;
}
