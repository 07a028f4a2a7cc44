// A CUDA runtime of one host process for the tests of the library's host side: "device" memory is host memory, copies happen
// at once, launches do nothing.  It counts what the tests ask about and keeps what the preparation's launch was given.
// The test links it with the library's host object; entry points that are neither here nor there return zero.
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <vector>

#include "../paper_2604_24432_b200/csrc/ksa_launch.h"

#define FAKE extern "C" __attribute__((visibility("default")))

namespace {
struct Counts { int streams_made, streams_gone, mallocs, frees, device_syncs, uploads_default, uploads_own; };
Counts g_n{};
const ksa::SeqInfo* g_seqs = nullptr;
int g_num_seqs = 0;
}  // namespace

// what the last ksa_qkv_prepare was launched with
FAKE Counts fake_counts() { return g_n; }
FAKE const void* fake_seqs() { return g_seqs; }
FAKE int fake_seqs_text(const void* seqs, int i) { return static_cast<const ksa::SeqInfo*>(seqs)[i].n_text; }

cudaError_t ksa::launch_prep(const PrepArgs& a, int64_t, int num_seqs, cudaStream_t)
{
    g_seqs = a.seqs; g_num_seqs = num_seqs;
    return cudaSuccess;
}

FAKE cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
FAKE cudaError_t cudaGetDeviceProperties_v2(cudaDeviceProp* p, int)
{
    std::memset(p, 0, sizeof *p);
    p->major = 10; p->multiProcessorCount = 148;
    return cudaSuccess;
}
FAKE cudaError_t cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* r)
{
    static int entry;
    *fn = &entry; *r = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
FAKE cudaError_t cudaMalloc(void** p, size_t n) { ++g_n.mallocs; *p = std::malloc(n); return cudaSuccess; }
FAKE cudaError_t cudaFree(void* p) { ++g_n.frees; std::free(p); return cudaSuccess; }
FAKE cudaError_t cudaMemset(void* p, int v, size_t n) { std::memset(p, v, n); return cudaSuccess; }
FAKE cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
FAKE cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t stream)
{
    ++(stream ? g_n.uploads_own : g_n.uploads_default);
    std::memcpy(d, s, n);
    return cudaSuccess;
}
FAKE cudaError_t cudaDeviceSynchronize() { ++g_n.device_syncs; return cudaSuccess; }
FAKE cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned)
{
    ++g_n.streams_made;
    *s = reinterpret_cast<cudaStream_t>(std::malloc(1));
    return cudaSuccess;
}
FAKE cudaError_t cudaStreamDestroy(cudaStream_t s) { ++g_n.streams_gone; std::free(s); return cudaSuccess; }
