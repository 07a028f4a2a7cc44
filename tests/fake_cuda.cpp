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
struct Retained { void* graph; cudaHostFn_t destroy; void* ptr; };
std::vector<Retained> g_retained;
void* g_graph = nullptr;                                 // the graph that calls are recorded into, null: none
}  // namespace

FAKE void fake_capture(void* graph) { g_graph = graph; }
FAKE void fake_graph_destroy(void* graph)
{
    for (size_t i = g_retained.size(); i-- > 0;)
        if (g_retained[i].graph == graph) {
            g_retained[i].destroy(g_retained[i].ptr);
            g_retained.erase(g_retained.begin() + (long)i);
        }
}
FAKE Counts fake_counts() { return g_n; }
// the schedule that the last ksa_qkv_prepare was launched with
FAKE const void* fake_seqs() { return g_seqs; }
FAKE int fake_seqs_text(const void* seqs, int i) { return static_cast<const ksa::SeqInfo*>(seqs)[i].n_text; }

cudaError_t ksa::launch_prep(const PrepArgs& a, int64_t, int, cudaStream_t)
{
    g_seqs = a.seqs;
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

// ---- stream capture: a user object's destructor runs when the graph that holds its one reference goes --------------------
FAKE cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s)
{
    *s = g_graph ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
FAKE cudaError_t cudaStreamGetCaptureInfo(cudaStream_t stream, cudaStreamCaptureStatus* s, unsigned long long*, cudaGraph_t* graph,
                                          const cudaGraphNode_t**, size_t*)
{
    *graph = static_cast<cudaGraph_t>(g_graph);
    return cudaStreamIsCapturing(stream, s);
}
namespace { Retained g_object; }
FAKE cudaError_t cudaUserObjectCreate(cudaUserObject_t* o, void* ptr, cudaHostFn_t destroy, unsigned, unsigned)
{
    g_object = Retained{nullptr, destroy, ptr};
    *o = reinterpret_cast<cudaUserObject_t>(&g_object);
    return cudaSuccess;
}
FAKE cudaError_t cudaGraphRetainUserObject(cudaGraph_t graph, cudaUserObject_t, unsigned, unsigned)
{
    g_retained.push_back(Retained{graph, g_object.destroy, g_object.ptr});
    return cudaSuccess;
}
