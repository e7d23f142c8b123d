// A CUDA runtime without a device, for tests of the library's host side: it is
// preloaded in front of libcudart, keeps device memory in host memory, runs no
// kernel and writes one line per call of interest to the file FAKE_CUDART_LOG:
//
//   L stream index clock stale yacc panels name K...   a kernel launch: the stream and
//        its launch count, the launches of every stream that come before it
//        (comma-separated counts), whether its descriptors or its work list are
//        freed memory or missing, the bytes behind the first one's yacc and behind the LD
//        panels of each (comma-separated), the kernel's name and the supernodes
//        of its work list
//   G / B / I / T       graph launch, begin of capture, instantiation, record of a timing event
//   H                   copy from host memory on a stream that the caller captures
//
// A captured launch is logged like an issued one.  fake_fail(what, n) makes the
// next n begins of capture (1), instantiations (2) or cluster launches and
// launches of k_adj_gemm (3) fail, (4) the n-th allocation from
// now on; every timed run takes 1 ms, those of the
// autotuner's next fake_slow(n) candidates 2.  fake_capturing(st): the stream
// that the caller captures.
#include <cuda_runtime.h>
#include <cxxabi.h>

#include <algorithm>
#include <math.h>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <set>
#include <string>
#include <vector>

using std::isfinite;
#include "common.cuh"

namespace {
struct Alloc { size_t bytes; bool live; };
std::map<char *, Alloc> g_mem;
std::map<const void *, std::string> g_name;
std::map<cudaStream_t, int> g_id;
std::vector<std::vector<int>> g_clock;      // per stream: launches known to come before its next one
std::map<cudaEvent_t, std::vector<int>> g_event;
std::set<cudaEvent_t> g_timing;
int g_fail[5];
cudaError_t g_last = cudaSuccess;            // as cudaGetLastError returns it
uintptr_t g_next = 0x1000;

FILE *out() {
    static FILE *f = std::fopen(std::getenv("FAKE_CUDART_LOG"), "a");
    return f;
}
template <typename H> H handle() { return reinterpret_cast<H>(g_next += 16); }
int id(cudaStream_t st) {
    auto it = g_id.emplace(st, (int)g_id.size()).first;
    if ((int)g_clock.size() <= it->second) g_clock.resize(it->second + 1);
    return it->second;
}
std::pair<char *const, Alloc> *find(const void *p) {
    auto it = g_mem.upper_bound((char *)p);
    if (it == g_mem.begin()) return nullptr;
    --it;
    return (const char *)p < it->first + it->second.bytes ? &*it : nullptr;
}
void merge(std::vector<int> &a, const std::vector<int> &b) {
    if (a.size() < b.size()) a.resize(b.size());
    for (size_t i = 0; i < b.size(); i++) a[i] = std::max(a[i], b[i]);
}

cudaError_t fails(int what) {
    if (g_fail[what] <= 0) return cudaSuccess;
    g_fail[what]--;
    return g_last = cudaErrorUnknown;
}

cudaError_t launch(const void *fun, void **args, cudaStream_t st, bool cluster) {
    const int s = id(st);
    std::vector<int> &c = g_clock[s];
    if ((int)c.size() <= s) c.resize(s + 1);
    const std::vector<int> before = c;
    const std::string &name = g_name[fun];
    auto has = [&](const char *x) { return name.find(x) != std::string::npos; };
    if ((cluster || has("k_adj_gemm")) && fails(3) != cudaSuccess) return cudaErrorUnknown;
    const char *descs = *static_cast<const char **>(args[0]);
    int stale = 0;
    long long yacc = -1;
    std::string panels = "-";
    if (auto *a = find(descs)) {
        const char *end = a->first + std::min<size_t>(a->second.bytes, 1 << 20);
        for (const char *w = a->first; w + 8 <= end; w += 8) {
            auto *t = find(*reinterpret_cast<void *const *>(w));
            stale |= t && !t->second.live;
        }
        const auto *d = reinterpret_cast<const selinv::ProbDesc *>(descs);
        const void *list = *static_cast<void *const *>(args[1]);
        auto *t = find(list);
        stale |= !list || (t && !t->second.live);
        if (a->second.bytes % sizeof(*d) == 0 && d->lu) stale |= !d->LDu || !d->Vt || !d->Zu || !d->Ut;
        if (has("k_selinv_oz")) {
            auto *t = find(d->yacc);
            yacc = t ? (long long)t->second.bytes : 0;
        }
        if (a->second.bytes % sizeof(*d) == 0)
            for (size_t i = 0; i < a->second.bytes / sizeof(*d); i++) {
                auto *t = find(d[i].LD);
                panels += "," + std::to_string(t ? t->second.bytes : 0);
            }
    }
    std::fprintf(out(), "L %d %d ", s, ++c[s]);
    for (size_t i = 0; i < before.size(); i++) std::fprintf(out(), "%s%d", i ? "," : "", before[i]);
    if (before.empty()) std::fprintf(out(), "0");
    std::fprintf(out(), " %d %lld %s %s", stale, yacc, panels.c_str(), name.c_str());
    // work lists: (problem, K), (problem, K << 8 | part), Item
    const bool k = has("k_linv<"), k8 = has("k_linv_cols") || has("k_dinv") || has("_digits");
    const bool item = !k && !k8 && !has("reduce") && (has("k_fma_") || has("k_lhat") || has("k_selinv") || has("k_diag"));
    std::set<int> ks;
    if (k || k8 || item) {
        const int *w = *static_cast<int **>(args[1]);
        const int n = *static_cast<int *>(args[2]);
        if (find(w))
            for (int i = 0; i < n; i++) ks.insert(item ? w[4 * i + 1] : (k8 ? w[2 * i + 1] >> 8 : w[2 * i + 1]));
    }
    for (int x : ks) std::fprintf(out(), " %d", x);
    std::fprintf(out(), "\n");
    std::fflush(out());
    return cudaSuccess;
}
void note(const char *what) {
    std::fprintf(out(), "%s\n", what);
    std::fflush(out());
}
}  // namespace

// A handle (the library makes them with the nothrow form) gets the address of the
// last one of its size that was given back.
static std::map<void *, size_t> g_handles;
static std::multimap<size_t, void *> g_given_back;
void *operator new(size_t n, const std::nothrow_t &) noexcept {
    auto it = g_given_back.find(n);
    void *p = it != g_given_back.end() ? it->second : std::malloc(n);
    if (it != g_given_back.end()) g_given_back.erase(it);
    g_handles[p] = n;
    return p;
}
void operator delete(void *p) noexcept {
    auto it = p ? g_handles.find(p) : g_handles.end();
    if (it == g_handles.end()) return std::free(p);
    g_given_back.emplace(it->second, p);
    g_handles.erase(it);
}
void operator delete(void *p, size_t) noexcept { operator delete(p); }

extern "C" {
static int g_slow, g_refused;
void fake_fail(int what, int n) { g_fail[what] = n; g_refused = 0; }
static cudaStream_t g_capturing;
void fake_capturing(cudaStream_t st) { g_capturing = st; }
void fake_slow(int candidates) { g_slow = 2 * candidates; }   // two timed runs each

void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *fun, char *, const char *device_name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {
    int status = 0;
    char *d = abi::__cxa_demangle(device_name, nullptr, nullptr, &status);
    std::string n = status == 0 ? d : device_name;
    std::free(d);
    n = n.substr(0, n.find("(selinv"));          // without the parameters
    std::replace(n.begin(), n.end(), ' ', '_');
    g_name[fun] = n;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fun) { *k = (cudaKernel_t)fun; return cudaSuccess; }
static dim3 g_grid, g_block;
static size_t g_shared;
static void *g_stream;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sh, struct CUstream_st *st) { g_grid = g; g_block = b; g_shared = sh; g_stream = st; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *sh, void *st) {
    *g = g_grid; *b = g_block; *sh = g_shared; *static_cast<void **>(st) = g_stream;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **args, size_t, cudaStream_t st) { return launch((const void *)k, args, st, false); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *cfg, const void *fun, void **args) { return launch(fun, args, cfg->stream, true); }

cudaError_t cudaMalloc(void **p, size_t n) {
    if (g_fail[4] > 0 && --g_fail[4] == 0) {
        g_fail[4] = 1;                           // (and the retry after the caches have been emptied)
        if (++g_refused == 2) g_fail[4] = g_refused = 0;
        return g_last = cudaErrorMemoryAllocation;
    }
    if (posix_memalign(p, 256, n ? n : 1)) return cudaErrorMemoryAllocation;
    g_mem[(char *)*p] = {n ? n : 1, true};
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {                  // (the address stays taken: a stale one is recognized)
    auto it = g_mem.find((char *)p);
    if (it != g_mem.end()) it->second.live = false;
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
    if (k == cudaMemcpyHostToDevice && st && st == g_capturing) note("H");
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) { if (n <= 64) std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
    std::memset(a, 0, sizeof(*a));
    a->type = find(p) ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) { static double scratch[128 * 128]; *p = scratch; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) { *n = 1; return cudaSuccess; }

cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = handle<cudaStream_t>(); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t st, cudaStreamCaptureStatus *s) {
    *s = st && st == g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { const int i = id(s); merge(g_clock[i], g_event[e]); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { g_timing.insert(*e = handle<cudaEvent_t>()); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = handle<cudaEvent_t>(); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    if (g_timing.count(e)) note("T");
    const int i = id(s);
    g_event[e] = g_clock[i];
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = g_slow-- > 0 ? 2.0f : 1.0f; return cudaSuccess; }

cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { note("B"); return fails(1); }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { *g = handle<cudaGraph_t>(); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { note("I"); *x = handle<cudaGraphExec_t>(); return fails(2); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { note("G"); return cudaSuccess; }
cudaError_t cudaGraphGetEdges(cudaGraph_t, cudaGraphNode_t *, cudaGraphNode_t *, cudaGraphEdgeData *, size_t *n) { *n = 0; return cudaSuccess; }
cudaError_t cudaGraphNodeGetType(cudaGraphNode_t, cudaGraphNodeType *t) { *t = cudaGraphNodeTypeKernel; return cudaSuccess; }
cudaError_t cudaGraphAddDependencies(cudaGraph_t, const cudaGraphNode_t *, const cudaGraphNode_t *, const cudaGraphEdgeData *, size_t) { return cudaSuccess; }
cudaError_t cudaGraphRemoveDependencies(cudaGraph_t, const cudaGraphNode_t *, const cudaGraphNode_t *, const cudaGraphEdgeData *, size_t) { return cudaSuccess; }
}
