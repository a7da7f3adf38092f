// A stand-in for the CUDA runtime, linked with the library's own object files: what the library queues is written down
// instead of run, and any call can be made to fail.  Device memory is whatever host memory a test hands out; memset and
// memcpy of it are done at once, kernels are only recorded.
//
// Every line of the log is one thing put on a stream, in the order of the calls; the kernels of a graph appear when the
// graph is launched, with the arguments its nodes had then.
#include <cuda_runtime.h>
#include <cxxabi.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <set>
#include <string>
#include <vector>

namespace {

struct Kernel {
    std::string name;                       // without namespaces and parameter list
    std::vector<size_t> params;             // bytes of every parameter that are compared
};
struct Node {
    const void* func;
    cudaKernelNodeParams shape;
    int cluster;
    std::vector<std::string> args;
};
struct Graph {
    std::vector<Node> nodes;
};
struct NodeRef {                            // what a cudaGraphNode_t points to (never freed)
    Graph* graph;
    size_t at;
};
NodeRef& ref(cudaGraphNode_t n) { return *reinterpret_cast<NodeRef*>(n); }

std::map<const void*, Kernel> kernels;
std::vector<std::string> lines;
std::map<std::string, int> calls, fail_at;  // calls of a function so far; which of them fails (-1: every one)
std::string fail_kernel;                    // launches of this kernel fail
std::set<const void*> capturing, device_memory;
long handles = 0x1000;

bool fails(const char* name) {
    const int n = ++calls[name];
    const auto it = fail_at.find(name);
    return it != fail_at.end() && (it->second < 0 || it->second == n);
}
cudaError_t result(const char* name) { return fails(name) ? cudaErrorUnknown : cudaSuccess; }

// "int const*" -> 8, "hl::PairArgs" -> 64 (its leading bytes)
size_t size_of(std::string t) {
    while (!t.empty() && t.front() == ' ') t.erase(0, 1);
    if (t.find('*') != std::string::npos) return 8;
    const std::pair<const char*, size_t> known[] = {
        {"PairArgs", 64}, {"PlaceArgs", 64}, {"ForwardRows", 48}, {"TableMap", 32}, {"ColdMarks", 40}, {"BitmapProbe", 8},
        {"HashProbe", 24}};
    for (const auto& k : known)
        if (t.find(k.first) != std::string::npos) return k.second;
    if (t == "bool") return 1;
    if (t == "int" || t == "unsigned int" || t == "float") return 4;
    if (t == "long" || t == "unsigned long" || t == "long long" || t == "unsigned long long") return 8;
    abort();
}

Kernel describe(const char* mangled) {
    int status = 0;
    char* text = abi::__cxa_demangle(mangled, nullptr, nullptr, &status);
    if (!text) abort();
    std::string s(text);
    free(text);
    Kernel k;
    const size_t close = s.rfind(')');
    size_t open = close, depth = 0;
    std::vector<size_t> commas;
    for (size_t i = close;; --i) {          // the parameter list, from its end
        const char c = s[i];
        if (c == ')' || c == '>') ++depth;
        if (c == '(' || c == '<') --depth;
        if (c == ',' && depth == 1) commas.insert(commas.begin(), i);
        if (depth == 0) {
            open = i;
            break;
        }
    }
    size_t at = open + 1;
    commas.push_back(close);
    for (size_t c : commas) {
        if (c > at) k.params.push_back(size_of(s.substr(at, c - at)));
        at = c + 1;
    }
    const size_t first = s.find("k_");
    for (size_t i = first; i < open; ++i)
        if (s[i] != ' ') k.name += s[i];
    return k;
}

std::vector<std::string> copy_args(const void* func, void** args) {
    std::vector<std::string> out;
    const Kernel& k = kernels.at(func);
    for (size_t i = 0; i < k.params.size(); ++i) out.emplace_back(static_cast<const char*>(args[i]), k.params[i]);
    return out;
}

std::string hex(const std::string& bytes) {
    std::string out;
    char b[3];
    for (unsigned char c : bytes) {
        snprintf(b, sizeof(b), "%02x", c);
        out += b;
    }
    return out;
}

void write_launch(const char* how, const Node& n, cudaStream_t s) {
    char head[256];
    snprintf(head, sizeof(head), "%s %p %s grid=%u block=%u smem=%u cluster=%d", how, (void*)s,
             kernels.at(n.func).name.c_str(), n.shape.gridDim.x, n.shape.blockDim.x, n.shape.sharedMemBytes, n.cluster);
    std::string line(head);
    for (const std::string& a : n.args) line += " " + hex(a);
    lines.push_back(line);
}

bool kernel_fails(const void* func) { return !fail_kernel.empty() && kernels.at(func).name.find(fail_kernel) == 0; }

void* handle() { return reinterpret_cast<void*>(handles += 0x10); }

}  // namespace

extern "C" {

// ---- for the tests ----
void fake_reset() {
    lines.clear();
    calls.clear();
    fail_at.clear();
    fail_kernel.clear();
    capturing.clear();
    device_memory.clear();
    handles = 0x1000;                       // (streams and events of two runs have the same names)
}
void fake_fail(const char* function, int nth) {
    calls[function] = 0;
    if (nth) fail_at[function] = nth;
    else fail_at.erase(function);
}
void fake_fail_kernel(const char* name) { fail_kernel = name ? name : ""; }
void fake_capture(void* stream, int on) {
    if (on) capturing.insert(stream);
    else capturing.erase(stream);
}
void fake_device_memory(const void* p) { device_memory.insert(p); }
int fake_calls(const char* function) { return calls[function]; }
int fake_lines() { return (int)lines.size(); }
const char* fake_line(int i) { return lines[i].c_str(); }

// ---- registration (called when the library is loaded) ----
void** __cudaRegisterFatBinary(void*) { return new void*; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* device_name, int, void*, void*, void*, void*, int*) {
    kernels[host] = describe(device_name);
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { abort(); }      // (nothing uses <<< >>>)

// ---- the runtime ----
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
    *v = 148;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetStreamPriorityRange(int* lo, int* hi) {
    *lo = 0;
    *hi = -5;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return result("cudaDeviceSynchronize"); }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void**, const void*) { return cudaErrorUnknown; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    if (!device_memory.count(p)) return cudaErrorUnknown;
    memset(a, 0, sizeof(*a));
    a->type = cudaMemoryTypeDevice;
    return cudaSuccess;
}
cudaError_t cudaMallocManaged(void**, size_t, unsigned) { return cudaErrorMemoryAllocation; }
cudaError_t cudaHostAlloc(void**, size_t, unsigned) { return cudaErrorMemoryAllocation; }
cudaError_t cudaMemAdvise(const void*, size_t, cudaMemoryAdvise, int) { return cudaErrorUnknown; }
cudaError_t cudaMemPrefetchAsync(const void*, size_t, int, cudaStream_t) { return cudaErrorUnknown; }
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaFreeHost(void*) { return cudaSuccess; }

cudaError_t cudaMemset(void* p, int v, size_t n) {
    memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) {
    if (fails("cudaMemsetAsync")) return cudaErrorUnknown;
    char line[160];
    snprintf(line, sizeof(line), "memset %p at=%p value=%d bytes=%zu", (void*)s, p, v, n);
    lines.push_back(line);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    char line[160];
    snprintf(line, sizeof(line), "copy %p to=%p from=%p bytes=%zu", (void*)st, d, s, n);
    lines.push_back(line);
    return cudaSuccess;
}

cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) {
    *s = static_cast<cudaStream_t>(handle());
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return result("cudaStreamSynchronize"); }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* st) {
    *st = capturing.count(s) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
    *e = static_cast<cudaEvent_t>(handle());
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 0.f;
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    if (fails("cudaEventRecord")) return cudaErrorUnknown;
    char line[96];
    snprintf(line, sizeof(line), "record %p event=%p", (void*)s, (void*)e);
    lines.push_back(line);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    if (fails("cudaStreamWaitEvent")) return cudaErrorUnknown;
    char line[96];
    snprintf(line, sizeof(line), "wait %p event=%p", (void*)s, (void*)e);
    lines.push_back(line);
    return cudaSuccess;
}

cudaError_t cudaLaunchKernel(const void* func, dim3 grid, dim3 block, void** args, size_t smem, cudaStream_t s) {
    if (fails("cudaLaunchKernel") || kernel_fails(func)) return cudaErrorLaunchOutOfResources;
    Node n{func, {}, 0, copy_args(func, args)};
    n.shape.gridDim = grid;
    n.shape.blockDim = block;
    n.shape.sharedMemBytes = (unsigned)smem;
    write_launch("plain", n, s);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* func, void** args) {
    if (fails("cudaLaunchKernel") || kernel_fails(func)) return cudaErrorLaunchOutOfResources;
    Node n{func, {}, 0, copy_args(func, args)};
    n.shape.gridDim = c->gridDim;
    n.shape.blockDim = c->blockDim;
    n.shape.sharedMemBytes = (unsigned)c->dynamicSmemBytes;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) n.cluster = (int)c->attrs[i].val.clusterDim.x;
    write_launch("plain", n, c->stream);
    return cudaSuccess;
}

cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) {
    if (fails("cudaGraphCreate")) return cudaErrorUnknown;
    *g = reinterpret_cast<cudaGraph_t>(new Graph);
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
    delete reinterpret_cast<Graph*>(g);
    return cudaSuccess;
}
cudaError_t cudaGraphAddKernelNode(cudaGraphNode_t* node, cudaGraph_t g, const cudaGraphNode_t* deps, size_t n_deps,
                                   const cudaKernelNodeParams* p) {
    Graph& graph = *reinterpret_cast<Graph*>(g);
    if (n_deps != (graph.nodes.empty() ? 0u : 1u)) abort();              // a chain is all the library makes
    if (n_deps && ref(deps[0]).at + 1 != graph.nodes.size()) abort();
    *node = reinterpret_cast<cudaGraphNode_t>(new NodeRef{&graph, graph.nodes.size()});
    graph.nodes.push_back(Node{p->func, *p, 0, copy_args(p->func, p->kernelParams)});
    return cudaSuccess;
}
cudaError_t cudaGraphKernelNodeSetAttribute(cudaGraphNode_t n, cudaLaunchAttributeID id, const cudaLaunchAttributeValue* v) {
    if (id == cudaLaunchAttributeClusterDimension) ref(n).graph->nodes.at(ref(n).at).cluster = (int)v->clusterDim.x;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
    if (fails("cudaGraphInstantiate")) return cudaErrorMemoryAllocation;
    *e = reinterpret_cast<cudaGraphExec_t>(new Graph(*reinterpret_cast<Graph*>(g)));
    return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
    calls["cudaGraphExecDestroy"]++;
    delete reinterpret_cast<Graph*>(e);
    return cudaSuccess;
}
cudaError_t cudaGraphExecKernelNodeSetParams(cudaGraphExec_t e, cudaGraphNode_t node, const cudaKernelNodeParams* p) {
    if (fails("cudaGraphExecKernelNodeSetParams")) return cudaErrorUnknown;
    Node& n = reinterpret_cast<Graph*>(e)->nodes.at(ref(node).at);
    if (n.func != p->func) abort();
    n.shape = *p;
    n.args = copy_args(p->func, p->kernelParams);
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s) {
    if (fails("cudaGraphLaunch")) return cudaErrorUnknown;
    for (const Node& n : reinterpret_cast<Graph*>(e)->nodes) write_launch("graph", n, s);
    return cudaSuccess;
}

}  // extern "C"
