// Runs of kernels launched as one graph.  On the bench platform a kernel launch costs the host 2.1 us, a graph launch 1.0 us
// however many kernels it holds, and changing the arguments of one of its kernels 0.28 us; building a graph of 1 to 12
// kernels costs 65 to 90 us (cudaGraphInstantiate 60 to 70, the first launch 2 to 20 more than a later one).  On the device,
// a kernel of a graph starts 0.8 us after the one before it.  The calls whose mini-batches are bound by the host collect
// their kernels (LaunchBatch) and launch them together; the graphs are kept (LaunchCache) and launched again as they are, or
// with the arguments that differ, as long as the call makes the same kernels.
#include <cstring>
#include <new>

#include "hl_common.cuh"

namespace hl {

namespace {

constexpr int kMaxNodes = 12, kMaxArgBytes = 4096, kMaxParams = 160;
constexpr int64_t kPlainNs = 2100, kGraphNs = 1000, kUpdateNs = 280, kBuildNs = 75000;

struct Node {
    const void* func;
    dim3 grid, block;
    unsigned smem;
    int cluster;                       // CTAs per cluster; 0: none
    int first_param, n_params;
    int first_byte, n_bytes;           // of its arguments, packed
};

// the kernels of one run, with copies of their arguments
struct Recording {
    int n = 0, params = 0, bytes = 0;
    Node node[kMaxNodes];
    uint16_t param_at[kMaxParams];     // offset of every argument in `arg`
    alignas(16) unsigned char arg[kMaxArgBytes];

    void clear() { n = params = bytes = 0; }

    bool add(const void* func, dim3 grid, dim3 block, size_t smem, int cluster, void** args, const uint32_t* sizes,
             int n_args) {
        int need = 0;
        for (int i = 0; i < n_args; ++i) need += (int)((sizes[i] + 15) & ~15u);
        if (n == kMaxNodes || params + n_args > kMaxParams || bytes + need > kMaxArgBytes) return false;
        Node& d = node[n++];
        d.func = func;
        d.grid = grid;
        d.block = block;
        d.smem = (unsigned)smem;
        d.cluster = cluster;
        d.first_param = params;
        d.n_params = n_args;
        d.first_byte = bytes;
        d.n_bytes = need;
        std::memset(arg + bytes, 0, need);                   // (padding compares equal)
        for (int i = 0; i < n_args; ++i) {
            param_at[params++] = (uint16_t)bytes;
            std::memcpy(arg + bytes, args[i], sizes[i]);
            bytes += (int)((sizes[i] + 15) & ~15u);
        }
        return true;
    }

    void kernel_params(int i, cudaKernelNodeParams* p, void** ptrs) {
        const Node& d = node[i];
        for (int k = 0; k < d.n_params; ++k) ptrs[k] = arg + param_at[d.first_param + k];
        std::memset(p, 0, sizeof(*p));
        p->func = const_cast<void*>(d.func);
        p->gridDim = d.grid;
        p->blockDim = d.block;
        p->sharedMemBytes = d.smem;
        p->kernelParams = ptrs;
    }
};

bool same_shape(const Node& a, const Node& b) {
    return a.grid.x == b.grid.x && a.grid.y == b.grid.y && a.grid.z == b.grid.z && a.block.x == b.block.x &&
           a.block.y == b.block.y && a.block.z == b.block.z && a.smem == b.smem;
}

bool same_node(const Recording& a, const Recording& b, int i) {
    const Node &x = a.node[i], &y = b.node[i];
    return same_shape(x, y) && x.n_bytes == y.n_bytes &&
           std::memcmp(a.arg + x.first_byte, b.arg + y.first_byte, x.n_bytes) == 0;
}

cudaError_t launch_now(const void* func, dim3 grid, dim3 block, size_t smem, int cluster, void** args, cudaStream_t stream) {
    if (cluster == 0) return cudaLaunchKernel(func, grid, block, args, smem, stream);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, func, args);
}

}  // namespace

// One kept graph: the recording it was last launched with, and its executable form.
struct LaunchCache::Entry {
    Recording rec;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaGraphNode_t node[kMaxNodes];
    uint64_t used = 0;

    ~Entry() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
    }

    bool same_arguments(const Recording& r) const {
        for (int i = 0; i < r.n; ++i)
            if (!same_node(rec, r, i)) return false;
        return true;
    }

    cudaError_t build(const Recording& r) {
        rec = r;
        cudaError_t e = cudaGraphCreate(&graph, 0);
        for (int i = 0; i < rec.n && e == cudaSuccess; ++i) {
            cudaKernelNodeParams p;
            void* ptrs[kMaxParams];
            rec.kernel_params(i, &p, ptrs);
            e = cudaGraphAddKernelNode(&node[i], graph, i ? &node[i - 1] : nullptr, i ? 1 : 0, &p);
            if (e == cudaSuccess && rec.node[i].cluster) {
                cudaKernelNodeAttrValue v = {};
                v.clusterDim.x = rec.node[i].cluster;
                v.clusterDim.y = v.clusterDim.z = 1;
                e = cudaGraphKernelNodeSetAttribute(node[i], cudaLaunchAttributeClusterDimension, &v);
            }
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
        return e;
    }

    // the arguments that differ from the last launch's (future launches only: one in flight keeps its own)
    cudaError_t update(const Recording& r, int* changed) {
        for (int i = 0; i < r.n; ++i) {
            if (same_node(rec, r, i)) continue;
            ++*changed;
            cudaKernelNodeParams p;
            void* ptrs[kMaxParams];
            const_cast<Recording&>(r).kernel_params(i, &p, ptrs);
            const cudaError_t e = cudaGraphExecKernelNodeSetParams(exec, node[i], &p);
            if (e != cudaSuccess) return e;
        }
        rec = r;
        return cudaSuccess;
    }
};

// The kernels of one run, and the graphs of them that there are.
struct LaunchCache::List {
    List* next = nullptr;
    uint64_t used = 0;
    int n = 0, graphs = 0;
    const void* func[kMaxNodes];
    int cluster[kMaxNodes];
    Entry* graph[kMaxVariants] = {};

    ~List() {
        for (int i = 0; i < graphs; ++i) delete graph[i];
    }
    bool has(const Recording& r) const {
        if (n != r.n) return false;
        for (int i = 0; i < n; ++i)
            if (func[i] != r.node[i].func || cluster[i] != r.node[i].cluster) return false;
        return true;
    }
    void drop(Entry* e) {
        for (int i = 0; i < graphs; ++i)
            if (graph[i] == e) {
                graph[i] = graph[--graphs];
                delete e;
                return;
            }
    }
};

LaunchCache::LaunchCache(int variants) : variants_(variants < kMaxVariants ? variants : kMaxVariants) {}
LaunchCache::~LaunchCache() {
    while (lists_) {
        List* l = lists_;
        lists_ = l->next;
        delete l;
    }
}

// the list of these kernels; a new one if they come for the first time (nullptr: no memory for it)
LaunchCache::List* LaunchCache::list_of(const void* recording) {
    const Recording& r = *static_cast<const Recording*>(recording);
    int n = 0;
    List** oldest = nullptr;
    for (List** l = &lists_; *l; l = &(*l)->next, ++n) {
        if ((*l)->has(r)) return *l;
        if (!oldest || (*l)->used < (*oldest)->used) oldest = l;
    }
    if (n >= kMaxLists) {
        List* gone = *oldest;
        *oldest = gone->next;
        delete gone;
    }
    List* l = new (std::nothrow) List();
    if (!l) return nullptr;
    l->n = r.n;
    for (int i = 0; i < r.n; ++i) {
        l->func[i] = r.node[i].func;
        l->cluster[i] = r.node[i].cluster;
    }
    l->next = lists_;
    lists_ = l;
    return l;
}

namespace {

cudaError_t launch_one_by_one(Recording& r, cudaStream_t stream) {
    for (int i = 0; i < r.n; ++i) {
        cudaKernelNodeParams p;
        void* ptrs[kMaxParams];
        r.kernel_params(i, &p, ptrs);
        const cudaError_t e = launch_now(p.func, p.gridDim, p.blockDim, p.sharedMemBytes, r.node[i].cluster, ptrs, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// what the calling thread is collecting
struct Collecting {
    LaunchCache* cache = nullptr;
    bool build_only = false;
    cudaStream_t stream = nullptr;
    cudaError_t failed = cudaSuccess;
    Recording rec;
};
thread_local Collecting t_now;

}  // namespace

// Launches a recording: as the kept graph that had these kernels and arguments, or as one with these kernels whose arguments
// are brought up to date (the one not used for longest), or kernel by kernel.
//
// Building a graph costs as much as some 30 plain launches, in the call that does it.  So none is built before the plain
// launches of this cache (and, for one more graph of kernels that have one, the arguments changed) have cost that much more
// than graphs would have: a program that makes a call a few times never pays for a graph, one that makes it for ever pays for
// plain launches twice at most, and graphs come one at a time, however many runs of kernels a call makes.
cudaError_t LaunchCache::launch(const void* recording, cudaStream_t stream) {
    Recording& r = *const_cast<Recording*>(static_cast<const Recording*>(recording));
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &capturing) != cudaSuccess || capturing != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return launch_one_by_one(r, stream);
    }
    std::lock_guard<std::mutex> lock(mutex_);
    List* l = list_of(recording);
    if (!l) return launch_one_by_one(r, stream);
    l->used = ++tick_;
    Entry *e = nullptr, *oldest = nullptr;
    for (int i = 0; i < l->graphs && !e; ++i) {
        if (l->graph[i]->same_arguments(r)) e = l->graph[i];
        if (!oldest || l->graph[i]->used < oldest->used) oldest = l->graph[i];
    }
    if (!e && l->graphs < variants_ && lost_ns_ >= kBuildNs) {
        lost_ns_ = 0;
        e = new (std::nothrow) Entry();
        if (e && e->build(r) == cudaSuccess) {
            l->graph[l->graphs++] = e;
        } else {                                             // (no memory for it: there are other ways)
            delete e;
            e = nullptr;
            cudaGetLastError();
        }
    }
    int64_t lost = 0;
    if (!e && oldest) {
        int changed = 0;
        e = oldest;
        if (e->update(r, &changed) != cudaSuccess) {
            l->drop(e);
            e = nullptr;
            cudaGetLastError();
        }
        if (l->graphs < variants_) lost = kUpdateNs * changed;
    }
    if (!e) lost = (kPlainNs - kUpdateNs) * r.n - kGraphNs;
    lost_ns_ = lost_ns_ + lost < kBuildNs ? lost_ns_ + lost : kBuildNs;
    if (!e) return launch_one_by_one(r, stream);
    e->used = ++tick_;
    return cudaGraphLaunch(e->exec, stream);
}

void LaunchCache::build(const void* recording) {
    std::lock_guard<std::mutex> lock(mutex_);
    List* l = list_of(recording);
    if (!l || l->graphs) return;
    Entry* e = new (std::nothrow) Entry();
    if (e && e->build(*static_cast<const Recording*>(recording)) == cudaSuccess) {
        l->graph[l->graphs++] = e;
    } else {
        delete e;
        cudaGetLastError();
    }
}

cudaError_t launch_flush() {
    Collecting& c = t_now;
    if (!c.cache || c.rec.n == 0) return cudaSuccess;
    if (c.build_only) {
        c.cache->build(&c.rec);
        c.rec.clear();
        return cudaSuccess;
    }
    const cudaError_t e = c.cache->launch(&c.rec, c.stream);
    c.rec.clear();
    if (e != cudaSuccess && c.failed == cudaSuccess) c.failed = e;
    return e;
}

cudaError_t launch_kernel(const void* func, dim3 grid, dim3 block, size_t smem, int cluster, void** args,
                          const uint32_t* sizes, int n_args, cudaStream_t stream) {
    Collecting& c = t_now;
    if (!c.cache) return launch_now(func, grid, block, smem, cluster, args, stream);
    if (c.stream != stream) {
        launch_flush();
        c.stream = stream;
    }
    if (c.rec.add(func, grid, block, smem, cluster, args, sizes, n_args)) return cudaSuccess;
    const cudaError_t e = launch_flush();
    if (e != cudaSuccess) return e;
    if (c.rec.add(func, grid, block, smem, cluster, args, sizes, n_args) || c.build_only) return cudaSuccess;
    return launch_now(func, grid, block, smem, cluster, args, stream);
}

bool launches_build_only() { return t_now.cache && t_now.build_only; }

namespace {
__global__ void __launch_bounds__(256) k_clear_words(uint32_t* p, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) p[i] = 0;
}
}  // namespace

// a kernel where it can be one more of a graph, else a memset
cudaError_t clear_words(uint32_t* p, int64_t n_words, cudaStream_t stream) {
    if (!t_now.cache) return cudaMemsetAsync(p, 0, sizeof(uint32_t) * n_words, stream);
    note_launches(1);
    return launch(k_clear_words, grid_for(n_words, 256, 296), 256, stream, p, n_words);
}

LaunchBatch::LaunchBatch(LaunchCache* cache, bool build_only) : mine_(cache != nullptr && t_now.cache == nullptr) {
    if (!mine_) return;
    t_now.cache = cache;
    t_now.build_only = build_only;
    t_now.stream = nullptr;
    t_now.failed = cudaSuccess;
    t_now.rec.clear();
}

int32_t LaunchBatch::end(int32_t st) {
    if (!mine_) return st;
    mine_ = false;
    launch_flush();
    t_now.cache = nullptr;
    return st != HL_OK || t_now.failed == cudaSuccess ? st : HL_ECUDA;
}

LaunchBatch::~LaunchBatch() { (void)end(); }

}  // namespace hl
