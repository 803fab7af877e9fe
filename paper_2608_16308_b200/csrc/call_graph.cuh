// The kernels of one library call, collected first and then submitted together.
//
// What bounds a short call is its launches.  On the B200 machine a kernel launch costs 2.3 - 2.9 us of the
// calling thread; a kernel that waits for the one before it to end starts on a 2 us grid (one 8 us
// kernel after the other: 10.24 us a call), while one launched with the programmatic
// attribute starts as its predecessor drains (8.44 us).  And a graph of the same kernels launches
// in 1.2 us, plus 0.25 us for every node whose arguments or grid changed, with the programmatic
// edges inside it but not in front of it.  So:
//   * the stream still has work (cudaStreamQuery, 0.2 us): the calling thread is ahead of the GPU. The kernels are
//     launched one by one, every one of them -- the first too -- with the programmatic attribute.  (Each executes pdl_wait before it
//     touches anything that an earlier kernel may still write; what k_finish and the batched decode over columns do before it -- a
//     ticket, the caller's x -- is sound because the kernel in front of them in the call had itself waited.)
//   * the stream is idle: the call's latency counts, and the host's share of it is the largest. From
//     the second call of the same sequence of kernels on, one launch of a graph that the handle keeps
//     (cudaGraphExecKernelNodeSetParams takes over the new arguments).  The call that builds the graph pays for it, once per handle
//     and sequence: 100 - 220 us of the calling thread (16 - 28 us launched one by one, 5 us from then on; three kernels).
//
// A handle keeps at most CALL_GRAPHS graphs, one per sequence of kernels (the paths that a handle's
// calls take), and replaces the least recently used one.  A sequence's first call on an idle stream
// launches its kernels one by one, so a handle that is used once never builds a graph; so do calls
// on a stream that is being captured (the kernels then become nodes of the caller's graph) and calls
// with kernel timing switched on (events between the kernels).
#pragma once

#include <string.h>

#include <new>

#include "internal.cuh"

namespace dbs {

constexpr int CALL_MAX_KERNELS = 8;
constexpr int CALL_MAX_ARGS = 16;
constexpr int CALL_ARG_BYTES = 1024;     // argument bytes of one kernel, at most (the Device struct is most of it)
constexpr int CALL_GRAPHS = 8;

struct CallNode {
    const void *func;
    dim3 grid, block;
    unsigned smem;
    int pdl;                             // may start while the kernel before it drains
    int n_args;
    int bytes;                           // argument bytes used
    int offset[CALL_MAX_ARGS];
    alignas(16) uint8_t args[CALL_ARG_BYTES];

    bool same_kernel(const CallNode &o) const {
        return func == o.func && block.x == o.block.x && smem == o.smem && pdl == o.pdl && n_args == o.n_args && bytes == o.bytes;
    }
    bool same_launch(const CallNode &o) const { return grid.x == o.grid.x && memcmp(args, o.args, (size_t)bytes) == 0; }
    void pointers(void **p) { for (int i = 0; i < n_args; ++i) p[i] = args + offset[i]; }
    cudaKernelNodeParams params(void **p) {
        cudaKernelNodeParams k = {};
        pointers(p);
        k.func = const_cast<void *>(func);
        k.gridDim = grid;
        k.blockDim = block;
        k.sharedMemBytes = smem;
        k.kernelParams = p;
        return k;
    }
};

// One call's kernels, in order.  Lives on the caller's stack.
struct CallList {
    int n = 0;
    int ev_before = -1, ev_after = -1;   // kernel timing: events are recorded in front of these positions
    bool overflow = false;
    CallNode node[CALL_MAX_KERNELS];

    template <typename... KArgs, typename... Args>
    void add(void (*kernel)(KArgs...), int grid, int block, size_t smem, bool pdl, Args... args) {
        static_assert(sizeof...(KArgs) == sizeof...(Args) && sizeof...(KArgs) <= CALL_MAX_ARGS, "one value per kernel parameter");
        if (n == CALL_MAX_KERNELS) { overflow = true; return; }
        CallNode &k = node[n++];
        k.func = reinterpret_cast<const void *>(kernel);
        k.grid = dim3((unsigned)grid);
        k.block = dim3((unsigned)block);
        k.smem = (unsigned)smem;
        k.pdl = pdl ? 1 : 0;
        k.n_args = 0;
        k.bytes = 0;
        (put<KArgs>(k, KArgs(args)), ...);
    }

   private:
    template <typename T> static void put(CallNode &k, T v) {
        static_assert(sizeof(T) <= CALL_ARG_BYTES - 128, "kernel argument too large");
        const int a = (int)alignof(T), o = (k.bytes + a - 1) / a * a;
        memset(k.args + k.bytes, 0, (size_t)(o - k.bytes));
        memcpy(k.args + o, &v, sizeof(T));
        k.offset[k.n_args++] = o;
        k.bytes = o + (int)sizeof(T);
    }
};

struct CallGraph {
    int n = 0;
    bool failed = false;                 // could not be built: this sequence stays with plain launches
    cudaGraphExec_t exec = nullptr;
    cudaGraph_t graph = nullptr;         // kept: its node handles name the nodes of `exec`
    cudaGraphNode_t gnode[CALL_MAX_KERNELS];
    CallNode *node = nullptr;            // as last launched (n of them)
    uint64_t used = 0;
};

struct CallGraphs {
    CallGraph g[CALL_GRAPHS];
    uint64_t clock = 0;

    static void clear(CallGraph &c) {
        if (c.exec) cudaGraphExecDestroy(c.exec);
        if (c.graph) cudaGraphDestroy(c.graph);
        delete[] c.node;
        c = CallGraph();
    }
    ~CallGraphs() { for (CallGraph &c : g) clear(c); }
};

inline cudaError_t launch_node(CallNode &k, cudaStream_t st, bool chained) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = k.grid;
    cfg.blockDim = k.block;
    cfg.dynamicSmemBytes = k.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = k.pdl || chained ? 1 : 0;
    void *p[CALL_MAX_ARGS];
    k.pointers(p);
    return cudaLaunchKernelExC(&cfg, k.func, p);
}

// The kernels one by one; `chained`: the first one too may start while its predecessor drains.
inline int launch_plain(dbspmspv_handle_s *h, CallList &l, cudaStream_t st, bool chained = false) {
    for (int i = 0; i < l.n; ++i) {
        if (i == l.ev_before) DBS_CUDA(cudaEventRecord(h->ev[0], st));
        if (i == l.ev_after) DBS_CUDA(cudaEventRecord(h->ev[1], st));
        DBS_CUDA(launch_node(l.node[i], st, chained));
    }
    if (l.n == l.ev_before) DBS_CUDA(cudaEventRecord(h->ev[0], st));
    if (l.n == l.ev_after) DBS_CUDA(cudaEventRecord(h->ev[1], st));
    return DBSPMSPV_OK;
}

// The sequence as a graph: a chain of kernel nodes, programmatic edges where the plain launch would
// carry the stream-serialisation attribute.
inline bool build_graph(CallGraph &c, CallList &l) {
    if (cudaGraphCreate(&c.graph, 0) != cudaSuccess) { c.graph = nullptr; return false; }
    for (int i = 0; i < l.n; ++i) {
        void *p[CALL_MAX_ARGS];
        const cudaKernelNodeParams kp = l.node[i].params(p);
        if (cudaGraphAddKernelNode(&c.gnode[i], c.graph, nullptr, 0, &kp) != cudaSuccess) return false;
        if (i == 0) continue;
        cudaGraphEdgeData edge = {};
        if (l.node[i].pdl) { edge.from_port = cudaGraphKernelNodePortProgrammatic; edge.type = cudaGraphDependencyTypeProgrammatic; }
        if (cudaGraphAddDependencies_v2(c.graph, &c.gnode[i - 1], &c.gnode[i], &edge, 1) != cudaSuccess) return false;
    }
    return cudaGraphInstantiate(&c.exec, c.graph, 0) == cudaSuccess;
}

// While any stream of the process is captured in the global mode, or this thread captures one, the runtime refuses calls that a
// capture could not express -- cudaStreamQuery and cudaGraphInstantiate among them -- and ends that capture with an error.  Here they
// concern a stream that is not captured, so they are made in the relaxed mode.
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { (void)cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { (void)cudaThreadExchangeStreamCaptureMode(&mode); }
};

// Submits the kernels of one call on `st`.
inline int submit_calls(dbspmspv_handle_s *h, CallList &l, cudaStream_t st) {
    if (l.overflow) return DBSPMSPV_ERR_CUDA;
    if (l.n == 0) return DBSPMSPV_OK;
    h->kernel_launches += l.n;
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (l.ev_before >= 0 || !h->graphs || cudaStreamIsCapturing(st, &capturing) != cudaSuccess || capturing != cudaStreamCaptureStatusNone) {
        (void)cudaGetLastError();
        return launch_plain(h, l, st);
    }
    RelaxedCapture relaxed;
    if (cudaStreamQuery(st) == cudaErrorNotReady) return launch_plain(h, l, st, true);
    CallGraphs &s = *h->graphs;
    CallGraph *c = nullptr, *oldest = &s.g[0];
    for (CallGraph &q : s.g) {
        if (q.n == l.n) {
            bool same = true;
            for (int i = 0; i < l.n && same; ++i) same = q.node[i].same_kernel(l.node[i]);
            if (same) { c = &q; break; }
        }
        if (q.used < oldest->used) oldest = &q;
    }
    if (!c) {                            // first call of this sequence: remember it, launch plainly
        CallGraphs::clear(*oldest);
        oldest->node = new (std::nothrow) CallNode[l.n];
        if (oldest->node) {
            for (int i = 0; i < l.n; ++i) oldest->node[i] = l.node[i];
            oldest->n = l.n;
            oldest->used = ++s.clock;
        }
        return launch_plain(h, l, st);
    }
    c->used = ++s.clock;
    if (c->failed) return launch_plain(h, l, st);
    if (!c->exec) {
        if (!build_graph(*c, l)) {
            (void)cudaGetLastError();
            if (c->graph) cudaGraphDestroy(c->graph);
            c->graph = nullptr;
            c->exec = nullptr;
            c->failed = true;
            return launch_plain(h, l, st);
        }
        for (int i = 0; i < l.n; ++i) c->node[i] = l.node[i];
    } else {
        for (int i = 0; i < l.n; ++i) {
            if (c->node[i].same_launch(l.node[i])) continue;
            void *p[CALL_MAX_ARGS];
            const cudaKernelNodeParams kp = l.node[i].params(p);
            DBS_CUDA(cudaGraphExecKernelNodeSetParams(c->exec, c->gnode[i], &kp));
            c->node[i] = l.node[i];
        }
    }
    DBS_CUDA(cudaGraphLaunch(c->exec, st));
    return DBSPMSPV_OK;
}

}  // namespace dbs
