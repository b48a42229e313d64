// resident.cu -- launches of the multi-step kernels (resident.cuh) from captured graphs.
#include "internal.h"

namespace axl {

namespace {

// The kernels' arguments for `steps` steps (storage must outlive the use of `args`).
struct ResArgs {
    const void* doms;
    const int* map;
    unsigned* flags;
    Clock* clock;
    int steps;
    unsigned epoch;
    unsigned* taken;
    void* args[7];
    ResArgs(const Resident& r, Clock* clk, int steps_) {
        char* m = static_cast<char*>(r.scratch);
        doms = m;
        map = reinterpret_cast<const int*>(m + r.off_map);
        flags = reinterpret_cast<unsigned*>(m + r.off_flags);
        clock = clk;
        steps = steps_;
        epoch = r.epoch;
        taken = reinterpret_cast<unsigned*>(m + r.off_taken);
        int n = 0;
        args[n++] = &doms;
        if (!r.cluster) args[n++] = &map;
        if (!r.cluster && !r.slab) args[n++] = &flags;
        args[n++] = &clock;
        args[n++] = &steps;
        if (!r.cluster) {
            args[n++] = &epoch;
            args[n++] = &taken;
        }
    }
};

}  // namespace

bool resident_usable(const Resident& r, cudaStream_t stream) {
    if (!r.on) return false;
    cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &s) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return s == cudaStreamCaptureStatusNone;
}

cudaError_t resident_capture(Resident* r, Clock* clock, cudaStream_t cap) {
    ResArgs a(*r, clock, 2);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(r->grid);
    cfg.blockDim = dim3(r->threads);
    cfg.dynamicSmemBytes = r->smem;
    cfg.stream = cap;
    cudaLaunchAttribute at[1];
    if (r->cluster) {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = r->grid;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    } else {
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
    }
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return e;
    e = cudaLaunchKernelExC(&cfg, r->kernel, a.args);
    const cudaError_t e2 = cudaStreamEndCapture(cap, &r->graph);
    if (e == cudaSuccess) e = e2;
    size_t nodes = 1;
    if (e == cudaSuccess) e = cudaGraphGetNodes(r->graph, &r->node, &nodes);
    if (e == cudaSuccess && nodes != 1) e = cudaErrorUnknown;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&r->exec, r->graph, 0);
    if (e != cudaSuccess) resident_drop_graph(r);
    return e;
}

cudaError_t resident_launch(Resident* r, Clock* clock, int steps, cudaStream_t stream) {
    ResArgs a(*r, clock, steps);
    cudaKernelNodeParams p = {};
    p.func = const_cast<void*>(r->kernel);
    p.gridDim = dim3(r->grid);
    p.blockDim = dim3(r->threads);
    p.sharedMemBytes = (unsigned)r->smem;
    p.kernelParams = a.args;
    cudaError_t e = cudaGraphExecKernelNodeSetParams(r->exec, r->node, &p);
    if (e == cudaSuccess) e = cudaGraphLaunch(r->exec, stream);
    if (e == cudaSuccess) r->epoch += (unsigned)steps;
    return e;
}

void resident_drop_graph(Resident* r) {
    if (r->exec) cudaGraphExecDestroy(r->exec);
    if (r->graph) cudaGraphDestroy(r->graph);
    r->exec = nullptr;
    r->graph = nullptr;
}

void resident_free(Resident* r) {
    resident_drop_graph(r);
    if (r->scratch) cudaFree(r->scratch);
    r->scratch = nullptr;
    r->on = false;
}

}  // namespace axl
