// Work space of kernels that are being captured into a graph.
//
// An allocation during capture would become a node of the graph, and a graph with
// such nodes can be instantiated only once and cannot be part of another graph.
// So the work space is allocated outside of it and held by the graph: a user
// object, of which every copy and every executable form of the graph owns a
// reference, marks it idle when the last one is gone and has run.  Idle work
// space serves the next capture; the context frees it.
#include <memory>
#include <mutex>
#include <vector>

#include "ctx.h"

struct CapturedWork {
    struct Item {
        void *p;
        size_t bytes;
        bool busy, own;              // in use; by a graph of the solver
        unsigned long long capture;  // id of the capture that took it
        cudaStream_t stream;
    };
    std::mutex m;
    std::vector<Item> items;
};

namespace {

struct Hold {
    std::shared_ptr<CapturedWork> work;  // outlives the context
    size_t item;
};
void CUDART_CB let_go(void *p) {
    Hold *h = (Hold *)p;
    {
        std::lock_guard<std::mutex> lock(h->work->m);
        h->work->items[h->item].busy = false;
    }
    delete h;
}

}  // namespace

bool bri_capturing(cudaStream_t s, unsigned long long *id, cudaGraph_t *graph) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamGetCaptureInfo(s, &st, id, graph) != cudaSuccess) {
        cudaGetLastError();  // the default stream while another one is captured: the launch reports it
        return false;
    }
    return st == cudaStreamCaptureStatusActive;
}

void *bri_captured_work(bri_ctx *ctx, cudaStream_t s, unsigned long long id, cudaGraph_t graph, size_t bytes) {
    if (!ctx->captured) ctx->captured = std::make_shared<CapturedWork>();
    CapturedWork &w = *ctx->captured;
    size_t at = (size_t)-1;
    {
        std::lock_guard<std::mutex> lock(w.m);
        for (size_t i = 0; i < w.items.size(); i++) {
            const CapturedWork::Item &it = w.items[i];
            // of the same capture and stream: in order with what used it before
            if (it.busy && it.capture == id && it.stream == s && it.bytes >= bytes) return it.p;
            if (!it.busy && it.bytes >= bytes && (at == (size_t)-1 || it.bytes < w.items[at].bytes)) at = i;
        }
        if (at == (size_t)-1) {
            void *p = nullptr;
            cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;  // not part of the capture
            cudaThreadExchangeStreamCaptureMode(&mode);
            const cudaError_t e = cudaMalloc(&p, bytes);
            cudaThreadExchangeStreamCaptureMode(&mode);
            if (e != cudaSuccess) {
                cudaGetLastError();
                return nullptr;
            }
            at = w.items.size();
            w.items.push_back({p, bytes, false, false, 0, nullptr});
        }
        w.items[at].busy = true;
        w.items[at].own = ctx->own_capture;
        w.items[at].capture = id;
        w.items[at].stream = s;
    }
    Hold *h = new Hold{ctx->captured, at};
    cudaUserObject_t held;
    if (cudaUserObjectCreate(&held, h, let_go, 1, cudaUserObjectNoDestructorSync) != cudaSuccess) {
        cudaGetLastError();
        let_go(h);
        return nullptr;
    }
    if (cudaGraphRetainUserObject(graph, held, 1, cudaGraphUserObjectMove) != cudaSuccess) {
        cudaGetLastError();
        cudaUserObjectRelease(held, 1);
        return nullptr;
    }
    std::lock_guard<std::mutex> lock(w.m);
    return w.items[at].p;
}

// frees what is idle, or all with the context; true if there was something
bool bri_captured_free(bri_ctx *ctx, bool all) {
    if (!ctx->captured) return false;
    std::lock_guard<std::mutex> lock(ctx->captured->m);
    bool some = false;
    for (CapturedWork::Item &it : ctx->captured->items)
        if (it.p && (all || !it.busy)) {
            cudaFree(it.p);
            it.p = nullptr;
            it.bytes = 0;
            some = true;
        }
    return some;
}

// a graph of the program, there or yet to run, refers to the context's fields
bool bri_in_program_graph(bri_ctx *ctx) {
    if (!ctx->captured) return false;
    std::lock_guard<std::mutex> lock(ctx->captured->m);
    for (const CapturedWork::Item &it : ctx->captured->items)
        if (it.busy && !it.own) return true;
    return false;
}
