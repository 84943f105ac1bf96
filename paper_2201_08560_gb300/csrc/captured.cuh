// Host-side helpers of the level-synchronous drivers: a pinned flag read and
// the captured round loop (a CUDA graph of several gated rounds, replayed
// until a device flag reads 0).
#pragma once

#include "b2sr_internal.cuh"

namespace b2sr {

// Pinned host word for loop-exit flags.
struct HostFlag {
    int32_t* p = nullptr;
    HostFlag() { if (cudaMallocHost(&p, sizeof(int32_t)) != cudaSuccess) { cudaGetLastError(); p = nullptr; } }
    ~HostFlag() { if (p) cudaFreeHost(p); }
};

inline b2sr_status read_flag(const int32_t* dev, HostFlag& hf, cudaStream_t s, int32_t* out) {
    if (!hf.p) return fail(B2SR_ERR_OOM, "pinned flag");
    B2SR_CUDA_TRY(cudaMemcpyAsync(hf.p, dev, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    B2SR_CUDA_TRY(cudaStreamSynchronize(s));
    *out = *hf.p;
    return B2SR_OK;
}

__device__ __forceinline__ bool gate_closed(const int32_t* gate) { return gate && *gate == 0; }

// ---------------------------------------------------------------------------
// end of a round, inside the round's last kernel
// ---------------------------------------------------------------------------
struct LoopFlags {  // device
    int32_t active;  // 1 while rounds have work
    int32_t found;   // this round found something
    int32_t level;   // rounds run
    uint32_t ticket;
};

// Called by every thread of every block of a gated kernel; `any`: the thread
// found something.  The last block to arrive moves the loop on: active <-
// found, one more level; true for its thread 0.
__device__ __forceinline__ bool finish_round(LoopFlags* f, int any) {
    const int found = __syncthreads_or(any);
    if (threadIdx.x != 0) return false;
    if (found) atomicOr(&f->found, 1);
    __threadfence();
    if (atomicAdd(&f->ticket, 1u) != gridDim.x - 1u) return false;
    __threadfence();
    f->ticket = 0u;
    f->active = atomicExch(&f->found, 0);
    f->level += 1;
    return true;
}

// ---------------------------------------------------------------------------
// round loop
// ---------------------------------------------------------------------------
// Runs rounds (body(stream, r) enqueues one; r counts from 0 within a batch of
// `per_graph`) until *active reads 0, reading it after every batch.  Every
// round must be gated on *active.  The first `eager_batches` batches are
// enqueued on the caller's stream; a loop that goes on longer captures a batch
// into a CUDA graph on a private stream and replays it.  (Capture,
// instantiation, the private stream and its pinned flag cost 200 to 250 us a
// call, more than all launches of a search that ends in a few batches:
// single-source BFS on R-MAT 12 took 312 us.)  Returns in *rounds the rounds
// enqueued; B2SR_ERR_NOT_CONVERGED if *active is still set after max_rounds.
constexpr int kEagerBatches = 4;

template <class Body>
b2sr_status run_captured(cudaStream_t user, int per_graph, int64_t max_rounds, const int32_t* active,
                                Body&& body, int64_t* rounds, int eager_batches = kEagerBatches) {
    *rounds = 0;
    for (int batch = 0; batch < eager_batches; ++batch) {
        for (int r = 0; r < per_graph; ++r) B2SR_TRY(body(user, r));
        *rounds += per_graph;
        int32_t got = 0;
        B2SR_CUDA_TRY(cudaMemcpyAsync(&got, active, sizeof(int32_t), cudaMemcpyDeviceToHost, user));
        B2SR_CUDA_TRY(cudaStreamSynchronize(user));
        if (!got) return B2SR_OK;
        if (*rounds >= max_rounds) return fail(B2SR_ERR_NOT_CONVERGED, "exceeded max_iters rounds");
    }
    cudaStream_t cs = nullptr;
    cudaEvent_t ev = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    HostFlag hf;
    auto cleanup = [&](b2sr_status st) {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        if (cs) {
            if (ev) {  // the caller's stream waits for everything enqueued here
                cudaEventRecord(ev, cs);
                cudaStreamWaitEvent(user, ev, 0);
            }
            cudaStreamDestroy(cs);
        }
        if (ev) cudaEventDestroy(ev);
        return st;
    };
    B2SR_CUDA_TRY(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    cudaError_t e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e != cudaSuccess) return cleanup(cuda_fail(e, "cudaEventCreate"));
    e = cudaEventRecord(ev, user);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(cs, ev, 0);
    if (e != cudaSuccess) return cleanup(cuda_fail(e, "order capture stream"));
    e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return cleanup(cuda_fail(e, "cudaStreamBeginCapture"));
    const int64_t l0 = b2sr_launch_count();
    b2sr_status st = B2SR_OK;
    for (int r = 0; r < per_graph && st == B2SR_OK; ++r) st = body(cs, r);
    e = cudaStreamEndCapture(cs, &graph);
    if (st != B2SR_OK) return cleanup(st);
    if (e != cudaSuccess) return cleanup(cuda_fail(e, "cudaStreamEndCapture"));
    const int64_t per_replay = b2sr_launch_count() - l0;
    note_launches(-per_replay);  // counted again per replay below
    e = cudaGraphInstantiate(&exec, graph, 0);
    if (e != cudaSuccess) return cleanup(cuda_fail(e, "cudaGraphInstantiate"));
    for (;;) {
        e = cudaGraphLaunch(exec, cs);
        if (e != cudaSuccess) return cleanup(cuda_fail(e, "cudaGraphLaunch"));
        note_launches(per_replay);
        *rounds += per_graph;
        int32_t got = 0;
        st = read_flag(active, hf, cs, &got);
        if (st != B2SR_OK) return cleanup(st);
        if (!got) return cleanup(B2SR_OK);
        if (*rounds >= max_rounds) return cleanup(fail(B2SR_ERR_NOT_CONVERGED, "exceeded max_iters rounds"));
    }
}

}  // namespace b2sr
