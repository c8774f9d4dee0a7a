// flux_run.cuh -- how the flux steps of one context are launched (not part of the C ABI): one
// launch per step and one that closes a run, runs of kFluxGraph steps replayed from a CUDA graph
// captured once per starting buffer on streams that can be captured.
#pragma once

#include "internal.cuh"
#include "mp_ctx.cuh"

namespace mp {

constexpr int kFluxGraph = 64;  // even: a replay ends on the buffer it started from

// Tables are an option that costs memory: more than 64 MB only where they take at most a quarter of
// what is free once the context's own arrays are in place, so that the capacity of a device (binary16
// storage above all) is not spent on them. The context then recomputes, as with MP_VARIANT_RECOMPUTE.
inline bool tables_fit(size_t bytes, size_t free_bytes) { return bytes <= (64u << 20) || bytes <= free_bytes / 4; }
inline bool tables_fit(size_t bytes)
{
    if (tables_fit(bytes, 0)) return true;  // no look-up for small contexts
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return tables_fit(bytes, free_b);
}

// launch(pending, programmatic): the step from buffer c->cur; pending: the previous launch was a
// step whose series is not appended yet. finish(parity): appends the series of the last step, which
// read buffer `parity`.
// A step reads its tables before griddepcontrol.wait. What is read there has to be finished and
// visible when the launch before it has merely started, and a programmatic launch may start,
// before its wait, while the table kernel's writes are still on their way. So the first step after
// set-up is an ordinary launch (or the first node of a graph), and every later one follows it.
template <typename Launch, typename Finish>
int run_flux(mp_ctx* c, long long n, Launch launch, Finish finish)
{
    cudaError_t le = cudaSuccess;  // first failed launch, if any
    auto run = [&](long long count) {
        for (long long k = 0; k < count; ++k) {
            const cudaError_t e = launch(k > 0 ? 1 : 0, !c->tables_new);
            c->tables_new = false;
            if (e != cudaSuccess && le == cudaSuccess) le = e;
            c->cur = 1 - c->cur;
        }
        if (count > 0) {
            const cudaError_t e = finish(1 - c->cur);
            if (e != cudaSuccess && le == cudaSuccess) le = e;
        }
    };
    const bool capturable =
        c->stream != nullptr && c->stream != cudaStreamLegacy && c->stream != cudaStreamPerThread;
    if (capturable && n >= 2 * kFluxGraph) {
        const int b = c->cur;
        c->tables_new = false;  // a graph starts when all work before it is done
        if (!c->exec[b]) {
            cudaError_t e = cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal);
            if (e == cudaSuccess) {
                run(kFluxGraph);
                e = cudaStreamEndCapture(c->stream, &c->graph[b]);
            }
            c->cur = b;
            if (e == cudaSuccess && le != cudaSuccess) e = le;
            if (e == cudaSuccess) e = cudaGraphInstantiate(&c->exec[b], c->graph[b], 0);
            if (e != cudaSuccess) return cuda_fail(e, "mp_step: graph capture");
        }
        for (; n >= kFluxGraph; n -= kFluxGraph) {
            MP_CUDA(cudaGraphLaunch(c->exec[b], c->stream));
            c->t += kFluxGraph;
        }
    }
    run(n);
    c->t += n;
    if (le != cudaSuccess) return cuda_fail(le, "mp_step: launch");
    MP_CUDA(cudaGetLastError());
    return MP_OK;
}

}  // namespace mp
