// A fixed-point loop on the device: one graph whose conditional WHILE node runs the iteration's kernels
// and the stopping check of molt::loop_check (the rule of the single-grid solver), so that the host reads
// the outcome once per stage instead of once per iteration.  Where no graph can be built the host runs the same
// iterations and rule.
#pragma once

#include <cmath>
#include <cstring>

#include "molt_internal.h"

namespace molt {

class LoopGraphs {
  public:
    ~LoopGraphs() {
        for (Slot& s : slots_) drop(s);
        if (stream_) cudaStreamDestroy(stream_);
        if (ls_) cudaFree(ls_);
        if (host_) cudaFreeHost(host_);
        if (red_host_) cudaFreeHost(red_host_);
    }

    // The state words; red: the residual words (kRedSlots) that the iteration's last kernel accumulates into.
    bool init() {
        return cudaMalloc(&ls_, sizeof(LoopState)) == cudaSuccess &&
               cudaMallocHost(&host_, sizeof(LoopState)) == cudaSuccess &&
               cudaMallocHost(&red_host_, kRedSlots * sizeof(unsigned long long)) == cudaSuccess;
    }

    // Runs the loop of the stage with coefficient `key` on st and waits for it; body(stream) launches one
    // iteration in place on `iterate`.  The graphs of the last two (key, iterate) are kept (a step of a new
    // size builds one, 60 to 80 us: 3D 32^3, 8 iterations 341 -> 413 us, 2863 by the sweeps).  *out is the final state.
    template <class Body>
    cudaError_t run(double key, const void* iterate, unsigned long long* red, double tol, int max_iter, bool fp32,
                    Body body, cudaStream_t st, LoopState* out) {
        Slot* s = nullptr;
        for (Slot& t : slots_)
            if (t.exec && t.key == key && t.iterate == iterate) s = &t;
        if (!s) {
            s = &slots_[next_];
            next_ ^= 1;
            drop(*s);
            if (build(*s, red, tol, max_iter, fp32, body) != cudaSuccess) {
                drop(*s);
                cudaGetLastError();
                return host_loop(red, tol, max_iter, fp32, body, st, out);
            }
            s->key = key;
            s->iterate = iterate;
        }
        cudaError_t e;
        if ((e = loop_init(ls_, red, st)) != cudaSuccess || (e = cudaGraphLaunch(s->exec, st)) != cudaSuccess ||
            (e = cudaMemcpyAsync(host_, ls_, sizeof(LoopState), cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
            (e = cudaStreamSynchronize(st)) != cudaSuccess)
            return e;
        *out = *host_;
        return cudaSuccess;
    }

  private:
    struct Slot {
        double key = 0.0;
        const void* iterate = nullptr;
        cudaGraph_t graph = nullptr;
        cudaGraphExec_t exec = nullptr;
    };
    Slot slots_[2];
    int next_ = 0;
    cudaStream_t stream_ = nullptr;
    LoopState* ls_ = nullptr;
    LoopState* host_ = nullptr;
    unsigned long long* red_host_ = nullptr;

    static void drop(Slot& s) {
        if (s.exec) cudaGraphExecDestroy(s.exec);
        if (s.graph) cudaGraphDestroy(s.graph);
        s = Slot();
    }

    // The loop driven by the host, which reads the residual back after every iteration.
    template <class Body>
    cudaError_t host_loop(unsigned long long* red, double tol, int max_iter, bool fp32, Body body, cudaStream_t st,
                          LoopState* out) {
        LoopState ls{};
        ls.best = INFINITY;
        bool out_nan = false;
        while (!ls.done) {
            cudaError_t e;
            if ((e = cudaMemsetAsync(red, 0, kRedSlots * sizeof(unsigned long long), st)) != cudaSuccess ||
                (e = body(st)) != cudaSuccess ||
                (e = cudaMemcpyAsync(red_host_, red, kRedSlots * sizeof(unsigned long long), cudaMemcpyDeviceToHost, st)) !=
                    cudaSuccess ||
                (e = cudaStreamSynchronize(st)) != cudaSuccess)
                return e;
            double wmax;
            std::memcpy(&ls.res, &red_host_[0], sizeof(double));
            std::memcpy(&wmax, &red_host_[1], sizeof(double));
            // as loop_check: tolerance, FP32 floor of 2 ulp of max|w|, stall at the FP32 noise floor, cap, NaN
            const double ulp = wmax * 5.9604644775390625e-08;
            ls.tol_used = fp32 ? std::fmax(tol, 2.0 * ulp) : tol;
            ls.k += 1;
            bool stop = ls.k >= max_iter;
            if (!std::isfinite(ls.res)) {
                stop = true;
            } else if (ls.res < ls.tol_used) {
                ls.converged = 1;
            } else if (ls.res < ls.best) {
                ls.best = ls.res;
                ls.stall = 0;
            } else if (fp32 && ls.res < 64.0 * ulp && ++ls.stall >= 6) {
                ls.converged = 1;
                ls.tol_used = ls.res;
            }
            ls.done = stop || ls.converged;
            out_nan = red_host_[2] != 0;
        }
        *out = ls;
        if (out_nan) out->converged = 0, out->res = NAN;
        return cudaSuccess;
    }

    template <class Body>
    cudaError_t build(Slot& s, unsigned long long* red, double tol, int max_iter, bool fp32, Body body) {
        cudaError_t e;
        if (!stream_ && (e = cudaStreamCreateWithFlags(&stream_, cudaStreamNonBlocking)) != cudaSuccess) return e;
        if ((e = cudaGraphCreate(&s.graph, 0)) != cudaSuccess) return e;
        cudaGraphConditionalHandle h;
        if ((e = cudaGraphConditionalHandleCreate(&h, s.graph, 1, cudaGraphCondAssignDefault)) != cudaSuccess) return e;
        cudaGraphNodeParams np = {};
        np.type = cudaGraphNodeTypeConditional;
        np.conditional.handle = h;
        np.conditional.type = cudaGraphCondTypeWhile;
        np.conditional.size = 1;
        cudaGraphNode_t node;
        if ((e = cudaGraphAddNode(&node, s.graph, nullptr, nullptr, 0, &np)) != cudaSuccess) return e;
        if ((e = cudaStreamBeginCaptureToGraph(stream_, np.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                               cudaStreamCaptureModeRelaxed)) != cudaSuccess)
            return e;
        cudaError_t launched = body(stream_);
        if (launched == cudaSuccess) launched = loop_check(h, ls_, red, tol, max_iter, fp32 ? 1 : 0, stream_);
        cudaGraph_t captured = nullptr;
        e = cudaStreamEndCapture(stream_, &captured);
        if (launched != cudaSuccess) return launched;
        if (e != cudaSuccess) return e;
        return cudaGraphInstantiate(&s.exec, s.graph, 0);
    }
};

}  // namespace molt
