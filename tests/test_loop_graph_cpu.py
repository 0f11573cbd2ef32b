"""The device-driven loop of the 3D and sixth-order solvers (csrc/loop_graph.h) where no graph can be built: the host
runs the same iterations under the same stopping rule and the stage succeeds.  The CUDA runtime is a fake
one whose graph calls fail, each in turn."""
import math

import pytest

from _host_unit import run_host_unit

PROGRAM = r"""
#include <cuda_runtime.h>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "loop_graph.h"

static int fail = 0;                        // which graph call fails
static int last = 0;
static cudaError_t step(int which) { return which == fail ? cudaErrorNotSupported : cudaSuccess; }
static cudaStream_t const kCapture = reinterpret_cast<cudaStream_t>(0x10), kUser = reinterpret_cast<cudaStream_t>(0x20);
template <class T> static T fake() { return reinterpret_cast<T>(0x30); }

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) { *p = std::malloc(n); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = std::malloc(n); return cudaSuccess; }
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaGetLastError() { last = 1; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = kCapture; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { *g = fake<cudaGraph_t>(); return step(1); }
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle* h, cudaGraph_t, unsigned, unsigned) {
    *h = 0;
    return step(2);
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t*, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                             cudaGraphNodeParams* p) {
    static cudaGraph_t body = fake<cudaGraph_t>();
    p->conditional.phGraph_out = &body;
    return step(3);
}
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*,
                                          size_t, cudaStreamCaptureMode) { return step(4); }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = fake<cudaGraph_t>(); return step(5); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
    *e = nullptr;
    return step(6);
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorUnknown; }
}
namespace molt {
cudaError_t loop_init(LoopState*, unsigned long long*, cudaStream_t) { return cudaSuccess; }
cudaError_t loop_check(cudaGraphConditionalHandle, LoopState*, unsigned long long*, double, int, int, cudaStream_t) {
    return cudaSuccess;
}
}  // namespace molt

int main() {
    // residuals over numbers; from iteration `bad` on (counted from 1, 0: never) one value is a NaN
    struct Case { const char* name; double res[12]; int n; bool fp32; double tol; int max_iter; int bad; };
    const double u = 5.9604644775390625e-08;   // 2^-24, max|w| = 1
    const Case cases[] = {
        {"converges", {1, 0.1, 0.01, 1e-9}, 4, false, 1e-6, 50},
        {"floor", {1, 0.1, 1.5 * u}, 3, true, 1e-30, 50},
        {"cap", {1, 0.5, 0.25, 0.125}, 4, false, 1e-6, 4},
        {"stall", {30 * u, 31 * u, 31 * u, 31 * u, 31 * u, 31 * u, 31 * u}, 7, true, 1e-30, 50},
        {"overflow", {1, 1e20, INFINITY}, 3, false, 1e-6, 50},
        {"nan", {1, 1e20, 0}, 3, false, 1e-6, 50, 3},
        {"others", {1, 0.1, 0.01, 1e-3, 1e-9}, 5, false, 1e-6, 50, 2},
        {"nancap", {1, 0.5, 0.25, 0.125}, 4, false, 1e-6, 4, 4},
    };
    for (fail = 1; fail <= 6; ++fail)
        for (const Case& c : cases) {
            molt::LoopGraphs loop;
            if (!loop.init()) return 1;
            unsigned long long red[molt::kRedSlots] = {7, 7, 7};
            int k = 0;
            auto body = [&](cudaStream_t s) {
                if (s == kUser) {
                    if (red[0] || red[1] || red[2] || k >= c.n) return cudaErrorUnknown;   // slots cleared, no iteration too many
                    const double r = c.res[k++], w = 1.0;
                    std::memcpy(&red[0], &r, 8);
                    std::memcpy(&red[1], &w, 8);
                    red[2] = c.bad && k >= c.bad ? 1 : 0;
                }
                return cudaSuccess;
            };
            molt::LoopState out{};
            last = 0;
            const cudaError_t e = loop.run(0.5, red, red, c.tol, c.max_iter, c.fp32, body, kUser, &out);
            std::printf("%d %s %d %d %d %.17g %.17g %d\n", fail, c.name, (int)e, out.k, out.converged, out.res, out.tol_used,
                        last);
        }
    return 0;
}
"""


@pytest.fixture(scope="module")
def outcomes(tmp_path_factory):
    out = {}
    for line in run_host_unit(tmp_path_factory.mktemp("loop"), PROGRAM).splitlines():
        f = line.split()
        out[int(f[0]), f[1]] = (int(f[2]), int(f[3]), int(f[4]), float(f[5]), float(f[6]), int(f[7]))
    return out


@pytest.mark.parametrize("call", range(1, 7))
def test_host_runs_the_loop_where_a_graph_call_fails(outcomes, call):
    u = 2.0 ** -24
    # error, iterations, converged, residual, tolerance, pending error cleared
    assert outcomes[call, "converges"] == (0, 4, 1, 1e-9, 1e-6, 1)
    assert outcomes[call, "floor"] == (0, 3, 1, 1.5 * u, 2 * u, 1)
    assert outcomes[call, "cap"] == (0, 4, 0, 0.125, 1e-6, 1)
    assert outcomes[call, "stall"] == (0, 7, 1, 31 * u, 31 * u, 1)
    e, k, conv, res, _, _ = outcomes[call, "overflow"]
    assert (e, k, conv) == (0, 3, 0) and math.isinf(res)
    # a NaN: the iteration ends when what is left of the residual does, never as converged
    for name, its in (("nan", 3), ("others", 5), ("nancap", 4)):
        e, k, conv, res, _, _ = outcomes[call, name]
        assert (e, k, conv) == (0, its, 0) and math.isnan(res), name
