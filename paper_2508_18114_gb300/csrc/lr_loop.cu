// A run of many steps as ONE device-side loop: the launches of `per` steps are the body
// of a conditional (while) node of a CUDA graph, and a last kernel in the body advances
// the step counter and says whether the body runs again. The host enqueues one graph
// however long the run is, so a call of a whole pulse returns at once (16 to 21
// launches a step fill the launch queue after ~60 steps and hold the host from then on) and
// contexts on several streams overlap. Everything that differs between calls is read from
// the counter, so a context builds its graph once (~0.4 ms).
//
// The kernels of a graph also follow one another faster than launches on a stream: one
// N = 2000, M = 20 pulse in FP32 takes 37.5 us a stage in place of 47.0.
//
// This file is compiled as relocatable device code: cudaGraphSetConditional is a
// function of the device runtime library.
#include "lr_internal.cuh"

namespace lr {

namespace {

__global__ void loop_begin(long long* c, LoopCount count) {
  c[0] = count.first;
  c[1] = count.first + count.n;
  c[2] = count.call;
}
__global__ void loop_next(long long* c, long long per, cudaGraphConditionalHandle h) {
  const long long v = c[0] + per;
  c[0] = v;
  cudaGraphSetConditional(h, v < c[1] ? 1u : 0u);
}

// This thread may make any call while another thread captures; what building a graph needs
// besides the graph is released at its end.
struct Build {
  cudaGraph_t graph = nullptr;
  cudaStream_t cap = nullptr;
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  Build() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~Build() {
    if (graph) cudaGraphDestroy(graph);
    if (cap) cudaStreamDestroy(cap);
    cudaThreadExchangeStreamCaptureMode(&mode);
  }
};

cudaError_t build(long long* c, long per, cudaError_t (*body)(void*, cudaStream_t), void* arg, cudaGraphExec_t* exec) {
  Build b;
  cudaError_t e;
  if ((e = cudaGraphCreate(&b.graph, 0)) != cudaSuccess) return e;
  cudaGraphConditionalHandle h;
  if ((e = cudaGraphConditionalHandleCreate(&h, b.graph, 1, cudaGraphCondAssignDefault)) != cudaSuccess) return e;
  cudaGraphNode_t loop;
  cudaGraphNodeParams np = {};
  np.type = cudaGraphNodeTypeConditional;
  np.conditional.handle = h;
  np.conditional.type = cudaGraphCondTypeWhile;
  np.conditional.size = 1;
  if ((e = cudaGraphAddNode(&loop, b.graph, nullptr, nullptr, 0, &np)) != cudaSuccess) return e;
  if ((e = cudaStreamCreateWithFlags(&b.cap, cudaStreamNonBlocking)) != cudaSuccess) return e;
  cudaGraph_t bg = np.conditional.phGraph_out[0];
  if ((e = cudaStreamBeginCaptureToGraph(b.cap, bg, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed)) != cudaSuccess)
    return e;
  e = body(arg, b.cap);
  if (e == cudaSuccess) {
    loop_next<<<1, 1, 0, b.cap>>>(c, per, h);
    e = cudaGetLastError();
  }
  const cudaError_t ee = cudaStreamEndCapture(b.cap, &bg);
  if (e != cudaSuccess) return e;
  if (ee != cudaSuccess) return ee;
  return cudaGraphInstantiate(exec, b.graph, 0);
}

}  // namespace

LoopCache::~LoopCache() {
  for (int i = 0; i < n; ++i) cudaGraphExecDestroy(e[i].exec);
}

cudaError_t device_loop_run(LoopRef loop, double dt, double tau, LoopCount count, long per,
                            cudaError_t (*body)(void*, cudaStream_t), void* arg, cudaStream_t s) {
  LoopCache& k = *loop.cache;
  cudaGraphExec_t exec = nullptr;
  for (int i = 0; i < k.n; ++i)
    if (k.e[i].dt == dt && k.e[i].tau == tau && k.e[i].c == loop.c) exec = k.e[i].exec;
  cudaError_t err;
  if (!exec) {
    if ((err = build(loop.c, per, body, arg, &exec)) != cudaSuccess) return err;
    int at = k.n;
    if (k.n < LOOP_KEPT) {
      ++k.n;
    } else {   // the oldest goes
      at = k.next;
      k.next = (at + 1) % LOOP_KEPT;
      cudaGraphExecDestroy(k.e[at].exec);
    }
    k.e[at] = {dt, tau, loop.c, exec};
  }
  loop_begin<<<1, 1, 0, s>>>(loop.c, count);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  return cudaGraphLaunch(exec, s);
}

}  // namespace lr
