// CG driver: the device-driven conditional graph, its cache, and the host loop.
//
// Graph of one launch (one "chunk" of up to check_interval iterations):
//
//   chunk_start --> WHILE (go) {
//                     U times: head: 4 sloppy hops (alpha), x_s / r_s update (beta, or request)
//                              tail: p = r_s + beta p
//                     IF (replacement requested) { r_s = r - A x_s, FP32 arithmetic; tail }  [three-level only]
//                     IF (reliable update requested) { x += x_s; r = b - A x in FP64; tail }
//                     loop control: go = active && chunks left && iter < maxiter
//                   }
//
// An iteration that requests an update pauses the solve (active = 0), so that the
// rest of the body's kernels return at once, and the branch resumes it. U, the
// iterations per body, is chosen per solve (iterations_per_body).
//
// The WHILE and IF conditions are set on the device (cudaGraphSetConditional)
// by a one-thread control kernel and by the finaliser of the update kernel,
// so reliable updates cost no host round trip. Every body execution takes U
// from the chunk counter, so one launch runs at most check_interval
// iterations whatever the state says. The host only reads the control block
// between launches (convergence, NaN, iteration cap, wall-clock limit).
//
// With use_graph = 0 the same kernels are launched directly and a requested
// reliable update pauses the chunk for the host instead.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "cg_engine.h"

namespace lqcd {

__global__ void k_chunk_start(Control* c, int chunk, int maxiter, cudaGraphConditionalHandle h_loop) {
  c->chunk_left = chunk;
  const int go = c->active && c->iter < maxiter && c->n_done < c->nsys && !(c->reason & REASON_NAN);
  cudaGraphSetConditional(h_loop, go ? 1u : 0u);
}

__global__ void k_loop_control(Control* c, int maxiter, cudaGraphConditionalHandle h_loop,
                               cudaGraphConditionalHandle h_rel, cudaGraphConditionalHandle h_mid, int has_mid,
                               int unroll) {
  cudaGraphSetConditional(h_rel, 0u);  // the next iteration's update decides afresh
  if (has_mid) cudaGraphSetConditional(h_mid, 0u);
  c->chunk_left -= unroll;
  const int go = c->active && c->chunk_left > 0 && c->iter < maxiter && c->n_done < c->nsys &&
                 !(c->reason & REASON_NAN);
  cudaGraphSetConditional(h_loop, go ? 1u : 0u);
}

// U, the iterations per body of the graph. The WHILE and IF nodes and the control
// kernel cost 7 to 14 us per body on GB300; an iteration launched behind a pause costs 6 us,
// and 5 us more per 1,000 blocks of a hop (which all start and return). So U must not
// pass the distance between pauses by much, and an update is due whenever the
// residual has fallen by delta (delta_mid: a replacement), on well-conditioned
// links every 2 iterations at 0.3 and every 3 at 0.1 (Haar-distributed links fall by 2.7 per
// iteration; others take longer, and lose less). Whole even-odd solves in ms, U = 1 / 2 / 4 / 8:
//   12^3 x 24 FP32, delta 0.9         3.05  3.17  3.43    -     (an update in each of 23 iterations)
//                   delta 0.3         2.16  2.01  2.12  2.44    (12 updates)
//                   delta 0.1         1.77  1.75  1.72  2.00    (8)
//                   delta 0.01        1.56  1.45  1.45  1.45    (5)
//                   delta 3e-6        1.31  1.16  1.13  1.14    (2)
//   24^3 x 48 FP32, delta 0.3        22.36 21.95 21.92 23.20    (17 of 60)
//             FP16, 0.003 and 3e-6   11.29 11.20 11.03 11.23    (5 pauses of 61)
//             FP32, delta 3e-6       14.33 13.89 13.77 13.71    (2)
//   two columns, delta 0.1           35.03 34.91 34.92    -     (5,184 blocks)
//   four columns, delta 0.1          60.86 60.97 61.22    -     (10,368 blocks)
//   32^4, 12 columns, FP16           91.57 91.91 94.33 95.28    (49,152 blocks, 5 pauses of 24)
//   16^4 FP32, delta 1e-5 (HMC trajectory) -    -   88.15 86.91   (2 of 93 in each solve)
constexpr int64_t MAX_SKIPPED_BLOCKS = 6144;
static int iterations_per_body(const CgEngine& E, const lqcd_solver_params& prm, int chunk) {
  const double delta = prm.sloppy_prec == LQCD_F64 ? 0.0  // paused at the end only
                       : E.has_mid() ? std::max(prm.delta, prm.delta_mid) : prm.delta;
  int u = E.blocks > MAX_SKIPPED_BLOCKS || delta > 0.3 ? 1 : delta > 0.1 ? 2 : delta > 1e-4 ? 4 : 8;
  while (chunk % u) u--;  // a chunk is a whole number of bodies
  return u;
}

struct GraphEntry {
  std::vector<unsigned char> key;
  cudaGraphExec_t exec;
  uint64_t body_kernels, reliable_kernels, mid_kernels;
  uint64_t last_use;
};

static std::mutex g_graph_mutex;
static std::vector<GraphEntry> g_graphs;
static uint64_t g_graph_clock = 0;
constexpr size_t MAX_GRAPHS = 16;

void release_graph_cache() {
  std::lock_guard<std::mutex> lock(g_graph_mutex);
  for (auto& e : g_graphs) cudaGraphExecDestroy(e.exec);
  g_graphs.clear();
}

namespace {

struct Capture {
  cudaStream_t s = nullptr;
  ~Capture() {
    if (s) {
      cudaStreamCaptureStatus cs;
      if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) {
        cudaGraph_t g = nullptr;
        cudaStreamEndCapture(s, &g);
        if (g) cudaGraphDestroy(g);
      }
      cudaStreamDestroy(s);
    }
    g_count_suspended = false;
  }
};

}  // namespace

#define LQCD_TRY_CUDA(expr, what)                  \
  do {                                             \
    cudaError_t e_ = (expr);                       \
    if (e_ != cudaSuccess) return cuda_fail(e_, what); \
  } while (0)

static int build_graph(CgEngine& E, int chunk, int unroll, int maxiter, GraphEntry* out) {
  Capture cap;
  LQCD_TRY_CUDA(cudaStreamCreateWithFlags(&cap.s, cudaStreamNonBlocking), "cg graph: stream");
  cudaGraph_t outer = nullptr;
  LQCD_TRY_CUDA(cudaGraphCreate(&outer, 0), "cg graph: create");
  struct GraphGuard {
    cudaGraph_t g;
    ~GraphGuard() { if (g) cudaGraphDestroy(g); }
  } guard{outer};
  cudaGraphConditionalHandle h_loop;
  LQCD_TRY_CUDA(cudaGraphConditionalHandleCreate(&h_loop, outer, 1, cudaGraphCondAssignDefault),
                "cg graph: loop handle");
  const cudaStreamCaptureMode mode = cudaStreamCaptureModeThreadLocal;
  g_count_suspended = true;

  // chunk start
  LQCD_TRY_CUDA(cudaStreamBeginCaptureToGraph(cap.s, outer, nullptr, nullptr, 0, mode), "cg graph: capture");
  k_chunk_start<<<1, 1, 0, cap.s>>>(E.ctrl, chunk, maxiter, h_loop);
  int st = after_launch("k_chunk_start");
  LQCD_TRY_CUDA(cudaStreamEndCapture(cap.s, &outer), "cg graph: end capture");
  if (st) return st;
  cudaGraphNode_t start = nullptr;
  size_t n = 1;
  LQCD_TRY_CUDA(cudaGraphGetNodes(outer, &start, &n), "cg graph: nodes");

  // WHILE node and its body
  cudaGraphNodeParams wp = {};
  wp.type = cudaGraphNodeTypeConditional;
  wp.conditional.handle = h_loop;
  wp.conditional.type = cudaGraphCondTypeWhile;
  wp.conditional.size = 1;
  cudaGraphNode_t wnode;
  LQCD_TRY_CUDA(cudaGraphAddNode(&wnode, outer, &start, nullptr, 1, &wp), "cg graph: while node");
  cudaGraph_t body = wp.conditional.phGraph_out[0];
  cudaGraphConditionalHandle h_rel, h_mid = 0;
  LQCD_TRY_CUDA(cudaGraphConditionalHandleCreate(&h_rel, body, 0, cudaGraphCondAssignDefault),
                "cg graph: reliable handle");
  const bool has_mid = E.has_mid();
  if (has_mid)
    LQCD_TRY_CUDA(cudaGraphConditionalHandleCreate(&h_mid, body, 0, cudaGraphCondAssignDefault),
                  "cg graph: replacement handle");

  // body: the iterations
  LQCD_TRY_CUDA(cudaStreamBeginCaptureToGraph(cap.s, body, nullptr, nullptr, 0, mode), "cg graph: capture");
  uint64_t c0 = g_captured_launches;
  for (int u = 0; u < unroll && !st; u++)
    if (!(st = E.head(cap.s, 1, h_rel, h_mid))) st = E.tail(cap.s);
  out->body_kernels = g_captured_launches - c0;
  cudaStreamCaptureStatus cs;
  const cudaGraphNode_t* deps = nullptr;
  size_t ndeps = 0;
  cudaError_t e = cudaStreamGetCaptureInfo(cap.s, &cs, nullptr, nullptr, &deps, nullptr, &ndeps);
  std::vector<cudaGraphNode_t> frontier(deps, deps + (e == cudaSuccess ? ndeps : 0));
  LQCD_TRY_CUDA(cudaStreamEndCapture(cap.s, &body), "cg graph: end capture");
  if (st) return st;
  if (e != cudaSuccess) return cuda_fail(e, "cg graph: capture info");

  // body: IF (FP32-arithmetic replacement requested)
  out->mid_kernels = 0;
  if (has_mid) {
    cudaGraphNodeParams mp = {};
    mp.type = cudaGraphNodeTypeConditional;
    mp.conditional.handle = h_mid;
    mp.conditional.type = cudaGraphCondTypeIf;
    mp.conditional.size = 1;
    cudaGraphNode_t mnode;
    LQCD_TRY_CUDA(cudaGraphAddNode(&mnode, body, frontier.data(), nullptr, frontier.size(), &mp),
                  "cg graph: replacement node");
    cudaGraph_t mg = mp.conditional.phGraph_out[0];
    LQCD_TRY_CUDA(cudaStreamBeginCaptureToGraph(cap.s, mg, nullptr, nullptr, 0, mode), "cg graph: capture");
    c0 = g_captured_launches;
    if (!(st = E.mid(cap.s))) st = E.tail(cap.s);
    out->mid_kernels = g_captured_launches - c0;
    LQCD_TRY_CUDA(cudaStreamEndCapture(cap.s, &mg), "cg graph: end capture");
    if (st) return st;
    frontier.assign(1, mnode);
  }

  // body: IF (reliable update requested)
  cudaGraphNodeParams ip = {};
  ip.type = cudaGraphNodeTypeConditional;
  ip.conditional.handle = h_rel;
  ip.conditional.type = cudaGraphCondTypeIf;
  ip.conditional.size = 1;
  cudaGraphNode_t inode;
  LQCD_TRY_CUDA(cudaGraphAddNode(&inode, body, frontier.data(), nullptr, frontier.size(), &ip),
                "cg graph: if node");
  cudaGraph_t rel = ip.conditional.phGraph_out[0];
  LQCD_TRY_CUDA(cudaStreamBeginCaptureToGraph(cap.s, rel, nullptr, nullptr, 0, mode), "cg graph: capture");
  c0 = g_captured_launches;
  if (!(st = E.reliable(cap.s))) st = E.tail(cap.s);
  out->reliable_kernels = g_captured_launches - c0;
  LQCD_TRY_CUDA(cudaStreamEndCapture(cap.s, &rel), "cg graph: end capture");
  if (st) return st;

  // body: loop control, after the IF node
  LQCD_TRY_CUDA(cudaStreamBeginCaptureToGraph(cap.s, body, &inode, nullptr, 1, mode), "cg graph: capture");
  c0 = g_captured_launches;
  k_loop_control<<<1, 1, 0, cap.s>>>(E.ctrl, maxiter, h_loop, h_rel, h_mid, has_mid ? 1 : 0, unroll);
  st = after_launch("k_loop_control");
  out->body_kernels += g_captured_launches - c0;
  LQCD_TRY_CUDA(cudaStreamEndCapture(cap.s, &body), "cg graph: end capture");
  if (st) return st;

  LQCD_TRY_CUDA(cudaGraphInstantiate(&out->exec, outer, 0), "cg graph: instantiate");
  return LQCD_OK;
}

static int cached_graph(CgEngine& E, const std::vector<unsigned char>& key, int chunk, int unroll,
                        int maxiter, GraphEntry* out) {
  std::lock_guard<std::mutex> lock(g_graph_mutex);
  for (auto& e : g_graphs) {
    if (e.key == key) {
      e.last_use = ++g_graph_clock;
      *out = e;
      return LQCD_OK;
    }
  }
  GraphEntry ne;
  ne.key = key;
  ne.exec = nullptr;
  int st = build_graph(E, chunk, unroll, maxiter, &ne);
  if (st) {
    if (ne.exec) cudaGraphExecDestroy(ne.exec);
    return st;
  }
  if (g_graphs.size() >= MAX_GRAPHS) {
    size_t lru = 0;
    for (size_t i = 1; i < g_graphs.size(); i++)
      if (g_graphs[i].last_use < g_graphs[lru].last_use) lru = i;
    cudaGraphExecDestroy(g_graphs[lru].exec);
    g_graphs.erase(g_graphs.begin() + lru);
  }
  ne.last_use = ++g_graph_clock;
  g_graphs.push_back(ne);
  *out = ne;
  return LQCD_OK;
}

static int read_ctrl(const Control* d, Control* h, cudaStream_t s) {
  cudaError_t e = cudaMemcpyAsync(h, d, sizeof(Control), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(e, "cg: control readback");
  return LQCD_OK;
}

int run_cg(CgEngine& E, const lqcd_solver_params& prm, std::vector<unsigned char> key, cudaStream_t s,
           std::chrono::steady_clock::time_point t0, Control* ctrl) {
  int st = E.init(s);
  if (st) return st;
  const int chunk = prm.check_interval > 0 ? prm.check_interval : 16;
  const int unroll = iterations_per_body(E, prm, chunk);
  key_append(key, unroll);
  GraphEntry ge;
  ge.exec = nullptr;
  if (prm.use_graph && (st = cached_graph(E, key, chunk, unroll, prm.maxiter, &ge))) return st;
  auto timed_out = [&]() {
    if (prm.timeout_ms <= 0) return false;
    const double el = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return el > prm.timeout_ms;
  };
  for (;;) {
    if ((st = read_ctrl(E.ctrl, ctrl, s))) return st;
    if (ctrl->reason & REASON_NAN) return fail(LQCD_ERR_NAN, "cg: NaN/Inf or non-positive p^dag A p");
    if (ctrl->n_done == ctrl->nsys) return LQCD_OK;
    if (ge.exec) {
      // device-driven: the final FP64 check at the iteration cap already ran
      if (ctrl->iter >= prm.maxiter) return fail(LQCD_ERR_NOT_CONVERGED, "cg: maxiter %d reached", prm.maxiter);
      if (timed_out()) return fail(LQCD_ERR_TIMEOUT, "cg: wall-clock limit %.1f ms exceeded", prm.timeout_ms);
      const Control before = *ctrl;
      cudaError_t e = cudaGraphLaunch(ge.exec, s);
      if (e != cudaSuccess) return cuda_fail(e, "cg: graph launch");
      if ((st = read_ctrl(E.ctrl, ctrl, s))) return st;
      const uint64_t bodies = (uint64_t)((chunk - ctrl->chunk_left) / unroll);
      const uint64_t rels = (uint64_t)(ctrl->n_reliable - before.n_reliable);
      const uint64_t mids = (uint64_t)(ctrl->n_mid - before.n_mid);
      count_launches(1 + bodies * ge.body_kernels + rels * ge.reliable_kernels + mids * ge.mid_kernels);
      continue;
    }
    // host-driven
    if (ctrl->iter >= prm.maxiter) {
      if ((st = E.reliable(s)) || (st = E.tail(s))) return st;
      if ((st = read_ctrl(E.ctrl, ctrl, s))) return st;
      if (ctrl->reason & REASON_NAN) return fail(LQCD_ERR_NAN, "cg: NaN/Inf in the true residual");
      if (ctrl->n_done != ctrl->nsys) return fail(LQCD_ERR_NOT_CONVERGED, "cg: maxiter %d reached", prm.maxiter);
      return LQCD_OK;
    }
    if (ctrl->active == 0) {
      // paused by the update's finaliser: the reason bits say which recomputation is due
      const bool mid_only = (ctrl->reason & REASON_MID) && !(ctrl->reason & (REASON_CONVERGED | REASON_RELIABLE));
      if ((st = mid_only ? E.mid(s) : E.reliable(s)) || (st = E.tail(s))) return st;
      continue;
    }
    if (timed_out()) return fail(LQCD_ERR_TIMEOUT, "cg: wall-clock limit %.1f ms exceeded", prm.timeout_ms);
    for (int i = 0; i < chunk; i++)
      if ((st = E.head(s, 0, 0, 0)) || (st = E.tail(s))) return st;
  }
}

}  // namespace lqcd
