// One Krylov-vector evaluation (Section 3, Eqs. 8-10 and the SIMPLE-like
// loop) in the mixed precision of fv_mixed.cu, captured once per grid as a
// CUDA graph whose pass loop is a device-side WHILE conditional node:
//
//   [base(U, if given)] -> J.v -> D w -> [TPF -> pass] x 3
//   -> while (the last pass says go on) { TPF -> pass } -> join
//
// The stop test of the loop (||phi_k|| <= eps ||phi_1||, round-off floor,
// pass cap) is taken on the device by the last block of each pass (fv_pass.cu),
// so a whole evaluation is one graph launch with no host round trip.  Per-call
// arguments (pointers, eps, omega) are arguments of the J.v node (and, for U,
// of the base node), updated in the executable graph before each launch; J.v
// hands them on to the other kernels through a small device block.
#include <algorithm>
#include <cstddef>
#include <cstring>

#include "fv_ff.cuh"
#include "fv_internal.cuh"
#include "fv_stencil_dev.cuh"
#include "fv_tc5.cuh"

namespace fv {

namespace {

// The evaluation's base flow when the call passes one: rounded (FV_MIXED) or
// split (FV_FF) into the grid's stored copy that the J.v kernel reads.
template <bool FF>
__global__ void k_base_from_call(const double* __restrict__ U, float* __restrict__ U32,
                                 float2* __restrict__ Uff, int64_t n) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const double d = __ldg(U + e);
    if (FF) {
      const ff a = f64_split(d);
      Uff[e] = make_float2(a.hi, a.lo);
    } else {
      U32[e] = f64_round_f32(d);
    }
  }
}

inline unsigned grid1d(int64_t n) {
  int64_t b = (n + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  return (unsigned)(b < 1 ? 1 : b);
}

}  // namespace

// The passes of one evaluation, captured on the stream cs: three passes in a
// row (three is the usual number; a loop that ends earlier makes the rest
// return at once), then a WHILE node for what may follow, then the join.  bs:
// a stream for the body's capture.  On an error the capture on cs is left to
// the caller.
static fv_status capture_passes(fv_grid* g, int prec, cudaStream_t cs, cudaStream_t bs, const CallBlock* cb,
                                LoopState* ls) {
  cudaStreamCaptureStatus cst;
  cudaGraph_t cap_graph;
  const cudaGraphNode_t* deps = nullptr;
  size_t ndeps = 0;
  FV_CUDA(cudaStreamGetCaptureInfo(cs, &cst, nullptr, &cap_graph, &deps, nullptr, &ndeps));
  cudaGraphConditionalHandle h;
  FV_CUDA(cudaGraphConditionalHandleCreate(&h, cap_graph, 0, cudaGraphCondAssignDefault));
  g->stream = cs;
  for (int q = 0; q < 3; ++q) {
    FV_TRY(tpf_solve_f32(g, g->r32, g->phis[q], prec, q > 0 ? &ls->status : nullptr));
    FV_TRY(launch_pass(g, prec, q, cb, ls, &h, true));
  }
  FV_CUDA(cudaStreamGetCaptureInfo(cs, &cst, nullptr, &cap_graph, &deps, nullptr, &ndeps));
  cudaGraphNodeParams cp = {};
  cp.type = cudaGraphNodeTypeConditional;
  cp.conditional.handle = h;
  cp.conditional.type = cudaGraphCondTypeWhile;
  cp.conditional.size = 1;
  cudaGraphNode_t cnode;
  FV_CUDA(cudaGraphAddNode(&cnode, cap_graph, deps, nullptr, ndeps, &cp));
  cudaGraph_t body = cp.conditional.phGraph_out[0];
  FV_CUDA(cudaStreamBeginCaptureToGraph(bs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
  g->stream = bs;
  fv_status s2 = tpf_solve_f32(g, g->r32, g->phis[3], prec);
  if (s2 == FV_OK) s2 = launch_pass(g, prec, 3, cb, ls, &h, true);
  cudaGraph_t bg = body;
  const cudaError_t e2 = cudaStreamEndCapture(bs, &bg);
  g->stream = cs;
  FV_TRY(s2);
  FV_CUDA(e2);
  FV_CUDA(cudaStreamUpdateCaptureDependencies(cs, &cnode, nullptr, 1, cudaStreamSetCaptureDependencies));
  return launch_join(g, cb, ls);
}

// The two streams that graphs are captured on, kept by each host thread for
// the device it last captured on (creating and destroying them costs more than
// the capture) and given back with the thread.
namespace {
struct CaptureStreams {
  int dev = -1;
  cudaStream_t s[2] = {nullptr, nullptr};
  void drop() {
    for (auto& q : s) {
      if (q) cudaStreamDestroy(q);
      q = nullptr;
    }
    dev = -1;
  }
  ~CaptureStreams() { drop(); }
};
thread_local CaptureStreams t_capture;
}  // namespace

void drop_capture_streams() { t_capture.drop(); }

fv_status capture_streams(cudaStream_t* cs, cudaStream_t* bs) {
  int dev = 0;
  FV_CUDA(cudaGetDevice(&dev));
  if (t_capture.dev != dev) {
    t_capture.drop();
    for (auto& q : t_capture.s) FV_CUDA(cudaStreamCreateWithFlags(&q, cudaStreamNonBlocking));
    t_capture.dev = dev;
  }
  *cs = t_capture.s[0];
  *bs = t_capture.s[1];
  return FV_OK;
}

namespace {
// the node captured last on s
fv_status last_node(cudaStream_t s, cudaGraphNode_t* node) {
  cudaStreamCaptureStatus cst;
  cudaGraph_t graph;
  const cudaGraphNode_t* deps = nullptr;
  size_t nd = 0;
  FV_CUDA(cudaStreamGetCaptureInfo(s, &cst, nullptr, &graph, &deps, nullptr, &nd));
  if (nd != 1) { set_error("graph: unexpected capture state"); return FV_ECUDA; }
  *node = deps[0];
  return FV_OK;
}
}  // namespace

// Build (once per grid, shift, form and kind of base flow) the executable
// graph of a Krylov-vector evaluation.
static fv_status build_graph(fv_grid* g, double sigma, GraphCache& gc, int prec, bool has_u) {
  const size_t slot = &gc - g->graphs;
  gc.d_call = (CallBlock*)(g->d_eval + slot * 256);
  gc.d_loop = (LoopState*)(g->d_eval + slot * 256 + 128);
  static_assert(sizeof(CallBlock) <= 128 && sizeof(LoopState) <= 128, "evaluation slots");
  cudaStream_t cs, bs;
  FV_TRY(capture_streams(&cs, &bs));
  const cudaStream_t saved = g->stream;
  FV_CUDA(cudaMemsetAsync(gc.d_call, 0, 256, saved));
  g->stream = cs;                     // the launch helpers enqueue on g->stream
  const bool prof = g->prof_on;
  g->prof_on = false;
  g->capturing = true;
  cudaGraph_t graph = nullptr;
  bool begun = false;
  auto capture = [&]() -> fv_status {
    FV_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    begun = true;
    const bool ff = prec == FV_FF;
    if (has_u) {
      if (ff) k_base_from_call<true><<<grid1d(g->nvel), 256, 0, cs>>>(nullptr, g->U32, g->Uff, g->nvel);
      else k_base_from_call<false><<<grid1d(g->nvel), 256, 0, cs>>>(nullptr, g->U32, g->Uff, g->nvel);
      FV_CHECK_LAUNCH();
      FV_TRY(last_node(cs, &gc.base_node));
    }
    // J.v straight from the float64 vector; the float-float predictor lands in
    // vff[1], the float32 one in w32
    if (ff) FV_TRY(launch_jv_ff(g, nullptr, nullptr, g->vff[1], sigma, gc.d_call, gc.d_loop));
    else FV_TRY(launch_jv_f32(g, nullptr, nullptr, g->w32, sigma, gc.d_call, gc.d_loop));
    FV_TRY(last_node(cs, &gc.jv_node));
    if (ff) FV_TRY(launch_div_ff(g, g->vff[1], g->r32));
    else FV_TRY(launch_div_f32(g, g->w32, g->r32));
    return capture_passes(g, prec, cs, bs, gc.d_call, gc.d_loop);
  };
  fv_status st = capture();
  const cudaError_t ec = begun ? cudaStreamEndCapture(cs, &graph) : cudaSuccess;
  g->stream = saved;
  g->prof_on = prof;
  g->capturing = false;
  if (st == FV_OK && ec != cudaSuccess) st = cuda_fail(ec, "cudaStreamEndCapture", __FILE__, __LINE__);
  auto finish = [&]() -> fv_status {
    // the arguments that change from call to call: U of the base node, x and
    // the call block of the J.v node
    FV_CUDA(cudaGraphKernelNodeGetParams(gc.jv_node, &gc.jv_kp));
    gc.patch = prec == FV_FF ? jv_patch_ff() : jv_patch_f32();
    const unsigned char* a = (const unsigned char*)gc.jv_kp.kernelParams[0];
    gc.jv_args.assign(a, a + gc.patch.size);
    if (has_u) FV_CUDA(cudaGraphKernelNodeGetParams(gc.base_node, &gc.base_kp));
    FV_CUDA(cudaGraphInstantiate(&gc.exec, graph, 0));
    return FV_OK;
  };
  if (st == FV_OK) st = finish();
  if (st != FV_OK) {
    if (graph) cudaGraphDestroy(graph);
    drop_capture_streams();           // a stream may still be capturing
    (void)cudaGetLastError();
    return st;
  }
  gc.graph = graph;
  gc.sigma = sigma;
  gc.prec = prec;
  gc.has_u = has_u;
  gc.ready = true;
  return FV_OK;
}

fv_status mixed_krylov_graph(const fv_grid* gcst, const double* U, const double* x, double* out,
                             double* p, double sigma, double eps, int max_pass, double omega,
                             bool sync, int* passes, double* phi1, double* phil, double* divl,
                             int* status, int prec) {
  fv_grid* g = const_cast<fv_grid*>(gcst);
  GraphCache* gc = nullptr;
  for (auto& c : g->graphs)
    if (c.ready && c.sigma == sigma && c.prec == prec && c.has_u == (U != nullptr)) gc = &c;
  if (!gc) {
    GraphCache* slot = nullptr;
    for (auto& c : g->graphs)
      if (!c.ready) { slot = &c; break; }
    if (!slot) slot = &g->graphs[0];
    destroy_graph_cache(*slot);
    FV_TRY(build_graph(g, sigma, *slot, prec, U != nullptr));
    gc = slot;
  }
  CallBlock cb;
  cb.U = nullptr;
  cb.x = x;
  if (U) g->base_ptr = nullptr;   // the graph overwrites the stored base copy
  cb.out = out;
  cb.p = p;
  cb.sigma = (float)sigma;
  cb.eps = (float)eps;
  cb.omega = (float)omega;
  cb.max_pass = max_pass;
  LoopState* dls = gc->d_loop;
  if (U) {
    void* args[4] = {&U, &g->U32, &g->Uff, &g->nvel};
    cudaKernelNodeParams kp = gc->base_kp;
    kp.kernelParams = args;
    FV_CUDA(cudaGraphExecKernelNodeSetParams(gc->exec, gc->base_node, &kp));
  }
  {
    std::memcpy(gc->jv_args.data() + gc->patch.x, &x, sizeof x);
    std::memcpy(gc->jv_args.data() + gc->patch.cb, &cb, sizeof cb);
    void* args[1] = {gc->jv_args.data()};
    cudaKernelNodeParams kp = gc->jv_kp;
    kp.kernelParams = args;
    FV_CUDA(cudaGraphExecKernelNodeSetParams(gc->exec, gc->jv_node, &kp));
  }
  count_launch();                     // one graph launch
  FV_CUDA(cudaGraphLaunch(gc->exec, g->stream));
  if (!sync) return FV_OK;
  LoopState hls;
  FV_CUDA(cudaMemcpyAsync(&hls, dls, sizeof(LoopState), cudaMemcpyDeviceToHost, g->stream));
  FV_CUDA(cudaStreamSynchronize(g->stream));
  if (passes) *passes = hls.pass;
  if (phi1) *phi1 = hls.phi1;
  if (phil) *phil = hls.phi_last;
  if (divl) *divl = hls.div_last;
  if (status) *status = hls.status;
  if (hls.status == 4) FV_CUDA(cudaMemsetAsync(g->d_fault, 0, sizeof(unsigned), g->stream));   // reported once
  return FV_OK;
}

fv_status take_fault(const fv_grid* g, bool* hit) {
  unsigned f = 0;
  FV_CUDA(cudaMemcpyAsync(&f, g->d_fault, sizeof(unsigned), cudaMemcpyDeviceToHost, g->stream));
  FV_CUDA(cudaMemsetAsync(g->d_fault, 0, sizeof(unsigned), g->stream));
  FV_CUDA(cudaStreamSynchronize(g->stream));
  *hit = f != 0;
  return FV_OK;
}

fv_status status_error(int status) {
  switch (status) {
    case 2: set_error("SIMPLE loop reached max_pass"); return FV_ENOCONV;
    case 3: set_error("SIMPLE loop: NaN/Inf in the correction"); return FV_ENAN;
    case 4:
      set_error("a bounded wait of a pressure transform or a Gram-Schmidt step gave up (device timeout), in this "
                "call or in one queued before it on the grid");
      return FV_ETIMEOUT;
    default: return FV_OK;
  }
}

fv_status graph_take_status(fv_grid* g, int* worst, bool with_fault) {
  *worst = 0;
  bool hit = false;
  if (with_fault) FV_TRY(take_fault(g, &hit));
  if (hit) *worst = 4;
  for (auto& c : g->graphs) {
    if (!c.ready) continue;
    int w = 0;
    FV_CUDA(cudaMemcpyAsync(&w, &c.d_loop->worst, sizeof(int), cudaMemcpyDeviceToHost, g->stream));
    FV_CUDA(cudaMemsetAsync(&c.d_loop->worst, 0, sizeof(int), g->stream));
    FV_CUDA(cudaStreamSynchronize(g->stream));
    *worst = std::max(*worst, w);
  }
  return FV_OK;
}

// Back-to-back launches of one kernel class of the mixed path on the grid's
// current workspace (left by a previous evaluation), timed with CUDA events on
// the grid's stream: average device time per launch.
fv_status bench_kernel(fv_grid* g, int kind, int reps, double* ms) {
  GraphCache* gc = nullptr;
  for (auto& c : g->graphs)
    if (c.ready) gc = &c;
  if (!gc) {
    // host-driven grids have no graph yet: capture one for its device blocks
    gc = &g->graphs[0];
    FV_TRY(build_graph(g, 0.0, *gc, FV_MIXED, false));
    FV_CUDA(cudaMemsetAsync(gc->d_call, 0, sizeof(CallBlock), g->stream));
    FV_CUDA(cudaMemsetAsync(gc->d_loop, 0, sizeof(LoopState), g->stream));
  }
  cudaEvent_t e0, e1;
  FV_CUDA(cudaEventCreate(&e0));
  FV_CUDA(cudaEventCreate(&e1));
  auto one = [&]() -> fv_status {
    switch (kind) {
      case FV_K_MOMENTUM: return launch_jv_f32(g, nullptr, g->vel_buf[1], g->w32, 0.0);
      case FV_K_DIVERGENCE: return launch_div_f32(g, g->w32, g->r32);
      case FV_K_CORRECT:
        // the second pass, the first that reads a float-float v
        return launch_pass(g, FV_MIXED, 1, (const CallBlock*)gc->d_call, gc->d_loop, nullptr, false);
      case FV_K_TPF_X: return tpf_one_transform_f32(g, 0);
      case FV_K_TPF_XINV: return tpf_one_transform_f32(g, 1);
      case FV_K_TPF_YZ: return tpf_one_transform_f32(g, 2);
      default: set_error("fv_bench_kernel: unsupported kind"); return FV_EINVAL;
    }
  };
  FV_TRY(one());                                   // warm-up
  FV_CUDA(cudaEventRecord(e0, g->stream));
  for (int r = 0; r < reps; ++r) FV_TRY(one());
  FV_CUDA(cudaEventRecord(e1, g->stream));
  FV_CUDA(cudaEventSynchronize(e1));
  float t = 0.f;
  FV_CUDA(cudaEventElapsedTime(&t, e0, e1));
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  *ms = t / reps;
  return FV_OK;
}

void destroy_graph_cache(GraphCache& c) {
  if (c.exec) cudaGraphExecDestroy(c.exec);
  if (c.graph) cudaGraphDestroy(c.graph);
  c = GraphCache();
}


// ===========================================================================
// Batched instances: several grids (uneven sizes, Reynolds numbers, lid
// angles) advance one Krylov-vector evaluation each in ONE graph launch.
// The momentum predictors of all instances are computed by a persistent
// work-queue kernel (blocks pull (instance, z-tile) items from an atomic
// counter, so small and large grids share the SMs); the SIMPLE loops then run
// as concurrent graph branches, one WHILE conditional node per instance.  The
// z-tile depth (planes per work item) is picked by fv_batch_autotune.
namespace {

constexpr int kBatchMax = 32;
constexpr int kBatchBlocks = 152 * 4;
constexpr int kBand = 1024;      // cells of a plane in one work item at most

struct BatchCall {
  const double* U[kBatchMax];
  const double* x[kBatchMax];
  double* out[kBatchMax];
  float eps, sigma;
  int n;
};

struct InstDesc {
  Met<float> m;
  float* U32;
  float* x32;
  float* w32;
  float inv_re;
  int tile_base;
  int bands;                     // of a plane
};

__global__ void k_batch_init(BatchCall bc, CallBlock* dcb, LoopState* dls) {
  const int i = threadIdx.x;
  if (i >= bc.n) return;
  CallBlock c;
  c.U = bc.U[i];
  c.x = bc.x[i];
  c.out = bc.out[i];
  c.p = nullptr;
  c.sigma = bc.sigma;
  c.eps = bc.eps;
  c.omega = 1.f;
  c.max_pass = 200;
  dcb[i] = c;
  LoopState& l = dls[i];
  l.phi1 = l.phi_prev = l.phi_last = l.div_last = 0.f;
  l.pass = l.nan = l.status = 0;
}

// U and x of every instance (blockIdx.y) rounded to float32, as one launch: one
// per instance left a gap and a partial last wave twelve times over.  Bound by
// memory (24 B per entry).
__global__ void __launch_bounds__(256) k_batch_round(const InstDesc* __restrict__ d,
                                                     const CallBlock* __restrict__ cb) {
  const double* U = cb[blockIdx.y].U;
  const double* x = cb[blockIdx.y].x;
  float* U32 = d[blockIdx.y].U32;
  float* x32 = d[blockIdx.y].x32;
  const int64_t n = 3 * d[blockIdx.y].m.ncell;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    U32[e] = f64_round_f32(__ldg(U + e));
    x32[e] = f64_round_f32(__ldg(x + e));
  }
}

// Momentum predictor (Eq. 10, float32) of every instance: blocks pull work
// items (instance, ppt consecutive z-planes, a band of kBand cells of them)
// from an atomic counter, the next one while they compute.  Bands, because
// whole planes of {48 .. 96}^3 (three of each) are 864 items for the 304 blocks
// that fit at a time, the largest last: the end of the kernel was a partial
// wave of them.  With k_batch_round in place of twelve rounding launches, the
// batch of twelve went from 1160 to 1135 us.  Bound by the latency of its
// loads, yet three or four blocks per SM (80, 64 registers, spilled) were
// slower: 1155 and 1156 us against 1135 with two (128 registers).
__global__ void __launch_bounds__(256) k_batch_jv(const InstDesc* __restrict__ d, int ninst,
                                                  int total, int ppt, float shift,
                                                  unsigned* __restrict__ counter) {
  __shared__ int s_tile[2];
  if (threadIdx.x == 0) s_tile[0] = (int)atomicAdd(counter, 1u);
  __syncthreads();
  int inst = 0;                  // items come in order: the search goes on from the last one
  for (int buf = 0;; buf ^= 1) {
    const int tile = s_tile[buf];
    if (tile >= total) return;
    if (threadIdx.x == 0) s_tile[buf ^ 1] = (int)atomicAdd(counter, 1u);
    while (inst + 1 < ninst && d[inst + 1].tile_base <= tile) ++inst;
    const Met<float> m = d[inst].m;
    const float* U = d[inst].U32;
    const float* V = d[inst].x32;
    float* out = d[inst].w32;
    const float inv_re = d[inst].inv_re;
    const int bands = d[inst].bands;
    const int item = tile - d[inst].tile_base;
    const int z0 = item / bands * ppt, t0 = item % bands * kBand;
    const int nx = m.n[0], ny = m.n[1], nz = m.n[2];
    const int plane = nx * ny;
    const int nc = (int)m.ncell;
    const int st[3] = {1, nx, plane};
    const int t1 = min(plane, t0 + kBand);
    for (int t = t0 + (int)threadIdx.x; t < t1; t += blockDim.x) {
      const int i = t % nx, j = t / nx;
      for (int kk = 0; kk < ppt; ++kk) {
        const int k = z0 + kk;
        if (k >= nz) break;
        const int pos[3] = {i, j, k};
        const int base = k * plane + t;
        float r0 = 0.f, r1 = 0.f, r2 = 0.f;
        if (i > 0)
          r0 = stencil::momentum_face<float, 0, true, float>(m, U, V, base, pos, st, inv_re, 0.f, shift);
        if (j > 0)
          r1 = stencil::momentum_face<float, 1, true, float>(m, U, V, base, pos, st, inv_re, 0.f, shift);
        if (k > 0)
          r2 = stencil::momentum_face<float, 2, true, float>(m, U, V, base, pos, st, inv_re, 0.f, shift);
        out[base] = r0;
        out[nc + base] = r1;
        out[2 * nc + base] = r2;
      }
    }
    __syncthreads();             // the next item is there, and everyone has read this one
  }
}

}  // namespace

struct BatchImpl {
  int n = 0;
  int ppt = 1;
  double sigma = 0.0;
  fv_grid* grids[kBatchMax] = {};
  cudaStream_t stream = nullptr;
  CallBlock* d_call = nullptr;
  LoopState* d_loop = nullptr;
  InstDesc* d_desc = nullptr;
  unsigned* d_counter = nullptr;
  int total_tiles = 0;
  double re[kBatchMax] = {};      // each instance's Re when the descriptors were uploaded
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  cudaGraphNode_t init_node = nullptr;
  bool ready = false;
};

static fv_status batch_descriptors(BatchImpl& b) {
  std::vector<InstDesc> h(b.n);
  int base = 0;
  for (int i = 0; i < b.n; ++i) {
    fv_grid* g = b.grids[i];
    h[i].m = g->met_f;
    h[i].U32 = g->U32;
    h[i].x32 = g->x32;
    h[i].w32 = g->w32;
    h[i].inv_re = float(1.0 / g->re);
    b.re[i] = g->re;
    h[i].tile_base = base;
    h[i].bands = (g->n[0] * g->n[1] + kBand - 1) / kBand;
    base += (g->n[2] + b.ppt - 1) / b.ppt * h[i].bands;
  }
  b.total_tiles = base;
  FV_CUDA(cudaMemcpy(b.d_desc, h.data(), b.n * sizeof(InstDesc), cudaMemcpyHostToDevice));
  return FV_OK;
}

static fv_status launch_batch_jv(BatchImpl& b, cudaStream_t s) {
  FV_CUDA(cudaMemsetAsync(b.d_counter, 0, sizeof(unsigned), s));
  const int blocks = std::min(kBatchBlocks, b.total_tiles);
  count_launch();
  k_batch_jv<<<blocks, 256, 0, s>>>(b.d_desc, b.n, b.total_tiles, b.ppt, float(b.sigma), b.d_counter);
  FV_CHECK_LAUNCH();
  return FV_OK;
}

static void batch_release_graph(BatchImpl& b) {
  if (b.exec) cudaGraphExecDestroy(b.exec);
  if (b.graph) cudaGraphDestroy(b.graph);
  b.exec = nullptr;
  b.graph = nullptr;
  b.ready = false;
}

// Capture the batch graph: init -> round -> batched J.v -> per-instance branches
// {D w -> three times (TPF -> pass) -> WHILE{TPF -> pass} -> join}.
static fv_status batch_build_graph(BatchImpl& b) {
  batch_release_graph(b);
  FV_TRY(batch_descriptors(b));
  cudaStream_t cs, bs;
  FV_TRY(capture_streams(&cs, &bs));
  std::vector<cudaStream_t> saved(b.n);
  for (int i = 0; i < b.n; ++i) {
    saved[i] = b.grids[i]->stream;
    b.grids[i]->capturing = b.grids[i]->in_batch = true;
  }
  cudaGraph_t graph = nullptr;
  bool begun = false;
  auto capture = [&]() -> fv_status {
    FV_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    begun = true;
    BatchCall bc = {};
    k_batch_init<<<1, kBatchMax, 0, cs>>>(bc, b.d_call, b.d_loop);
    FV_CHECK_LAUNCH();
    int64_t longest = 0;
    for (int i = 0; i < b.n; ++i) longest = std::max(longest, b.grids[i]->nvel);
    k_batch_round<<<dim3(grid1d(longest), b.n), 256, 0, cs>>>(b.d_desc, b.d_call);
    FV_CHECK_LAUNCH();
    FV_TRY(launch_batch_jv(b, cs));
    // one stream captures every branch: each starts from the J.v node, and the
    // capture ends where they all have
    cudaGraphNode_t jv;
    FV_TRY(last_node(cs, &jv));
    std::vector<cudaGraphNode_t> ends(b.n);
    for (int i = 0; i < b.n; ++i) {
      fv_grid* g = b.grids[i];
      g->stream = cs;
      FV_CUDA(cudaStreamUpdateCaptureDependencies(cs, &jv, nullptr, 1, cudaStreamSetCaptureDependencies));
      FV_TRY(launch_div_f32(g, g->w32, g->r32));
      FV_TRY(capture_passes(g, FV_MIXED, cs, bs, b.d_call + i, b.d_loop + i));
      FV_TRY(last_node(cs, &ends[i]));
    }
    FV_CUDA(cudaStreamUpdateCaptureDependencies(cs, ends.data(), nullptr, ends.size(),
                                                cudaStreamSetCaptureDependencies));
    return FV_OK;
  };
  fv_status st = capture();
  const cudaError_t ec = begun ? cudaStreamEndCapture(cs, &graph) : cudaSuccess;
  for (int i = 0; i < b.n; ++i) {
    b.grids[i]->stream = saved[i];
    b.grids[i]->capturing = b.grids[i]->in_batch = false;
  }
  if (st == FV_OK && ec != cudaSuccess) st = cuda_fail(ec, "cudaStreamEndCapture", __FILE__, __LINE__);
  if (st != FV_OK) {
    if (graph) cudaGraphDestroy(graph);
    drop_capture_streams();           // a stream may still be capturing
    (void)cudaGetLastError();
    return st;
  }
  size_t nroot = 0;
  FV_CUDA(cudaGraphGetRootNodes(graph, nullptr, &nroot));
  std::vector<cudaGraphNode_t> roots(nroot);
  FV_CUDA(cudaGraphGetRootNodes(graph, roots.data(), &nroot));
  if (nroot != 1) {
    cudaGraphDestroy(graph);
    set_error("batch graph: unexpected root count");
    return FV_ECUDA;
  }
  b.init_node = roots[0];
  FV_CUDA(cudaGraphInstantiate(&b.exec, graph, 0));
  b.graph = graph;
  b.ready = true;
  return FV_OK;
}

}  // namespace fv

struct fv_batch {
  fv::BatchImpl impl;
};

using namespace fv;

extern "C" {

fv_status fv_batch_set_tile(fv_batch* b, int ppt);

fv_status fv_batch_create(int n, fv_grid* const* grids, void* cuda_stream, fv_batch** out) {
  if (!out || !grids || n < 1 || n > kBatchMax) {
    set_error("fv_batch_create: need 1..32 grids");
    return FV_EINVAL;
  }
  *out = nullptr;
  for (int i = 0; i < n; ++i)
    if (!grids[i]) { set_error("fv_batch_create: NULL grid"); return FV_EINVAL; }
  fv_batch* b = new fv_batch();
  BatchImpl& B = b->impl;
  B.n = n;
  for (int i = 0; i < n; ++i) B.grids[i] = grids[i];
  B.stream = (cudaStream_t)cuda_stream;
  cudaError_t e = cudaSuccess;
  if (e == cudaSuccess) e = cudaMalloc((void**)&B.d_call, kBatchMax * sizeof(CallBlock));
  if (e == cudaSuccess) e = cudaMalloc((void**)&B.d_loop, kBatchMax * sizeof(LoopState));
  if (e == cudaSuccess) e = cudaMalloc((void**)&B.d_desc, kBatchMax * sizeof(InstDesc));
  if (e == cudaSuccess) e = cudaMalloc((void**)&B.d_counter, sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMemset(B.d_loop, 0, kBatchMax * sizeof(LoopState));
  if (e != cudaSuccess) {
    cuda_fail(e, "cudaMalloc", __FILE__, __LINE__);
    fv_batch_destroy(b);
    return FV_ENOMEM;
  }
  *out = b;
  return FV_OK;
}

void fv_batch_destroy(fv_batch* b) {
  if (!b) return;
  BatchImpl& B = b->impl;
  batch_release_graph(B);
  void* ptrs[] = {B.d_call, B.d_loop, B.d_desc, B.d_counter};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  delete b;
}

fv_status fv_batch_krylov(fv_batch* b, const double* const* U, const double* const* x,
                          double* const* out, double eps, double sigma, int* passes) {
  if (!b || !U || !x || !out) { set_error("fv_batch_krylov: NULL argument"); return FV_EINVAL; }
  BatchImpl& B = b->impl;
  if (!(eps > 0) || sigma < 0) { set_error("fv_batch_krylov: bad eps/sigma"); return FV_EINVAL; }
  BatchCall bc = {};
  for (int i = 0; i < B.n; ++i) {
    if (!U[i] || !x[i] || !out[i] || x[i] == out[i]) {
      set_error("fv_batch_krylov: bad pointer");
      return FV_EINVAL;
    }
    bc.U[i] = U[i];
    bc.x[i] = x[i];
    bc.out[i] = out[i];
  }
  bc.n = B.n;
  bc.eps = (float)eps;
  bc.sigma = (float)sigma;
  if (!B.ready || B.sigma != sigma) {
    B.sigma = sigma;
    FV_TRY(batch_build_graph(B));
  } else {
    // an instance's Re changed (fv_grid_set_re): the graph reads the
    // descriptor table at run time, so uploading it again is enough
    bool stale = false;
    for (int i = 0; i < B.n; ++i) stale |= B.grids[i]->re != B.re[i];
    if (stale) {
      FV_CUDA(cudaStreamSynchronize(B.stream));
      FV_TRY(batch_descriptors(B));
    }
  }
  void* dcb = B.d_call;
  void* dls = B.d_loop;
  void* args[3] = {&bc, &dcb, &dls};
  cudaKernelNodeParams kp = {};
  kp.func = (void*)k_batch_init;
  kp.gridDim = dim3(1);
  kp.blockDim = dim3(kBatchMax);
  kp.kernelParams = args;
  FV_CUDA(cudaGraphExecKernelNodeSetParams(B.exec, B.init_node, &kp));
  // the batch rounds each instance's U into the grid's U32, replacing a
  // base flow registered on that grid
  for (int i = 0; i < B.n; ++i) B.grids[i]->base_ptr = nullptr;
  count_launch();
  FV_CUDA(cudaGraphLaunch(B.exec, B.stream));
  if (passes) {
    std::vector<LoopState> h(B.n);
    FV_CUDA(cudaMemcpyAsync(h.data(), B.d_loop, B.n * sizeof(LoopState), cudaMemcpyDeviceToHost,
                            B.stream));
    FV_CUDA(cudaStreamSynchronize(B.stream));
    for (int i = 0; i < B.n; ++i) passes[i] = h[i].pass;
    int worst = 1;
    for (int i = 0; i < B.n; ++i) {
      if (h[i].status == 4) FV_CUDA(cudaMemsetAsync(B.grids[i]->d_fault, 0, sizeof(unsigned), B.stream));
      worst = std::max(worst, h[i].status == 0 ? 2 : h[i].status);
    }
    if (worst != 1) {
      const fv_status e = status_error(worst);
      set_error(std::string("fv_batch_krylov: an instance did not converge: ") + fv_last_error());
      return e;
    }
  }
  return FV_OK;
}

fv_status fv_batch_autotune(fv_batch* b, int* best_ppt, double* ms) {
  if (!b || !best_ppt) { set_error("fv_batch_autotune: NULL argument"); return FV_EINVAL; }
  BatchImpl& B = b->impl;
  static const int cand[4] = {1, 2, 4, 8};
  cudaEvent_t e0, e1;
  FV_CUDA(cudaEventCreate(&e0));
  FV_CUDA(cudaEventCreate(&e1));
  double best = 1e30;
  int bp = 1;
  for (int c = 0; c < 4; ++c) {
    B.ppt = cand[c];
    FV_TRY(batch_descriptors(B));
    FV_TRY(launch_batch_jv(B, B.stream));          // warm-up
    FV_CUDA(cudaEventRecord(e0, B.stream));
    for (int r = 0; r < 10; ++r) FV_TRY(launch_batch_jv(B, B.stream));
    FV_CUDA(cudaEventRecord(e1, B.stream));
    FV_CUDA(cudaEventSynchronize(e1));
    float t = 0.f;
    FV_CUDA(cudaEventElapsedTime(&t, e0, e1));
    if (ms) ms[c] = t / 10.0;
    if (t < best) { best = t; bp = cand[c]; }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  *best_ppt = bp;
  B.ppt = 0;                                       // force the graph rebuild below
  return fv_batch_set_tile(b, bp);
}

fv_status fv_batch_set_tile(fv_batch* b, int ppt) {
  if (!b || ppt < 1 || ppt > 64) { set_error("fv_batch_set_tile: bad argument"); return FV_EINVAL; }
  BatchImpl& B = b->impl;
  if (B.ppt != ppt) {
    B.ppt = ppt;
    batch_release_graph(B);
  }
  return FV_OK;
}

}  // extern "C"

extern "C" fv_status fv_bench_kernel(fv_grid* g, int kind, int reps, double* ms_per_launch) {
  if (!g || !ms_per_launch || reps < 1) { fv::set_error("fv_bench_kernel: bad argument"); return FV_EINVAL; }
  return fv::bench_kernel(g, kind, reps, ms_per_launch);
}
