// The server (sgn_serve.cu) on a fake device: host memory with a limit, streams that have always
// finished, layouts and states that only occupy memory.  Each scenario prints one line.
#include <cuda_runtime.h>

#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "sgn.h"
#include "sgn_2d.h"

// ---- memory -------------------------------------------------------------------------------
static std::mutex mem_mu;
static std::map<void*, size_t> blocks;
static size_t limit_bytes = (size_t)1 << 40, used_bytes = 0;
struct CUmemPoolHandle_st {
  size_t threshold = 0, reserved = 0, in_use = 0;
  std::map<void*, size_t> live;
};
static CUmemPoolHandle_st default_pool;

static cudaError_t get(void** p, size_t n) {
  std::lock_guard<std::mutex> lk(mem_mu);
  if (used_bytes + n > limit_bytes) return cudaErrorMemoryAllocation;
  used_bytes += n;
  *p = malloc(n);
  blocks[*p] = n;
  return cudaSuccess;
}
static cudaError_t pool_get(void** p, size_t n, CUmemPoolHandle_st* m) {
  std::lock_guard<std::mutex> lk(mem_mu);
  const size_t grow = m->in_use + n > m->reserved ? m->in_use + n - m->reserved : 0;
  if (used_bytes + grow > limit_bytes) return cudaErrorMemoryAllocation;
  used_bytes += grow;
  m->reserved += grow;
  m->in_use += n;
  *p = malloc(n);
  m->live[*p] = n;
  return cudaSuccess;
}
static void pool_trim(CUmemPoolHandle_st* m, size_t keep) {
  const size_t to = m->in_use > keep ? m->in_use : keep;
  if (m->reserved > to) {
    used_bytes -= m->reserved - to;
    m->reserved = to;
  }
}
static bool pool_put(void* p, CUmemPoolHandle_st* m) {
  auto it = m->live.find(p);
  if (it == m->live.end()) return false;
  m->in_use -= it->second;
  m->live.erase(it);
  free(p);
  pool_trim(m, m->threshold);
  return true;
}
static CUmemPoolHandle_st* server_pool = nullptr;
static std::atomic<int> relaxed{0}, strict_frees{0};
static std::atomic<bool> watch_frees{false};

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) { return get(p, n); }
cudaError_t cudaFree(void* p) {
  if (watch_frees && !relaxed) strict_frees++;
  std::lock_guard<std::mutex> lk(mem_mu);
  auto it = blocks.find(p);
  if (it == blocks.end()) {                  // of a pool, or null
    pool_put(p, &default_pool);
    return cudaSuccess;
  }
  used_bytes -= it->second;
  blocks.erase(it);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return pool_get(p, n, &default_pool); }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t m, cudaStream_t) {
  return pool_get(p, n, m);
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
  std::lock_guard<std::mutex> lk(mem_mu);
  if (!pool_put(p, &default_pool) && server_pool) pool_put(p, server_pool);
  return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* m, const cudaMemPoolProps*) {
  *m = server_pool = new CUmemPoolHandle_st();
  return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t m) {
  std::lock_guard<std::mutex> lk(mem_mu);
  used_bytes -= m->reserved;
  server_pool = nullptr;
  delete m;
  return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t m, cudaMemPoolAttr, void* v) {
  m->threshold = *static_cast<uint64_t*>(v);
  return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t m, size_t keep) {
  std::lock_guard<std::mutex> lk(mem_mu);
  pool_trim(m, keep);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* fr, size_t* tot) {
  *fr = *tot = (size_t)1 << 30;              // the device's; another program holds some of it
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int* lo, int* hi) { *lo = 0; *hi = -3; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = reinterpret_cast<cudaStream_t>(malloc(1));
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned f, int) {
  return cudaStreamCreateWithFlags(s, f);
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  *e = reinterpret_cast<cudaEvent_t>(malloc(1));
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode* m) {
  relaxed = *m == cudaStreamCaptureModeRelaxed;
  *m = relaxed ? cudaStreamCaptureModeGlobal : cudaStreamCaptureModeRelaxed;
  return cudaSuccess;
}
}

// ---- the library under the server ------------------------------------------------------------
struct sgn_ctx {};
struct sgn_layout {
  std::vector<long long> off;
  void* mem = nullptr;
  bool refused = false;                      // its solve graph could not be built
};
struct sgn_state {
  void* mem = nullptr;
};
static size_t layout_bytes = 0, state_bytes = 0;       // per point
static std::atomic<int> layouts{0};
static std::atomic<bool> refuse_graph{false};

extern "C" {
sgn_status sgn_create(sgn_ctx** c, int, size_t) { *c = new sgn_ctx(); return SGN_OK; }
void sgn_destroy(sgn_ctx* c) { delete c; }
sgn_status sgn_layout_create(sgn_ctx*, int count, const sgn_grid* g, sgn_layout** out) {
  *out = nullptr;
  sgn_layout* l = new sgn_layout();
  l->off.assign(1, 0);
  for (int i = 0; i < count; ++i) l->off.push_back(l->off.back() + (long long)g[i].nx * g[i].ny);
  if (get(&l->mem, layout_bytes * l->off.back()) != cudaSuccess) {
    delete l;
    return SGN_ERR_NOMEM;
  }
  layouts++;
  *out = l;
  return SGN_OK;
}
void sgn_layout_destroy(sgn_layout* l) {
  cudaFree(l->mem);
  delete l;
}
sgn_status sgn_layout_offsets(const sgn_layout* l, long long* o) {
  memcpy(o, l->off.data(), sizeof(long long) * l->off.size());
  return SGN_OK;
}
long long sgn_layout_points(const sgn_layout* l) { return l->off.back(); }
sgn_status sgn_spectral_grad(sgn_ctx*, const sgn_layout*, const double*, double*, sgn_stream) {
  return SGN_OK;
}
sgn_status sgn_apply_operator(sgn_ctx*, const sgn_layout*, const double*, const double*,
                              const double*, double*, sgn_stream) {
  return SGN_OK;
}
sgn_status sgn_pcg_async(sgn_ctx*, const sgn_layout* l, const double*, const double*, const double*,
                         double*, double, int, sgn_precision, sgn_pcg_info* info, sgn_stream) {
  if (refuse_graph.exchange(false)) const_cast<sgn_layout*>(l)->refused = true;
  for (size_t i = 0; i + 1 < l->off.size(); ++i) {
    info[i] = sgn_pcg_info{};
    info[i].iters = l->refused ? 2 : 1;      // 2: driven by the host
  }
  return SGN_OK;
}
sgn_status sgn_state_create(sgn_ctx*, const sgn_layout* l, double*, double*, double*, const double*,
                            double*, sgn_state** out) {
  *out = nullptr;
  sgn_state* s = new sgn_state();
  if (get(&s->mem, state_bytes * l->off.back()) != cudaSuccess) {
    delete s;
    return SGN_ERR_NOMEM;
  }
  *out = s;
  return SGN_OK;
}
sgn_status sgn_state_init(sgn_state*, sgn_stream) { return SGN_OK; }
void sgn_state_free(sgn_state* s) {
  cudaFree(s->mem);
  delete s;
}
sgn_status sgn_state_get_stats(sgn_state*, sgn_state_stats* o) {
  *o = sgn_state_stats{};
  return SGN_OK;
}
sgn_status sgn_step_rk4(sgn_state*, const double*, int, const sgn_opts*, sgn_stream) { return SGN_OK; }
sgn_status sgn_step_abk(sgn_state*, int, const double*, int, const sgn_opts*, sgn_stream) {
  return SGN_OK;
}
sgn_status sgn_step_linimp(sgn_state*, const double*, int, const sgn_opts*, sgn_stream) {
  return SGN_OK;
}
}
namespace sgn {
static double hist[1 << 20];
sgn_status state_attach(sgn_state*, cudaStream_t) { return SGN_OK; }
double* state_rk4_prev(sgn_state*) { return hist; }
double* state_rk4_last(sgn_state*) { return hist; }
bool layout_graph_refused(const sgn_layout* l) { return l->refused; }
bool mr2d_side_ok(int) { return false; }
bool mr_size_ok(int) { return false; }
}  // namespace sgn

// ---- scenarios ------------------------------------------------------------------------------
static double host[3 << 20];

// one request; its status, and the iterations of its report
static int serve(sgn_server* S, int kind, int dim, int n, double L, sgn_scheme scheme, int* iters) {
  sgn_request q{};
  q.kind = (decltype(q.kind))kind;
  q.grid = sgn_grid{dim, n, dim == 2 ? n : 1, L, dim == 2 ? L : 0.0, 9.81};
  q.eta = q.u_or_b = q.h = host;
  q.host_memory = 1;
  q.scheme = scheme;
  q.dt = 0.1;
  q.nsteps = 2;
  q.opts.rtol = 1e-10;
  q.opts.maxit = 100;
  q.opts.prec = SGN_PREC_MIXED;
  uint64_t t = 0;
  sgn_status e = sgn_batch_submit(S, &q, &t);
  if (e) return e;
  sgn_result r{};
  for (int i = 0; i < 40000 && (e = sgn_batch_poll(S, t, &r)) == SGN_ERR_PENDING; ++i)
    std::this_thread::sleep_for(std::chrono::microseconds(100));
  if (iters) *iters = r.info.iters;
  sgn_result_release(S, t);
  return e;
}

int main(int argc, char** argv) {
  const std::string what = argc > 1 ? argv[1] : "";
  sgn_ctx ctx;
  sgn_server* S = nullptr;
  if (sgn_server_create(&ctx, 0.0, &S)) return 2;
  auto used = [&] {
    std::lock_guard<std::mutex> lk(mem_mu);
    return used_bytes;
  };
  layout_bytes = state_bytes = 400;
  // 24 grids of 64 x 64: their layouts are kept (39 MB), and 3 MB of the pool
  auto fill = [&] {
    for (int i = 0; i < 24; ++i)
      if (serve(S, SGN_REQ_SOLVE, 2, 64, 10.0 + i, SGN_SCHEME_RK4, nullptr)) exit(3);
    for (int i = 0; i < 2000 && used() < 39000000; ++i)
      std::this_thread::sleep_for(std::chrono::milliseconds(1));
    if (used() < 39000000) exit(4);
  };
  int st = -1, it = 0;
  if (what == "submit") {                    // no room for the request's own arrays
    fill();
    limit_bytes = used() + 100000;
    st = serve(S, SGN_REQ_SOLVE, 2, 128, 5.0, SGN_SCHEME_RK4, &it);
  } else if (what == "state") {              // a 2d run: none for its state
    fill();
    layout_bytes = 100;
    state_bytes = 1000;
    limit_bytes = used() + 6000000;
    st = serve(S, SGN_REQ_RUN, 2, 128, 5.0, SGN_SCHEME_RK4, &it);
  } else if (what == "solve1d") {            // a 1d solve: none for its group's layout
    if (serve(S, SGN_REQ_SOLVE, 1, 4096, 5.0, SGN_SCHEME_RK4, nullptr)) return 3;
    fill();
    limit_bytes = used() + 1000000;
    st = serve(S, SGN_REQ_SOLVE, 1, 4096, 5.0, SGN_SCHEME_RK4, &it);
  } else if (what == "pack1d") {             // none for its packed arrays
    layout_bytes = 1;
    if (serve(S, SGN_REQ_SOLVE, 1, 16384, 5.0, SGN_SCHEME_RK4, nullptr)) return 3;
    layout_bytes = 400;
    fill();
    layout_bytes = 1;
    limit_bytes = used() + 700000;
    st = serve(S, SGN_REQ_SOLVE, 1, 16384, 5.0, SGN_SCHEME_RK4, &it);
  } else if (what == "run1d" || what == "multistep1d") {     // a run: none for its layout or state
    fill();
    limit_bytes = used() + 1000000;
    st = serve(S, SGN_REQ_RUN, 1, 4096, 5.0, what == "run1d" ? SGN_SCHEME_RK4 : SGN_SCHEME_AB2, &it);
  } else if (what == "too_large") {          // more than there is: refused, as before
    fill();
    limit_bytes = used() + 1000000;
    layout_bytes = 40000;
    st = serve(S, SGN_REQ_SOLVE, 2, 64, 5.0, SGN_SCHEME_RK4, &it);
  } else if (what == "graph") {              // a solve graph that could not be built, once
    refuse_graph = true;
    if (serve(S, SGN_REQ_SOLVE, 2, 64, 10.0, SGN_SCHEME_RK4, &it) || it != 2) return 3;
    std::this_thread::sleep_for(std::chrono::milliseconds(100));
    st = serve(S, SGN_REQ_SOLVE, 2, 64, 10.0, SGN_SCHEME_RK4, &it);
    const int n = layouts;                   // and the next request takes the kept layout
    std::this_thread::sleep_for(std::chrono::milliseconds(100));
    if (serve(S, SGN_REQ_SOLVE, 2, 64, 10.0, SGN_SCHEME_RK4, nullptr) || layouts != n) st = 6;
  } else if (what == "idle") {               // nothing to do: the memory goes back by itself
    const size_t before = used();
    fill();
    watch_frees = true;
    for (int i = 0; i < 8000 && used() > before; ++i)
      std::this_thread::sleep_for(std::chrono::milliseconds(1));
    watch_frees = false;
    st = used() > before ? 1 : 0;
    it = strict_frees;                       // frees that a capture of another thread would see
    if (serve(S, SGN_REQ_SOLVE, 2, 64, 10.0, SGN_SCHEME_RK4, nullptr)) st = 5;
  }
  printf("status %d iters %d\n", st, it);
  sgn_server_destroy(S);
  printf("left %zu blocks\n", blocks.size());
  return 0;
}
