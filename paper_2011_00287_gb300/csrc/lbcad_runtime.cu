// lbcad_runtime.cu -- host runtime behind the C ABI of include/lbcad.h: parameter
// validation, device memory pool, the seeded initial state, the step loop (optionally
// replayed from a captured CUDA graph), field exchange and FP64 observables.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <algorithm>
#include <exception>
#include <memory>
#include <new>
#include <string>
#include <type_traits>
#include <utility>
#include <vector>

#include "lbcad.h"
#include "lbcad_coefs.h"
#include "lbcad_internal.h"
#include "lbcad_validate.h"

using namespace lbcad;

namespace {

thread_local std::string g_create_err;

struct Inst {
  lbcad_grid g;
  lbcad_params p;
  long long N = 0;
  void* gb[2] = {nullptr, nullptr};  // populations, parity 0/1
  void* qb[2] = {nullptr, nullptr};
  void* pb[2] = {nullptr, nullptr};
  void* ub[2] = {nullptr, nullptr};
  void* S = nullptr;   // default path: stress, mu, flux divergence, psi (12 per site)
  long long SN = 0;    // sites it holds
  void* sig = nullptr;
  void* mu = nullptr;
  void* H = nullptr;
  void* rq = nullptr;  // Heun: right-hand side at t (6 per site)
  void* qp = nullptr;  // Heun: predicted Q, psi (6 per site)
  void* trig = nullptr;  // (cos, sin) of 2 pi x/nx, 2 pi y/ny, 2 pi z/nz for the centroid sums
  long long blk0 = 0, nblk = 0;
};

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    cudaGetDevice(&prev);
    if (dev >= 0 && dev != prev) cudaSetDevice(dev);
  }
  ~DeviceGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

}  // namespace

void lbcad::set_thread_error(const char* msg) { g_create_err = msg ? msg : ""; }

struct lbcad_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  int prec = LBCAD_FP32;
  lbcad_alloc_fn alloc = nullptr;
  lbcad_free_fn free = nullptr;
  void* user = nullptr;
  std::vector<Inst> inst;
  std::vector<void*> allocs;
  void* desc[2] = {nullptr, nullptr};
  long long total_blocks = 0;
  int64_t step = 0;
  int graph_steps = 0;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t gexec = nullptr;
  double* obs_partial = nullptr;
  double* obs_out = nullptr;
  double* staging = nullptr;
  size_t staging_bytes = 0;
  int path = LBCAD_PATH_FUSED;
  int integrator = LBCAD_EULER;
  int coupling = LBCAD_LAGGED;
  int vel = LBCAD_D3Q19;          // velocity set of the populations
  int lb_form = LBCAD_LB_BODY_FORCE;
  int stencil = LBCAD_STENCIL_ISO;
  bool scratch_ready = false;
  MarchItem* items = nullptr;  // work items of the default path, all lists of all groups
  size_t items_cap = 0;        // bytes, as the other capacities
  StepPlan plan;               // the launches of a step and their scratch
  ScratchRule rule;            // the bound on the scratch that the plan was made for
  char* scratch = nullptr;     // of the Euler step, which its launches use in turn
  std::vector<StepWork> work;  // one per launch of the plan
  std::vector<FusedObs> obs;
  std::vector<MarchDesc<float>> desc32[2];  // by step parity
  std::vector<MarchDesc<double>> desc64[2];
  int cfg_index = 0;
  // a6 sums of the fused step (see FusedObs): slots per (block, run of items), per-instance
  // bookkeeping, and the sums of the latest state; obs_valid while they describe the state
  double* obs_slots = nullptr;
  size_t obs_slots_cap = 0;
  int* obs_map = nullptr;  // per group: slot_inst [nslots], then nslot, slot_lo, slot_hi [ninst each]
  size_t obs_map_cap = 0;
  unsigned* obs_cnt = nullptr;
  double* obs_latest = nullptr;
  bool observe = true;     // fused steps form the a6 sums (lbcad_set_observe)
  bool obs_valid = false;
  void* adj_lam = nullptr;  // cotangent of the initial state of the last lbcad_adjoint
  void* adj_host = nullptr;  // pinned: the gradient's way to the caller's memory
  size_t adj_host_bytes = 0;
  // buffers of lbcad_adjoint, kept for the next call (reused when large enough)
  void* adj_buf[8] = {};
  size_t adj_bytes[8] = {};
  std::string err;
  size_t elem() const { return prec == LBCAD_FP64 ? sizeof(double) : sizeof(float); }
  // the radius-2 stencils run on the staged path only
  bool staged_only() const { return stencil != LBCAD_STENCIL_ISO; }
  // sync coupling or Heun on the fused path: the LB half in k_march_lb on a fixed tile
  // shape, then the order-parameter kernels
  bool sync_split() const { return !staged_only() && (coupling == LBCAD_SYNC || integrator == LBCAD_HEUN); }
  // D3Q19 with the body force: the two-kernel path and the adjoint cover this LB only
  bool default_lb() const { return vel == LBCAD_D3Q19 && lb_form == LBCAD_LB_BODY_FORCE; }
  // variant of the fused kernels (see LaunchFused)
  int fused_variant() const { return (vel == LBCAD_D3Q15 ? 1 : 0) + (lb_form == LBCAD_LB_STRESS_EQ ? 2 : 0); }
  int q() const { return vel == LBCAD_D3Q15 ? 15 : 19; }
};

namespace {

int fail(lbcad_ctx* c, int code, const std::string& msg) {
  if (c) c->err = msg; else g_create_err = msg;
  return code;
}

// What an entry point returns for an exception of the host runtime (no memory for a list, a vector or a message).
int caught(lbcad_ctx* c) noexcept {
  std::string& err = c ? c->err : g_create_err;
  err.clear();
  err += "no host memory";  // fits the string's own buffer: cannot throw in turn
  return LBCAD_E_OOM;
}

#define CK(ctx, call)                                                                          \
  do {                                                                                         \
    cudaError_t e_ = (call);                                                                   \
    if (e_ != cudaSuccess)                                                                     \
      return fail((ctx), LBCAD_E_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_));    \
  } while (0)

void* dev_alloc(lbcad_ctx* c, size_t bytes) {
  bytes = (bytes + 255) & ~(size_t)255;
  void* p = nullptr;
  if (c->allocs.size() == c->allocs.capacity()) c->allocs.reserve(2 * c->allocs.size() + 16);  // before there is a p to lose
  if (c->alloc) {
    p = c->alloc(bytes, c->user);
  } else if (cudaMalloc(&p, bytes) != cudaSuccess) {
    cudaGetLastError();
    p = nullptr;
  }
  if (p) c->allocs.push_back(p);
  return p;
}

// Gives one allocation of the context back, with no work on it in flight.
void dev_free(lbcad_ctx* c, void* p) {
  c->allocs.erase(std::find(c->allocs.begin(), c->allocs.end(), p));
  if (c->free) c->free(p, c->user); else cudaFree(p);
}

// Makes `p` hold at least `bytes`: a larger buffer replaces it (the old one stays with the context until it is
// destroyed).  If there is none, p and its capacity stay as they were.
template <typename P>
bool grow(lbcad_ctx* c, P*& p, size_t& cap, size_t bytes) {
  if (bytes <= cap) return true;
  P* q = (P*)dev_alloc(c, bytes);
  if (!q) return false;
  p = q;
  cap = bytes;
  return true;
}

// Buffer i of lbcad_adjoint: the one of an earlier call if it is large enough, else a new one
// (the old one stays with the context until it is destroyed).
void* adj_buffer(lbcad_ctx* c, int i, size_t bytes) {
  if (c->adj_buf[i] && c->adj_bytes[i] >= bytes) return c->adj_buf[i];
  void* p = dev_alloc(c, bytes);
  if (p) {
    c->adj_buf[i] = p;
    c->adj_bytes[i] = bytes;
  }
  return p;
}

void release(lbcad_ctx* c) {
  if (!c) return;
  DeviceGuard dg(c->device);
  if (c->stream) cudaStreamSynchronize(c->stream);
  if (c->gexec) cudaGraphExecDestroy(c->gexec);
  if (c->graph) cudaGraphDestroy(c->graph);
  if (c->adj_host) cudaFreeHost(c->adj_host);
  for (void* p : c->allocs) {
    if (c->free) c->free(p, c->user); else cudaFree(p);
  }
  c->allocs.clear();
  if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
}

template <typename T>
InstDesc<T> make_desc(const Inst& I, int parity) {
  InstDesc<T> d;
  std::memset(&d, 0, sizeof(d));
  d.nx = I.g.nx; d.ny = I.g.ny; d.nz = I.g.nz;
  d.vel = (I.p.lattice == LBCAD_D3Q15) ? 1 : 0;
  d.N = I.N;
  d.blk0 = I.blk0;
  d.nblk = I.nblk;
  const int a = parity, b = parity ^ 1;
  d.g_in = (const T*)I.gb[a]; d.g_out = (T*)I.gb[b];
  d.q_in = (const T*)I.qb[a]; d.q_out = (T*)I.qb[b];
  d.psi_in = (const T*)I.pb[a]; d.psi_out = (T*)I.pb[b];
  d.u_in = (const T*)I.ub[a]; d.u_out = (T*)I.ub[b];
  d.sig = (T*)I.sig; d.mu = (T*)I.mu; d.H = (T*)I.H;
  d.rq = (T*)I.rq; d.qp = (T*)I.qp;
  d.trig = (const T*)I.trig;
  d.c = coefs<T>(I.p);
  return d;
}

template <typename T>
MarchDesc<T> make_march_desc(const Inst& I, int parity, bool shifted) {
  MarchDesc<T> d;
  std::memset(&d, 0, sizeof(d));
  d.nx = I.g.nx; d.ny = I.g.ny; d.nz = I.g.nz;
  d.plane = (unsigned)((long long)I.g.nx * I.g.ny);
  d.N = (unsigned)I.N;
  const long long N = I.N;
  const int a = parity, b = parity ^ 1, q = (I.p.lattice == LBCAD_D3Q15) ? 15 : 19;
  auto comps = [&](auto* dst, void* base, int n, long long stride) {
    for (int k = 0; k < n; ++k) dst[k] = base ? (T*)base + k * stride : nullptr;
  };
  comps(d.g_in, I.gb[a], q, N);
  comps(d.g_out, I.gb[b], q, N);
  comps(d.q_in, I.qb[a], 5, N);
  comps(d.q_out, I.qb[b], 5, N);
  d.psi_in = (const T*)I.pb[a];
  d.psi_out = (T*)I.pb[b];
  comps(d.u_in, I.ub[a], 3, N);
  comps(d.u_out, I.ub[b], 3, N);
  comps(d.S, I.S, 6, 2 * I.SN);
  comps(d.H, I.H, 5, N);
  comps(d.rq, I.rq, 6, N);
  comps(d.qp, I.qp, 6, N);
  comps(d.Hp, I.sig, 6, N);
  d.trig = (const T*)I.trig;
  d.mass0 = shifted ? (double)(T)I.p.rho0 * (double)N : 0.0;
  d.c = coefs<T>(I.p);
  return d;
}

// SplitMix64 (Steele, Lea & Flood 2014): output number k of the stream started at seed.
inline uint64_t splitmix64(uint64_t seed, uint64_t k) {
  uint64_t z = seed + k * 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

inline double unit_noise(uint64_t seed, int inst, long long site, int comp) {
  const uint64_t k = 1ULL + ((uint64_t)inst << 40) + 5ULL * (uint64_t)site + (uint64_t)comp;
  return 2.0 * ((double)(splitmix64(seed, k) >> 11) * (1.0 / 9007199254740992.0)) - 1.0;
}

// Seeded initial droplet in FP64 on the host: psi = tanh((R - r)/2); a cholesteric
// helix about z of order S0 plus noise inside r < R; Q = 0 outside.
void init_host(const lbcad_grid& g, const lbcad_params& p, uint64_t seed, int inst, std::vector<double>& q5,
               std::vector<double>& psi) {
  const long long N = (long long)g.nx * g.ny * g.nz;
  q5.assign(5 * N, 0.0);
  psi.assign(N, 0.0);
  for (int z = 0; z < g.nz; ++z)
    for (int y = 0; y < g.ny; ++y)
      for (int x = 0; x < g.nx; ++x) {
        const long long s = x + (long long)g.nx * (y + (long long)g.ny * z);
        const double dx = x - p.centre[0], dy = y - p.centre[1], dz = z - p.centre[2];
        const double r = std::sqrt(dx * dx + dy * dy + dz * dz);
        psi[s] = std::tanh((p.R - r) / 2.0);
        if (r < p.R) {
          const double n0 = std::cos(p.q0 * dz), n1 = std::sin(p.q0 * dz);
          double Q[5] = {p.S0 * (n0 * n0 - 1.0 / 3.0), p.S0 * (n0 * n1), 0.0, p.S0 * (n1 * n1 - 1.0 / 3.0), 0.0};
          for (int k = 0; k < 5; ++k) q5[k * N + s] = Q[k] + p.noise * unit_noise(seed, inst, s, k);
        }
      }
}

// v into p[0 .. n) (the rest populations of the initial state, on the device).
template <typename T>
__global__ void k_fill(T* __restrict__ p, long long n, T v) {
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x)
    p[k] = v;
}

template <typename T>
int upload_init(lbcad_ctx* c, Inst& I, uint64_t seed, int idx) {
  std::vector<double> q5, psi;
  init_host(I.g, I.p, seed, idx, q5, psi);
  const long long N = I.N;
  std::vector<T> tq(5 * N), tp(N);
  for (long long k = 0; k < 5 * N; ++k) tq[k] = (T)q5[k];
  for (long long k = 0; k < N; ++k) tp[k] = (T)psi[k];
  // populations at rest: w_i rho0, which the shifted FP32 storage holds as 0
  const bool shifted = (c->prec == LBCAD_FP32);
  const int q = c->q();
  T* g0 = (T*)I.gb[0];
  if (shifted) {
    CK(c, cudaMemsetAsync(g0, 0, q * N * sizeof(T), c->stream));
  } else {
    for (int i = 0; i < q; ++i) {
      const double w = (q == 15) ? lat15_w(i) : lat_w(i);
      k_fill<T><<<1024, 256, 0, c->stream>>>(g0 + i * N, N, (T)(w * I.p.rho0));
      CK(c, cudaGetLastError());
    }
  }
  CK(c, cudaMemcpyAsync(I.qb[0], tq.data(), 5 * N * sizeof(T), cudaMemcpyHostToDevice, c->stream));
  CK(c, cudaMemcpyAsync(I.pb[0], tp.data(), N * sizeof(T), cudaMemcpyHostToDevice, c->stream));
  CK(c, cudaMemsetAsync(I.ub[0], 0, 3 * N * sizeof(T), c->stream));
  CK(c, cudaStreamSynchronize(c->stream));
  return LBCAD_OK;
}

int upload_descs(lbcad_ctx* c);
std::vector<lbcad_grid> boxes_of(const lbcad_ctx* c);
bool place_scratch(lbcad_ctx* c);
void drop_scratch(lbcad_ctx* c);
int prepare_fused(lbcad_ctx* c, int cfg_index);
int ensure_scratch(lbcad_ctx* c);
int default_shape(const lbcad_ctx* c);

int create_impl(int n, const lbcad_grid* grids, const lbcad_params* params, uint64_t seed, lbcad_ctx** out) {
  g_create_err.clear();
  if (!out) return fail(nullptr, LBCAD_E_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (n < 1 || !grids || !params) return fail(nullptr, LBCAD_E_INVALID_ARG, "need n >= 1 grids and params");
  for (int i = 0; i < n; ++i) {
    std::string v = validate(grids[i], params[i]);
    if (!v.empty()) return fail(nullptr, LBCAD_E_INVALID_ARG, "instance " + std::to_string(i) + ": " + v);
    if (params[i].precision != params[0].precision)
      return fail(nullptr, LBCAD_E_INVALID_ARG, "all instances must share one precision");
    if (params[i].integrator != params[0].integrator || params[i].coupling != params[0].coupling)
      return fail(nullptr, LBCAD_E_INVALID_ARG, "all instances must share one integrator and one coupling");
    if (params[i].lattice != params[0].lattice || params[i].lb_form != params[0].lb_form ||
        params[i].stencil != params[0].stencil)
      return fail(nullptr, LBCAD_E_INVALID_ARG, "all instances must share one lattice, lb_form and stencil");
  }
  lbcad_ctx* c = new (std::nothrow) lbcad_ctx();
  if (!c) return fail(nullptr, LBCAD_E_OOM, "host allocation failed");
  std::unique_ptr<lbcad_ctx, void (*)(lbcad_ctx*)> own(c, lbcad_destroy);
  const lbcad_params& p0 = params[0];
  c->prec = p0.precision;
  c->integrator = p0.integrator;
  c->coupling = p0.coupling;
  c->vel = p0.lattice;
  c->lb_form = p0.lb_form;
  c->stencil = p0.stencil;
  c->alloc = p0.alloc;
  c->free = p0.free;
  c->user = p0.alloc_user;
  if ((c->alloc == nullptr) != (c->free == nullptr))
    return fail(nullptr, LBCAD_E_INVALID_ARG, "alloc and free callbacks must be given together");
  if (p0.device >= 0) c->device = p0.device;
  else if (cudaGetDevice(&c->device) != cudaSuccess) return fail(nullptr, LBCAD_E_CUDA, "no CUDA device");
  DeviceGuard dg(c->device);
  int code = LBCAD_OK;
  auto bail = [&](int cd, const std::string& m) {
    g_create_err = m.empty() ? c->err : m;
    return cd;
  };
  if (p0.stream) {
    c->stream = (cudaStream_t)p0.stream;
  } else {
    if (cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking) != cudaSuccess)
      return bail(LBCAD_E_CUDA, "cudaStreamCreateWithFlags failed");
    c->own_stream = true;
  }
  const size_t es = c->elem();
  long long blk = 0;
  long long maxN = 0;
  c->inst.resize(n);
  for (int i = 0; i < n; ++i) {
    Inst& I = c->inst[i];
    I.g = grids[i];
    I.p = params[i];
    I.N = (long long)I.g.nx * I.g.ny * I.g.nz;
    maxN = I.N > maxN ? I.N : maxN;
    I.blk0 = blk;
    I.nblk = (I.N + kStepBlock - 1) / kStepBlock;
    blk += I.nblk;
    for (int par = 0; par < 2; ++par) {
      I.gb[par] = dev_alloc(c, (size_t)c->q() * I.N * es);
      I.qb[par] = dev_alloc(c, 5 * I.N * es);
      I.pb[par] = dev_alloc(c, I.N * es);
      I.ub[par] = dev_alloc(c, 3 * I.N * es);
      if (!I.gb[par] || !I.qb[par] || !I.pb[par] || !I.ub[par]) return bail(LBCAD_E_OOM, "device allocation failed");
    }
    const int L = I.g.nx + I.g.ny + I.g.nz;
    I.trig = dev_alloc(c, 2 * (size_t)L * es);
    if (!I.trig) return bail(LBCAD_E_OOM, "device allocation failed");
    std::vector<double> tr(2 * (size_t)L);
    const int len[3] = {I.g.nx, I.g.ny, I.g.nz};
    for (int a = 0, k = 0; a < 3; ++a)
      for (int x = 0; x < len[a]; ++x, ++k) {
        const double ph = 2.0 * M_PI * (double)x / (double)len[a];
        tr[2 * k] = std::cos(ph);
        tr[2 * k + 1] = std::sin(ph);
      }
    cudaError_t te;
    std::vector<float> tf(tr.begin(), tr.end());
    if (c->prec == LBCAD_FP64)
      te = cudaMemcpyAsync(I.trig, tr.data(), tr.size() * sizeof(double), cudaMemcpyHostToDevice, c->stream);
    else
      te = cudaMemcpyAsync(I.trig, tf.data(), tf.size() * sizeof(float), cudaMemcpyHostToDevice, c->stream);
    if (te == cudaSuccess) te = cudaStreamSynchronize(c->stream);
    if (te != cudaSuccess) return bail(LBCAD_E_CUDA, std::string("trig table upload: ") + cudaGetErrorString(te));
  }
  c->obs_cnt = (unsigned*)dev_alloc(c, n * sizeof(unsigned));
  c->obs_latest = (double*)dev_alloc(c, (size_t)n * 12 * sizeof(double));
  if (!c->obs_cnt || !c->obs_latest) return bail(LBCAD_E_OOM, "device allocation failed");
  if (cudaMemsetAsync(c->obs_cnt, 0, n * sizeof(unsigned), c->stream) != cudaSuccess ||
      cudaStreamSynchronize(c->stream) != cudaSuccess)
    return bail(LBCAD_E_CUDA, "a6 counter initialisation failed");
  c->total_blocks = blk;
  if (blk >= (1LL << 31)) return bail(LBCAD_E_INVALID_ARG, "too many blocks for one launch");
  const size_t dsz = (c->prec == LBCAD_FP64 ? sizeof(InstDesc<double>) : sizeof(InstDesc<float>)) * n;
  for (int par = 0; par < 2; ++par) {
    c->desc[par] = dev_alloc(c, dsz);
    if (!c->desc[par]) return bail(LBCAD_E_OOM, "device allocation failed");
  }
  c->obs_partial = (double*)dev_alloc(c, kObsMaxBlocks * 12 * sizeof(double));
  c->obs_out = (double*)dev_alloc(c, 12 * sizeof(double));
  if (!c->obs_partial || !c->obs_out) return bail(LBCAD_E_OOM, "device allocation failed");
  // last, the scratch of the Euler step and the work lists; near the end of the memory a smaller scratch, for more
  // launches
  const bool scratch = !c->staged_only() && !c->sync_split();
  long long before = 0;  // the scratch that did not fit
  for (;; c->rule = c->rule.tighter()) {
    c->plan = plan_step(boxes_of(c), !scratch, c->rule);
    if (before == 0 || c->plan.scratch < before) {
      code = LBCAD_E_OOM;
      if (!scratch || place_scratch(c)) {
        if (upload_descs(c) != LBCAD_OK) return bail(LBCAD_E_CUDA, "");
        code = prepare_fused(c, default_shape(c));
      }
      if (code == LBCAD_OK) break;
      if (code != LBCAD_E_OOM || !scratch) return bail(code, "");
      drop_scratch(c);
      before = c->plan.scratch;
    }
    if (c->rule.tightest()) return bail(LBCAD_E_OOM, "device allocation failed");
  }
  if (c->staged_only() || c->sync_split()) {
    if ((code = ensure_scratch(c)) != LBCAD_OK) return bail(code, "");
  }
  if (c->staged_only()) c->path = LBCAD_PATH_STAGED;
  for (int i = 0; i < n; ++i) {
    code = (c->prec == LBCAD_FP64) ? upload_init<double>(c, c->inst[i], seed, i)
                                   : upload_init<float>(c, c->inst[i], seed, i);
    if (code != LBCAD_OK) return bail(code, "");
  }
  *out = own.release();
  return LBCAD_OK;
}

// The descriptors of the default path, which stay on the host.  (After the first time their vectors have the room.)
void march_descs(lbcad_ctx* c) {
  for (int par = 0; par < 2; ++par) {
    c->desc32[par].clear();
    c->desc64[par].clear();
    for (const Inst& I : c->inst) {
      if (c->prec == LBCAD_FP64) c->desc64[par].push_back(make_march_desc<double>(I, par, false));
      else c->desc32[par].push_back(make_march_desc<float>(I, par, true));
    }
  }
}

int upload_descs(lbcad_ctx* c) {
  const int n = (int)c->inst.size();
  march_descs(c);
  for (int par = 0; par < 2; ++par) {
    if (c->prec == LBCAD_FP64) {
      std::vector<InstDesc<double>> h(n);
      for (int i = 0; i < n; ++i) h[i] = make_desc<double>(c->inst[i], par);
      CK(c, cudaMemcpyAsync(c->desc[par], h.data(), n * sizeof(h[0]), cudaMemcpyHostToDevice, c->stream));
      CK(c, cudaStreamSynchronize(c->stream));
    } else {
      std::vector<InstDesc<float>> h(n);
      for (int i = 0; i < n; ++i) h[i] = make_desc<float>(c->inst[i], par);
      CK(c, cudaMemcpyAsync(c->desc[par], h.data(), n * sizeof(h[0]), cudaMemcpyHostToDevice, c->stream));
      CK(c, cudaStreamSynchronize(c->stream));
    }
  }
  return LBCAD_OK;
}

std::vector<lbcad_grid> boxes_of(const lbcad_ctx* c) {
  std::vector<lbcad_grid> b;
  for (const Inst& I : c->inst) b.push_back(I.g);
  return b;
}

// Allocates the scratch of the plan and gives every instance its place in it; false: no memory.
bool place_scratch(lbcad_ctx* c) {
  c->scratch = (char*)dev_alloc(c, 12 * (size_t)c->plan.scratch * c->elem());
  if (!c->scratch) return false;
  for (size_t i = 0; i < c->inst.size(); ++i) {
    c->inst[i].SN = c->plan.place[i].sites;
    c->inst[i].S = c->scratch + 12 * (size_t)c->plan.place[i].at * c->elem();
  }
  return true;
}

void drop_scratch(lbcad_ctx* c) {
  if (c->scratch) dev_free(c, c->scratch);
  c->scratch = nullptr;
}

// Before a step of the default path.  The scratch is missing only where another owner of the memory took its place
// while shrink_scratch had given it back.
int ensure_step_scratch(lbcad_ctx* c) {
  if (c->scratch || c->staged_only() || c->sync_split()) return LBCAD_OK;
  if (!place_scratch(c)) return fail(c, LBCAD_E_OOM, "scratch allocation failed");
  march_descs(c);
  return LBCAD_OK;
}

// A smaller scratch for the step, in more launches, where another call needs its memory: it holds something only while
// a step runs.  False: it is as small as it gets, or there is no memory for the lists of more launches.
bool shrink_scratch(lbcad_ctx* c) {
  if (!c->scratch || cudaStreamSynchronize(c->stream) != cudaSuccess) return false;
  const std::vector<lbcad_grid> boxes = boxes_of(c);
  ScratchRule rule = c->rule;
  StepPlan plan;
  do {
    if (rule.tightest()) return false;
    rule = rule.tighter();
    plan = plan_step(boxes, false, rule);
  } while (plan.scratch >= c->plan.scratch);
  drop_scratch(c);
  std::swap(c->plan, plan);
  const bool smaller = prepare_fused(c, c->cfg_index) == LBCAD_OK;
  if (smaller) c->rule = rule;
  else std::swap(c->plan, plan);  // that of the lists still in use
  return ensure_step_scratch(c) == LBCAD_OK && smaller;
}

// dev_alloc for a call after lbcad_create, which may take memory from the step's scratch.
void* dev_alloc_or_shrink(lbcad_ctx* c, size_t bytes) {
  void* p = dev_alloc(c, bytes);
  while (!p && shrink_scratch(c)) p = dev_alloc(c, bytes);
  return p;
}

// Scratch (sigma, mu, H per site) of the two-kernel and staged paths, allocated on first
// use; Heun contexts also hold the right-hand side at t and the predicted state.
int ensure_scratch(lbcad_ctx* c) {
  if (c->scratch_ready) return LBCAD_OK;
  const size_t es = c->elem();
  for (Inst& I : c->inst) {
    if (!I.sig) I.sig = dev_alloc_or_shrink(c, 10 * I.N * es);  // (an earlier call may have found room for some)
    if (!I.H) I.H = dev_alloc_or_shrink(c, 5 * I.N * es);
    if (!I.sig || !I.H) return fail(c, LBCAD_E_OOM, "scratch allocation failed");
    I.mu = (char*)I.sig + 9 * I.N * es;
    if (c->sync_split()) {
      // the default path's stress and mu; Heun's H and mu at the predicted state follow in the same place once
      // the predictor has read them
      I.S = I.sig;
      I.SN = I.N;
    }
    if (c->integrator == LBCAD_HEUN) {
      I.rq = dev_alloc(c, 6 * I.N * es);
      I.qp = dev_alloc(c, 6 * I.N * es);
      if (!I.rq || !I.qp) return fail(c, LBCAD_E_OOM, "scratch allocation failed");
    }
  }
  const int r = upload_descs(c);
  c->scratch_ready = r == LBCAD_OK;
  return r;
}

// Tile shape of a new context: candidate 0 (rows of 32 sites) or 3 (rows of 16), whichever covers the boxes
// with fewer sites beyond their edges; 0, with its longer rows, when they tie.
int default_shape(const lbcad_ctx* c) {
  if (c->prec == LBCAD_FP64) return 0;
  long long wide = 0, square = 0;
  for (const Inst& I : c->inst) {
    wide += (long long)((I.g.nx + 31) / 32 * 32) * ((I.g.ny + 7) / 8 * 8) * I.g.nz;
    square += (long long)((I.g.nx + 15) / 16 * 16) * ((I.g.ny + 15) / 16 * 16) * I.g.nz;
  }
  return square < wide ? 3 : 0;
}

// Largest step (sites) whose kernels are launched with programmatic dependent launch.
constexpr long long kEarlySites = 1 << 20;

// The items of a group of instances for tx x ty tiles and at most `blocks` resident blocks, appended to `out`.
// Each box is cut into slabs of about `len` planes; blocks take items in turn, so the slowest block works
// through ceil(items / blocks) of them, each its planes plus what an item costs besides (two more planes
// to load and to carry, and a start without overlap: about one plane's time).  The length is the one with the
// shortest such time, up to 32 planes: neighbouring columns then stay close enough in z to find their halos
// in L2.  za, zn: of a single box only the planes za ... za + zn - 1, modulo its height (zn 0: all of each box).
MarchWork add_items(const lbcad_ctx* c, const StepWork& g, int tx, int ty, int blocks, std::vector<MarchItem>& out,
                    int za = 0, int zn = 0) {
  constexpr double kItemPlanes = 1.0;
  auto columns = [&](const lbcad_grid& b) { return (long long)((b.nx + tx - 1) / tx) * ((b.ny + ty - 1) / ty); };
  int tallest = 0;
  auto height = [&](const lbcad_grid& b) { return zn > 0 ? zn : b.nz; };
  for (int i = 0; i < g.ninst; ++i) tallest = std::max(tallest, height(c->inst[g.first + i].g));
  auto slabs_of = [&](const lbcad_grid& b, int n) {  // slabs of box b when the tallest box has n
    return std::max(1, (int)(((long long)height(b) * n + tallest - 1) / tallest));
  };
  int best = 1;
  double best_time = -1.0;
  for (int n = (tallest + 31) / 32; n <= tallest; ++n) {
    long long items = 0;
    for (int i = 0; i < g.ninst; ++i) items += columns(c->inst[g.first + i].g) * slabs_of(c->inst[g.first + i].g, n);
    const double t = (double)((items + blocks - 1) / blocks) * ((tallest + n - 1) / n + kItemPlanes);
    if (best_time < 0.0 || t < best_time) {
      best = n;
      best_time = t;
    }
  }
  MarchWork w;
  const size_t first = out.size();
  long long sites = 0;
  for (int i = 0; i < g.ninst; ++i) {
    const lbcad_grid& b = c->inst[g.first + i].g;
    sites += c->inst[g.first + i].N;
    const int slabs = slabs_of(b, best);
    for (int k = 0; k < slabs; ++k) {
      const int end = za + (int)((long long)height(b) * (k + 1) / slabs);
      for (int zb = za + (int)((long long)height(b) * k / slabs), ze; zb < end; zb = ze) {
        const int turn = (zb + b.nz) / b.nz - 1, base = turn * b.nz;  // zb >= -nz; an item ends at the box's edge
        ze = std::min(end, base + b.nz);
        for (int y0 = 0; y0 < b.ny; y0 += ty)
          for (int x0 = 0; x0 < b.nx; x0 += tx) out.push_back(MarchItem{i, x0, y0, zb - base, ze - base});
      }
    }
  }
  w.items = (const MarchItem*)(first * sizeof(MarchItem));  // offset; the list's address is added when it is uploaded
  w.nitems = (int)(out.size() - first);
  w.grid = w.nitems < blocks ? w.nitems : blocks;
  // Dependent launch hides a kernel's start-up (FP32 Euler, us a step with it and without: 16^3 11.7 and 16.4, 32^3 16.3
  // and 19.5, 64^3 34.1 and 39.0, 96^3 86.0 and 90.4, 112^3 139.4 and 142.2, 128^3 189.7 and 193.7), but blocks that
  // start early disturb the even spread of a large step's blocks (160^3 348.4 and 349.0, 192^3 618 and 605, 256^3 1404 and
  // 1362).  The line lies on the safe side of where the two meet, about 2^22 sites.
  w.early = sites <= kEarlySites;
  return w;
}

void drop_graph(lbcad_ctx* c) {
  if (c->gexec) { cudaGraphExecDestroy(c->gexec); c->gexec = nullptr; }
  if (c->graph) { cudaGraphDestroy(c->graph); c->graph = nullptr; }
}

// Work items of the default path for tile shape `cfg_index`, and the slots of its a6 sums.  Where there is no memory
// for them, on the host or the device, everything stays as it was.
int prepare_fused(lbcad_ctx* c, int cfg_index) try {
  FusedCfg cfg;
  const int v = c->fused_variant();
  const bool split = c->sync_split(), heun = c->integrator == LBCAD_HEUN, many = c->inst.size() > 1;
  cudaError_t e = (c->prec == LBCAD_FP64) ? LaunchFused<double, false>::prepare(v, cfg_index, many, split, heun, &cfg)
                                          : LaunchFused<float, true>::prepare(v, cfg_index, many, split, heun, &cfg);
  if (e == cudaErrorNotSupported)
    return fail(c, LBCAD_E_UNSUPPORTED, "this velocity set and LB form do not come in that tile shape");
  if (e != cudaSuccess) return fail(c, LBCAD_E_CUDA, std::string("fused kernel set-up: ") + cudaGetErrorString(e));
  if (cfg.fields_per_sm < 1 || cfg.lb_per_sm < 1)
    return fail(c, LBCAD_E_UNSUPPORTED, "fused tile shape does not fit on an SM");
  int sms = 0;
  CK(c, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device));
  auto blocks = [&](int per_sm) { return sms * (per_sm > 0 ? per_sm : 1); };
  std::vector<MarchItem> t;
  std::vector<StepWork> work;
  for (const StepPart& part : c->plan.parts) {
    StepWork w;
    w.first = part.first;
    w.ninst = part.ninst;
    w.sz0 = part.sz0;
    w.fields = add_items(c, w, cfg.fx, cfg.fy, blocks(cfg.fields_per_sm), t, part.fz, part.fn);
    w.lb = add_items(c, w, cfg.lx, cfg.ly, blocks(cfg.lb_per_sm), t, part.lz, part.ln);
    work.push_back(w);
  }
  for (StepWork& g : work) {
    if (split) {
      g.op[0] = add_items(c, g, cfg.lx, cfg.ly, blocks(cfg.op_per_sm[0]), t);
      if (heun) {
        g.pred = add_items(c, g, cfg.fx, cfg.fy, blocks(cfg.pred_per_sm), t);
        g.op[1] = add_items(c, g, cfg.lx, cfg.ly, blocks(cfg.op_per_sm[1]), t);
      }
    }
  }
  // the runs of each block, as k_march_lb forms them: slot (block, run) -> instance, and each instance's slot
  // count and range
  std::vector<int> map;
  std::vector<FusedObs> obs;
  size_t nslots = 0;
  for (const StepWork& g : work) {
    const MarchItem* items = t.data() + (size_t)g.lb.items / sizeof(MarchItem);
    const int grid = g.lb.grid;
    std::vector<std::vector<int>> runs(grid);
    size_t maxrun = 1;
    for (int b = 0; b < grid; ++b) {
      for (int i = b; i < g.lb.nitems; i += grid)
        if (runs[b].empty() || runs[b].back() != items[i].inst) runs[b].push_back(items[i].inst);
      maxrun = std::max(maxrun, runs[b].size());
    }
    const size_t at = map.size(), n = (size_t)grid * maxrun;
    map.resize(at + n + 3 * (size_t)g.ninst, -1);
    int* nslot = map.data() + at + n;
    int* slot_lo = nslot + g.ninst;
    int* slot_hi = slot_lo + g.ninst;
    for (int i = 0; i < g.ninst; ++i) nslot[i] = 0;
    for (int b = 0; b < grid; ++b)
      for (size_t j = 0; j < runs[b].size(); ++j) {
        const int sl = (int)(b * maxrun + j), i = runs[b][j];
        map[at + sl] = i;
        if (nslot[i]++ == 0) slot_lo[i] = sl;
        slot_hi[i] = sl + 1;
      }
    FusedObs ob{};
    ob.slots = (double*)(nslots * 12 * sizeof(double));  // offsets; the arrays' addresses are added below
    ob.slot_inst = (const int*)(at * sizeof(int));
    ob.nslot = (const int*)((at + n) * sizeof(int));
    ob.maxrun = (int)maxrun;
    // slabs of one instance: their slots follow one another
    if (g.ninst == 1 && !obs.empty() && work[obs.size() - 1].first == g.first) {
      ob.slots = obs.back().slots;
      ob.slot0 = obs.back().slot0 + work[obs.size() - 1].lb.grid;
    }
    obs.push_back(ob);
    if (g.ninst == 1)
      for (size_t k = obs.size(); k > 0 && work[k - 1].first == g.first; --k) obs[k - 1].total = ob.slot0 + grid;
    nslots += n;
  }
  // the launches in use keep their lists until all of the new ones have a place
  if (!grow(c, c->items, c->items_cap, t.size() * sizeof(MarchItem)) ||
      !grow(c, c->obs_slots, c->obs_slots_cap, nslots * 12 * sizeof(double)) ||
      !grow(c, c->obs_map, c->obs_map_cap, map.size() * sizeof(int)))
    return fail(c, LBCAD_E_OOM, "work list allocation failed");
  auto place = [](auto*& p, void* base) { p = (std::remove_reference_t<decltype(p)>)((char*)base + (size_t)p); };
  for (size_t i = 0; i < work.size(); ++i) {
    StepWork& g = work[i];
    for (MarchWork* w : {&g.fields, &g.lb, &g.op[0], &g.pred, &g.op[1]}) place(w->items, c->items);
    FusedObs& ob = obs[i];
    place(ob.slots, c->obs_slots);
    place(ob.slot_inst, c->obs_map);
    place(ob.nslot, c->obs_map);
    ob.slot_lo = ob.nslot + g.ninst;
    ob.slot_hi = ob.slot_lo + g.ninst;
    ob.cnt = c->obs_cnt + g.first;
    ob.latest = c->obs_latest + 12 * (size_t)g.first;
  }
  drop_graph(c);  // a captured step reads the lists that change here
  CK(c, cudaMemcpyAsync(c->items, t.data(), t.size() * sizeof(MarchItem), cudaMemcpyHostToDevice, c->stream));
  CK(c, cudaMemcpyAsync(c->obs_map, map.data(), map.size() * sizeof(int), cudaMemcpyHostToDevice, c->stream));
  // the kernels leave the per-instance counters at zero; reset them here as well, so that a
  // launch that failed part-way cannot shift the next sums
  CK(c, cudaMemsetAsync(c->obs_cnt, 0, c->inst.size() * sizeof(unsigned), c->stream));
  CK(c, cudaStreamSynchronize(c->stream));
  c->work = std::move(work);
  c->obs = std::move(obs);
  c->obs_valid = false;
  c->cfg_index = cfg_index;
  return LBCAD_OK;
} catch (const std::exception&) {
  return caught(c);
}

cudaError_t launch_fused(lbcad_ctx* c, int par) {
  const int v = c->fused_variant();
  const bool split = c->sync_split(), heun = c->integrator == LBCAD_HEUN, sync = c->coupling == LBCAD_SYNC;
  auto run = [&](auto launch, const auto& d) {
    using L = decltype(launch);
    cudaError_t e = cudaSuccess;
    for (size_t i = 0; i < c->work.size() && e == cudaSuccess; ++i) {
      const StepWork& g = c->work[i];
      e = split ? L::split_step(v, c->cfg_index, g, heun, sync, d.data() + g.first, c->stream)
                : L::step(v, c->cfg_index, g, d.data() + g.first, c->obs[i], c->observe, c->stream);
    }
    return e;
  };
  return c->prec == LBCAD_FP64 ? run(LaunchFused<double, false>{}, c->desc64[par])
                               : run(LaunchFused<float, true>{}, c->desc32[par]);
}

int launch_steps(lbcad_ctx* c, int64_t n) {
  for (int64_t k = 0; k < n; ++k) {
    const int par = (int)(c->step & 1);
    cudaError_t e;
    const bool heun = c->integrator == LBCAD_HEUN, sync = c->coupling == LBCAD_SYNC;
    if (c->path == LBCAD_PATH_FUSED) {
      e = launch_fused(c, par);
    } else if (c->path == LBCAD_PATH_STAGED) {
      e = (c->prec == LBCAD_FP64)
              ? Launch<double, false>::staged((const InstDesc<double>*)c->desc[par], (int)c->inst.size(),
                                              c->total_blocks, kStepBlock, heun, sync, c->vel, c->lb_form,
                                              c->stencil, c->stream)
              : Launch<float, true>::staged((const InstDesc<float>*)c->desc[par], (int)c->inst.size(),
                                            c->total_blocks, kStepBlock, heun, sync, c->vel, c->lb_form,
                                            c->stencil, c->stream);
    } else if (c->prec == LBCAD_FP64)
      e = Launch<double, false>::step((const InstDesc<double>*)c->desc[par], (int)c->inst.size(), c->total_blocks,
                                      kStepBlock, c->stream);
    else
      e = Launch<float, true>::step((const InstDesc<float>*)c->desc[par], (int)c->inst.size(), c->total_blocks,
                                    kStepBlock, c->stream);
    if (e != cudaSuccess) return fail(c, LBCAD_E_CUDA, std::string("step launch: ") + cudaGetErrorString(e));
    c->step++;
  }
  return LBCAD_OK;
}

template <typename T>
InstDesc<T> desc_now(const lbcad_ctx* c, int inst) {
  return make_desc<T>(c->inst[inst], (int)(c->step & 1));
}

int ensure_staging(lbcad_ctx* c, size_t bytes) {
  if (c->staging_bytes >= bytes) return LBCAD_OK;
  // the old buffer stays in the pool until destroy; staging only grows
  void* p = dev_alloc_or_shrink(c, bytes);
  if (!p) return fail(c, LBCAD_E_OOM, "staging allocation failed");
  c->staging = (double*)p;
  c->staging_bytes = bytes;
  return LBCAD_OK;
}

int ncomp_of(uint32_t mask, int q = 19) {
  return ((mask & LBCAD_FIELD_G) ? q : 0) + ((mask & LBCAD_FIELD_RHO) ? 1 : 0) + ((mask & LBCAD_FIELD_U) ? 3 : 0) +
         ((mask & LBCAD_FIELD_Q) ? 5 : 0) + ((mask & LBCAD_FIELD_PSI) ? 1 : 0);
}

}  // namespace

extern "C" {

int lbcad_lattice(int32_t* c57, double* w19) {
  if (!c57 || !w19) return LBCAD_E_INVALID_ARG;
  for (int i = 0; i < 19; ++i) {
    for (int a = 0; a < 3; ++a) c57[3 * i + a] = lat_c(i, a);
    w19[i] = lat_w(i);
  }
  return LBCAD_OK;
}

int lbcad_velocity_set(int32_t lattice, int32_t* c, double* w) {
  if (!c || !w || (lattice != LBCAD_D3Q19 && lattice != LBCAD_D3Q15)) return LBCAD_E_INVALID_ARG;
  const int q = (lattice == LBCAD_D3Q15) ? 15 : 19;
  for (int i = 0; i < q; ++i) {
    for (int a = 0; a < 3; ++a) c[3 * i + a] = (q == 15) ? lat15_c(i, a) : lat_c(i, a);
    w[i] = (q == 15) ? lat15_w(i) : lat_w(i);
  }
  return q;
}

int lbcad_create(const lbcad_grid* grid, const lbcad_params* params, uint64_t seed, lbcad_ctx** out) try {
  return create_impl(1, grid, params, seed, out);
} catch (const std::exception&) {
  return caught(nullptr);
}

int lbcad_create_batch(int32_t n, const lbcad_grid* grids, const lbcad_params* params, uint64_t seed,
                       lbcad_ctx** out) try {
  return create_impl(n, grids, params, seed, out);
} catch (const std::exception&) {
  return caught(nullptr);
}

int lbcad_set_path(lbcad_ctx* c, int32_t path) try {
  if (!c) return LBCAD_E_INVALID_ARG;
  if (path != LBCAD_PATH_FUSED && path != LBCAD_PATH_TWO_KERNEL && path != LBCAD_PATH_STAGED)
    return fail(c, LBCAD_E_INVALID_ARG, "unknown path");
  if (path != LBCAD_PATH_STAGED && c->staged_only())
    return fail(c, LBCAD_E_UNSUPPORTED, "radius-2 contexts run on the staged path only");
  if (path == LBCAD_PATH_TWO_KERNEL && (!c->default_lb() || c->sync_split()))
    return fail(c, LBCAD_E_UNSUPPORTED, "the two-kernel path covers the Euler, lagged step of D3Q19 with the body force");
  DeviceGuard dg(c->device);
  if (path != LBCAD_PATH_FUSED) {
    int r = ensure_scratch(c);
    if (r) return r;
  }
  if (path != c->path) {
    if (c->gexec) { cudaGraphExecDestroy(c->gexec); c->gexec = nullptr; }
    if (c->graph) { cudaGraphDestroy(c->graph); c->graph = nullptr; }
    c->path = path;
    c->obs_valid = false;
  }
  return LBCAD_OK;
} catch (const std::exception&) {
  return caught(c);
}

int lbcad_autotune(lbcad_ctx* c, int32_t reps, int32_t* chosen, float* ms_per_cfg, int32_t ncfg) try {
  if (!c || reps < 1) return LBCAD_E_INVALID_ARG;
  if (c->staged_only()) return fail(c, LBCAD_E_UNSUPPORTED, "tile shapes belong to the fused path (Euler, lagged)");
  if (c->sync_split()) return fail(c, LBCAD_E_UNSUPPORTED, "sync coupling and Heun run on one fixed fused tile shape");
  DeviceGuard dg(c->device);
  if (int r = ensure_step_scratch(c)) return r;
  const int n = (c->prec == LBCAD_FP64) ? LaunchFused<double, false>::num_configs()
                                        : LaunchFused<float, true>::num_configs();
  const int par = (int)(c->step & 1);
  const int before = c->cfg_index;
  cudaEvent_t e0, e1;
  CK(c, cudaEventCreate(&e0));
  CK(c, cudaEventCreate(&e1));
  // three rounds over the candidates, each candidate timed over `reps` launches after one
  // untimed launch; a candidate's time is its best round (rounds interleave the candidates,
  // so a drift of the clocks during tuning does not favour one of them)
  constexpr int kRounds = 3;
  std::vector<float> best_of(n, -1.f);
  int code = LBCAD_OK;
  for (int round = 0; round < kRounds && code == LBCAD_OK; ++round) {
    for (int k = 0; k < n && code == LBCAD_OK; ++k) {
      if (round > 0 && best_of[k] < 0.f) continue;  // does not fit
      code = prepare_fused(c, k);
      if (code == LBCAD_E_UNSUPPORTED || code == LBCAD_E_OOM) {  // no such shape, or no memory for its lists
        code = LBCAD_OK;
        continue;
      }
      if (code != LBCAD_OK) break;
      float ms = -1.f;
      cudaError_t e = launch_fused(c, par);
      if (e == cudaSuccess) e = cudaEventRecord(e0, c->stream);
      for (int r = 0; r < reps && e == cudaSuccess; ++r) e = launch_fused(c, par);
      if (e == cudaSuccess) e = cudaEventRecord(e1, c->stream);
      if (e == cudaSuccess) e = cudaEventSynchronize(e1);
      if (e == cudaSuccess && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess) ms /= reps;
      if (e != cudaSuccess) code = fail(c, LBCAD_E_CUDA, std::string("autotune: ") + cudaGetErrorString(e));
      else if (best_of[k] < 0.f || ms < best_of[k]) best_of[k] = ms;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  int best = -1;
  for (int k = 0; k < n; ++k) {
    if (best_of[k] >= 0.f && (best < 0 || best_of[k] < best_of[best])) best = k;
    if (code == LBCAD_OK && ms_per_cfg && k < ncfg) ms_per_cfg[k] = best_of[k];
  }
  if (code == LBCAD_OK && best < 0) code = fail(c, LBCAD_E_UNSUPPORTED, "no fused tile shape fits");
  if (code != LBCAD_OK) {
    const std::string why = c->err;
    prepare_fused(c, before);
    c->err = why;
    return code;
  }
  int r = prepare_fused(c, best);
  if (r) return r;
  if (chosen) *chosen = best;
  return LBCAD_OK;
} catch (const std::exception&) {
  return caught(c);
}

int lbcad_set_tiles(lbcad_ctx* c, int32_t cfg) try {
  if (!c) return LBCAD_E_INVALID_ARG;
  if (c->staged_only()) return fail(c, LBCAD_E_UNSUPPORTED, "tile shapes belong to the fused path (Euler, lagged)");
  if (c->sync_split()) return fail(c, LBCAD_E_UNSUPPORTED, "sync coupling and Heun run on one fixed fused tile shape");
  DeviceGuard dg(c->device);
  const int n = (c->prec == LBCAD_FP64) ? LaunchFused<double, false>::num_configs()
                                        : LaunchFused<float, true>::num_configs();
  if (cfg < 0 || cfg >= n) return fail(c, LBCAD_E_INVALID_ARG, "tile shape index out of range");
  return prepare_fused(c, cfg);
} catch (const std::exception&) {
  return caught(c);
}

int lbcad_set_observe(lbcad_ctx* c, int32_t on) try {
  if (!c || (on != 0 && on != 1)) return LBCAD_E_INVALID_ARG;
  if (c->observe != (on == 1)) {
    c->observe = on == 1;
    drop_graph(c);
    c->obs_valid = false;
  }
  return LBCAD_OK;
} catch (const std::exception&) {
  return caught(c);
}

int lbcad_set_graph(lbcad_ctx* c, int32_t steps_per_graph) try {
  if (!c) return LBCAD_E_INVALID_ARG;
  // a replay must leave the ping-pong parity unchanged, so a graph holds an even number of steps
  if (steps_per_graph < 0 || (steps_per_graph & 1))
    return fail(c, LBCAD_E_INVALID_ARG, "steps_per_graph must be 0 or a positive even number");
  DeviceGuard dg(c->device);
  if (c->gexec) { cudaGraphExecDestroy(c->gexec); c->gexec = nullptr; }
  if (c->graph) { cudaGraphDestroy(c->graph); c->graph = nullptr; }
  c->graph_steps = steps_per_graph;
  return LBCAD_OK;
} catch (const std::exception&) {
  return caught(c);
}

int lbcad_step(lbcad_ctx* c, int64_t n) try {
  if (!c || n < 0) return LBCAD_E_INVALID_ARG;
  DeviceGuard dg(c->device);
  if (c->path == LBCAD_PATH_FUSED)
    if (int r = ensure_step_scratch(c)) return r;
  int64_t left = n;
  if (c->graph_steps > 0) {
    if ((c->step & 1) && left > 0) {
      int r = launch_steps(c, 1);
      if (r) return r;
      left--;
    }
    while (left >= c->graph_steps) {
      if (!c->gexec) {
        const int64_t step0 = c->step;
        CK(c, cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal));
        int r = launch_steps(c, c->graph_steps);
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamEndCapture(c->stream, &g);
        c->step = step0;
        if (r) { if (g) cudaGraphDestroy(g); return r; }
        if (e != cudaSuccess) return fail(c, LBCAD_E_CUDA, std::string("graph capture: ") + cudaGetErrorString(e));
        c->graph = g;
        CK(c, cudaGraphInstantiate(&c->gexec, c->graph, 0));
      }
      CK(c, cudaGraphLaunch(c->gexec, c->stream));
      c->step += c->graph_steps;
      left -= c->graph_steps;
    }
  }
  int r = launch_steps(c, left);
  // after a fused step the a6 sums of the new state are in obs_latest
  if (r == LBCAD_OK && n > 0) c->obs_valid = c->path == LBCAD_PATH_FUSED && c->observe && !c->sync_split();
  return r;
} catch (const std::exception&) {
  return caught(c);
}

int lbcad_get_fields(lbcad_ctx* c, int32_t inst, uint32_t mask, void* dst, size_t bytes, int32_t dst_is_device) try {
  if (!c) return LBCAD_E_INVALID_ARG;
  if (inst < 0 || inst >= (int)c->inst.size()) return fail(c, LBCAD_E_INVALID_ARG, "instance out of range");
  if (!dst || mask == 0 || (mask & ~31u)) return fail(c, LBCAD_E_INVALID_ARG, "bad dst or mask");
  const long long N = c->inst[inst].N;
  const size_t need = (size_t)ncomp_of(mask, c->q()) * N * sizeof(double);
  if (bytes < need) return fail(c, LBCAD_E_INVALID_ARG, "dst too small");
  DeviceGuard dg(c->device);
  double* target = (double*)dst;
  if (!dst_is_device) {
    int r = ensure_staging(c, need);
    if (r) return r;
    target = c->staging;
  }
  cudaError_t e = (c->prec == LBCAD_FP64)
                      ? Launch<double, false>::get_fields(desc_now<double>(c, inst), mask, target, c->stream)
                      : Launch<float, true>::get_fields(desc_now<float>(c, inst), mask, target, c->stream);
  if (e != cudaSuccess) return fail(c, LBCAD_E_CUDA, std::string("get_fields: ") + cudaGetErrorString(e));
  if (!dst_is_device) CK(c, cudaMemcpyAsync(dst, target, need, cudaMemcpyDeviceToHost, c->stream));
  CK(c, cudaStreamSynchronize(c->stream));
  return LBCAD_OK;
} catch (const std::exception&) {
  return caught(c);
}

int lbcad_set_fields(lbcad_ctx* c, int32_t inst, uint32_t mask, const void* src, size_t bytes,
                     int32_t src_is_device) try {
  if (!c) return LBCAD_E_INVALID_ARG;
  if (inst < 0 || inst >= (int)c->inst.size()) return fail(c, LBCAD_E_INVALID_ARG, "instance out of range");
  if (!src || mask == 0 || (mask & ~31u) || (mask & LBCAD_FIELD_RHO))
    return fail(c, LBCAD_E_INVALID_ARG, "bad src or mask (RHO cannot be set)");
  const long long N = c->inst[inst].N;
  const size_t need = (size_t)ncomp_of(mask, c->q()) * N * sizeof(double);
  if (bytes < need) return fail(c, LBCAD_E_INVALID_ARG, "src too small");
  DeviceGuard dg(c->device);
  const double* from = (const double*)src;
  if (!src_is_device) {
    int r = ensure_staging(c, need);
    if (r) return r;
    CK(c, cudaMemcpyAsync(c->staging, src, need, cudaMemcpyHostToDevice, c->stream));
    from = c->staging;
  }
  Inst& I = c->inst[inst];
  const int par = (int)(c->step & 1);
  cudaError_t e;
  if (c->prec == LBCAD_FP64)
    e = Launch<double, false>::set_fields(desc_now<double>(c, inst), mask, from, (double*)I.gb[par],
                                          (double*)I.qb[par], (double*)I.pb[par], (double*)I.ub[par], c->stream);
  else
    e = Launch<float, true>::set_fields(desc_now<float>(c, inst), mask, from, (float*)I.gb[par], (float*)I.qb[par],
                                        (float*)I.pb[par], (float*)I.ub[par], c->stream);
  if (e != cudaSuccess) return fail(c, LBCAD_E_CUDA, std::string("set_fields: ") + cudaGetErrorString(e));
  c->obs_valid = false;
  CK(c, cudaStreamSynchronize(c->stream));
  return LBCAD_OK;
} catch (const std::exception&) {
  return caught(c);
}

int lbcad_state_bytes(lbcad_ctx* c, int32_t inst, size_t* bytes) try {
  if (!c || !bytes) return LBCAD_E_INVALID_ARG;
  if (inst < 0 || inst >= (int)c->inst.size()) return fail(c, LBCAD_E_INVALID_ARG, "instance out of range");
  *bytes = (size_t)(c->q() + 9) * (size_t)c->inst[inst].N * c->elem();
  return LBCAD_OK;
} catch (const std::exception&) {
  return caught(c);
}

namespace {
// Copies the current-parity state buffers of one instance to/from a contiguous buffer.
int copy_state(lbcad_ctx* c, int inst, void* ext, size_t bytes, bool ext_is_device, bool to_ext) {
  if (inst < 0 || inst >= (int)c->inst.size()) return fail(c, LBCAD_E_INVALID_ARG, "instance out of range");
  size_t need = 0;
  lbcad_state_bytes(c, inst, &need);
  if (!ext || bytes < need) return fail(c, LBCAD_E_INVALID_ARG, "state buffer missing or too small");
  DeviceGuard dg(c->device);
  Inst& I = c->inst[inst];
  const int par = (int)(c->step & 1);
  const size_t es = c->elem(), N = (size_t)I.N;
  void* parts[4] = {I.gb[par], I.qb[par], I.pb[par], I.ub[par]};
  const size_t sizes[4] = {(size_t)c->q() * N * es, 5 * N * es, N * es, 3 * N * es};
  const cudaMemcpyKind kind = to_ext ? (ext_is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost)
                                     : (ext_is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice);
  size_t off = 0;
  for (int k = 0; k < 4; ++k) {
    char* e = (char*)ext + off;
    if (to_ext) CK(c, cudaMemcpyAsync(e, parts[k], sizes[k], kind, c->stream));
    else CK(c, cudaMemcpyAsync(parts[k], e, sizes[k], kind, c->stream));
    off += sizes[k];
  }
  if (!to_ext) c->obs_valid = false;
  CK(c, cudaStreamSynchronize(c->stream));
  return LBCAD_OK;
}
}  // namespace

int lbcad_get_state(lbcad_ctx* c, int32_t inst, void* dst, size_t bytes, int32_t dst_is_device) try {
  if (!c) return LBCAD_E_INVALID_ARG;
  return copy_state(c, inst, dst, bytes, dst_is_device != 0, true);
} catch (const std::exception&) {
  return caught(c);
}

int lbcad_set_state(lbcad_ctx* c, int32_t inst, const void* src, size_t bytes, int32_t src_is_device) try {
  if (!c) return LBCAD_E_INVALID_ARG;
  return copy_state(c, inst, const_cast<void*>(src), bytes, src_is_device != 0, false);
} catch (const std::exception&) {
  return caught(c);
}

int lbcad_observables(lbcad_ctx* c, int32_t inst, lbcad_obs* out) try {
  if (!c || !out) return LBCAD_E_INVALID_ARG;
  if (inst < 0 || inst >= (int)c->inst.size()) return fail(c, LBCAD_E_INVALID_ARG, "instance out of range");
  DeviceGuard dg(c->device);
  const double* src = c->obs_latest + 12 * (size_t)inst;  // summed by the fused step
  if (!c->obs_valid) {  // another path, or the state was set: a separate reduction pass
    const Inst& I = c->inst[inst];
    long long nb = ((long long)I.g.ny * I.g.nz + kObsRowsPerBlock - 1) / kObsRowsPerBlock;
    if (nb > kObsMaxBlocks) nb = kObsMaxBlocks;
    cudaError_t e = (c->prec == LBCAD_FP64)
                        ? Launch<double, false>::observables(desc_now<double>(c, inst), c->obs_partial, (int)nb,
                                                             c->obs_out, c->stream)
                        : Launch<float, true>::observables(desc_now<float>(c, inst), c->obs_partial, (int)nb,
                                                           c->obs_out, c->stream);
    if (e != cudaSuccess) return fail(c, LBCAD_E_CUDA, std::string("observables: ") + cudaGetErrorString(e));
    src = c->obs_out;
  }
  double h[12];
  CK(c, cudaMemcpyAsync(h, src, sizeof(h), cudaMemcpyDeviceToHost, c->stream));
  CK(c, cudaStreamSynchronize(c->stream));
  out->mass = h[0];
  out->sum_psi = h[1];
  for (int a = 0; a < 3; ++a) {
    out->mom[a] = h[2 + a];
    out->cm_cos[a] = h[5 + a];
    out->cm_sin[a] = h[8 + a];
  }
  out->sum_phic = h[11];
  for (double v : h)
    if (!std::isfinite(v)) return fail(c, LBCAD_E_NAN, "non-finite value in observables");
  return LBCAD_OK;
} catch (const std::exception&) {
  return caught(c);
}

}  // extern "C"

namespace {

// Copies of one stored state: g (19), Q (5), psi (1), u (3) components of n sites.
template <typename T>
struct StateBuf {
  T* g;
  T* q;
  T* p;
  T* u;
};

template <typename T>
StateBuf<T> state_at(T* base, long long N) {
  return StateBuf<T>{base, base + 19 * N, base + 24 * N, base + 25 * N};
}

// Descriptor of one replayed step: from state `in` to `out`, its force to F (3 values per site).
template <typename T>
MarchDesc<T> replay_desc(const MarchDesc<T>& base, long long N, const StateBuf<T>& in, const StateBuf<T>& out, T* F) {
  MarchDesc<T> d = base;
  for (int i = 0; i < 19; ++i) {
    d.g_in[i] = in.g + i * N;
    d.g_out[i] = out.g + i * N;
  }
  for (int k = 0; k < 5; ++k) {
    d.q_in[k] = in.q + k * N;
    d.q_out[k] = out.q + k * N;
  }
  for (int a = 0; a < 3; ++a) {
    d.u_in[a] = in.u + a * N;
    d.u_out[a] = out.u + a * N;
    d.F[a] = F + a * N;
  }
  d.psi_in = in.p;
  d.psi_out = out.p;
  return d;
}

// Periodic centroid (per-axis circular mean of phi_c) from the FP64 moments.
void centroid_of(const lbcad_obs& o, const lbcad_grid& g, double X[3]) {
  const double L[3] = {(double)g.nx, (double)g.ny, (double)g.nz};
  for (int a = 0; a < 3; ++a) {
    double ang = std::atan2(o.cm_sin[a], o.cm_cos[a]);
    if (ang < 0) ang += 2.0 * 3.14159265358979323846;
    X[a] = ang * L[a] / (2.0 * 3.14159265358979323846);
  }
}

template <typename T, bool SHIFT>
int adjoint_impl(lbcad_ctx* c, int64_t nsteps, int k, double* dzeta, double* dq0, double* dQ0, double* J_out) {
  Inst& I = c->inst[0];
  const long long N = I.N;
  const int S = (int)((nsteps + k - 1) / k);
  const size_t st = 28 * (size_t)N;  // elements of one stored state
  const size_t fs = 3 * (size_t)N;   // elements of one step's force
  // buffers through the context's allocator, kept for the next call
  c->adj_lam = nullptr;
  T* ck = (T*)adj_buffer(c, 0, (size_t)S * st * sizeof(T));
  T* seg = (T*)adj_buffer(c, 1, (size_t)(k + 1) * st * sizeof(T));
  T* lam = (T*)adj_buffer(c, 2, 2 * st * sizeof(T));
  T* work = (T*)adj_buffer(c, 3, (kAdjWorkA + kAdjWorkL + kAdjWorkB) * (size_t)N * sizeof(T));
  T* fl = (T*)adj_buffer(c, 4, (size_t)k * fs * sizeof(T));
  // items of the reverse kernel that marches
  int tx = 0, ty = 0, per_sm = 0, sms = 0;
  CK(c, (LaunchAdj<T, SHIFT>::fields_shape(&tx, &ty, &per_sm)));
  CK(c, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device));
  std::vector<MarchItem> items;
  MarchWork aw = add_items(c, c->work[0], tx, ty, sms * std::max(per_sm, 1), items);
  const int nb = aw.grid;
  double* pg = (double*)adj_buffer(c, 5, (2 * (size_t)nb + 2) * sizeof(double));
  MarchItem* ai = (MarchItem*)adj_buffer(c, 6, items.size() * sizeof(MarchItem));
  if (!ck || !seg || !lam || !work || !fl || !pg || !ai) return fail(c, LBCAD_E_OOM, "adjoint buffers");
  T* A = work;
  T* L2 = A + kAdjWorkA * N;
  T* B = L2 + kAdjWorkL * N;
  aw.items = ai;
  CK(c, cudaMemcpyAsync(ai, items.data(), items.size() * sizeof(MarchItem), cudaMemcpyHostToDevice, c->stream));
  double* total = pg + 2 * nb;
  CK(c, cudaMemsetAsync(pg, 0, (2 * (size_t)nb + 2) * sizeof(double), c->stream));
  using Step = LaunchFused<T, SHIFT>;
  CK(c, Step::prepare_replay(c->cfg_index));
  const MarchDesc<T> base = make_march_desc<T>(I, 0, SHIFT);

  lbcad_obs o0, o1;
  int r = lbcad_observables(c, 0, &o0);
  if (r) return r;
  // forward with a checkpoint at the start of every segment
  for (int sgi = 0; sgi < S; ++sgi) {
    const int par = (int)(c->step & 1);
    const StateBuf<T> cb = state_at<T>(ck + (size_t)sgi * st, N);
    CK(c, cudaMemcpyAsync(cb.g, I.gb[par], 19 * N * sizeof(T), cudaMemcpyDeviceToDevice, c->stream));
    CK(c, cudaMemcpyAsync(cb.q, I.qb[par], 5 * N * sizeof(T), cudaMemcpyDeviceToDevice, c->stream));
    CK(c, cudaMemcpyAsync(cb.p, I.pb[par], N * sizeof(T), cudaMemcpyDeviceToDevice, c->stream));
    CK(c, cudaMemcpyAsync(cb.u, I.ub[par], 3 * N * sizeof(T), cudaMemcpyDeviceToDevice, c->stream));
    const int64_t len = std::min<int64_t>(k, nsteps - (int64_t)sgi * k);
    r = lbcad_step(c, len);
    if (r) return r;
  }
  r = lbcad_observables(c, 0, &o1);
  if (r) return r;
  double X0[3], X1[3], dX[3], ks[3], kc[3];
  centroid_of(o0, I.g, X0);
  centroid_of(o1, I.g, X1);
  const double L[3] = {(double)I.g.nx, (double)I.g.ny, (double)I.g.nz};
  double J = 0.0;
  for (int a = 0; a < 3; ++a) {
    double d = X1[a] - X0[a];
    d -= L[a] * std::round(d / L[a]);  // minimum image
    dX[a] = d;
    J += 0.5 * d * d;
    const double r2 = o1.cm_cos[a] * o1.cm_cos[a] + o1.cm_sin[a] * o1.cm_sin[a];
    const double coef = (L[a] / (2.0 * 3.14159265358979323846)) / r2;
    ks[a] = coef * o1.cm_cos[a];
    kc[a] = coef * o1.cm_sin[a];
  }
  // seed: only psi at the final time enters J
  StateBuf<T> lcur = state_at<T>(lam, N), lnxt = state_at<T>(lam + st, N);
  CK(c, cudaMemsetAsync(lam, 0, st * sizeof(T), c->stream));
  cudaError_t e = LaunchAdj<T, SHIFT>::seed(desc_now<T>(c, 0), dX, ks, kc, lcur.p, c->stream);
  if (e != cudaSuccess) return fail(c, LBCAD_E_CUDA, std::string("adjoint seed: ") + cudaGetErrorString(e));

  for (int sgi = S - 1; sgi >= 0; --sgi) {
    const int len = (int)std::min<int64_t>(k, nsteps - (int64_t)sgi * k);
    // replay the segment: states 0 .. len of this segment into seg (state 0 = checkpoint), by the kernels of
    // the step, so that the replayed states are the forward's, and the force of each step into fl
    CK(c, cudaMemcpyAsync(seg, ck + (size_t)sgi * st, st * sizeof(T), cudaMemcpyDeviceToDevice, c->stream));
    for (int j = 0; j < len; ++j) {
      const MarchDesc<T> md = replay_desc<T>(base, N, state_at<T>(seg + (size_t)j * st, N),
                                             state_at<T>(seg + (size_t)(j + 1) * st, N), fl + (size_t)j * fs);
      e = cudaSuccess;
      for (size_t w = 0; w < c->work.size() && e == cudaSuccess; ++w)
        e = Step::replay(c->cfg_index, c->work[w], &md, c->stream);
      if (e != cudaSuccess) return fail(c, LBCAD_E_CUDA, std::string("adjoint replay: ") + cudaGetErrorString(e));
    }
    // reverse steps
    for (int j = len - 1; j >= 0; --j) {
      const StateBuf<T> in = state_at<T>(seg + (size_t)j * st, N);
      AdjDescHost<T> h;
      h.I = make_desc<T>(I, 0);
      h.I.g_in = in.g; h.I.q_in = in.q; h.I.psi_in = in.p; h.I.u_in = in.u;
      h.F = fl + (size_t)j * fs;
      h.lg = lcur.g; h.lq = lcur.q; h.lp = lcur.p; h.lu = lcur.u;
      h.A = A; h.L = L2; h.B = B;
      h.work = aw;
      h.og = lnxt.g; h.oq = lnxt.q; h.op = lnxt.p; h.ou = lnxt.u;
      h.pgrad = pg;
      e = LaunchAdj<T, SHIFT>::reverse_step(h, c->stream);
      if (e != cudaSuccess) return fail(c, LBCAD_E_CUDA, std::string("adjoint reverse step: ") + cudaGetErrorString(e));
      std::swap(lcur, lnxt);
    }
  }
  e = adj_accumulate(pg, nb, total, c->stream);
  if (e != cudaSuccess) return fail(c, LBCAD_E_CUDA, std::string("adjoint sums: ") + cudaGetErrorString(e));
  // lcur holds the cotangent of the checkpointed initial state
  c->adj_lam = lcur.g;
  double tot[2];
  CK(c, cudaMemcpyAsync(tot, total, sizeof(tot), cudaMemcpyDeviceToHost, c->stream));
  // through pinned memory kept with the context: a fresh pageable vector costs its page faults and a staged copy on
  // every call (64^3: 0.4 ms)
  const size_t qn = 5 * (size_t)N;
  std::vector<T> plain;
  if (dQ0 && c->adj_host_bytes < qn * sizeof(T)) {
    if (c->adj_host) cudaFreeHost(c->adj_host);
    c->adj_host_bytes = 0;
    if (cudaHostAlloc(&c->adj_host, qn * sizeof(T), cudaHostAllocDefault) != cudaSuccess) {
      cudaGetLastError();
      c->adj_host = nullptr;
      plain.resize(qn);  // no page-locked memory left: the copy only takes longer
    } else {
      c->adj_host_bytes = qn * sizeof(T);
    }
  }
  T* const hq = plain.empty() ? (T*)c->adj_host : plain.data();
  if (dQ0) CK(c, cudaMemcpyAsync(hq, lcur.q, qn * sizeof(T), cudaMemcpyDeviceToHost, c->stream));
  CK(c, cudaStreamSynchronize(c->stream));
  if (dzeta) *dzeta = tot[0];
  if (dq0) *dq0 = tot[1];
  if (J_out) *J_out = J;
  if (dQ0)
    for (size_t i = 0; i < qn; ++i) dQ0[i] = (double)hq[i];
  for (double v : tot)
    if (!std::isfinite(v)) return fail(c, LBCAD_E_NAN, "non-finite adjoint gradient");
  return LBCAD_OK;
}

}  // namespace

extern "C" {

int lbcad_adjoint(lbcad_ctx* c, int64_t nsteps, int32_t ckpt_every, double* dJ_dzeta, double* dJ_dq0,
                  double* dJ_dQ0, double* J) try {
  if (!c) return LBCAD_E_INVALID_ARG;
  if (c->inst.size() != 1) return fail(c, LBCAD_E_UNSUPPORTED, "the adjoint runs on single-instance contexts");
  if (c->staged_only() || c->sync_split() || !c->default_lb())
    return fail(c, LBCAD_E_UNSUPPORTED, "the adjoint differentiates the Euler, lagged step of D3Q19 with the body force");
  if (nsteps < 1 || ckpt_every < 1) return fail(c, LBCAD_E_INVALID_ARG, "need nsteps >= 1 and ckpt_every >= 1");
  DeviceGuard dg(c->device);
  if (int r = ensure_step_scratch(c)) return r;
  const int k = (int)std::min<int64_t>(ckpt_every, nsteps);
  const int r = c->prec == LBCAD_FP64 ? adjoint_impl<double, false>(c, nsteps, k, dJ_dzeta, dJ_dq0, dJ_dQ0, J)
                                      : adjoint_impl<float, true>(c, nsteps, k, dJ_dzeta, dJ_dq0, dJ_dQ0, J);
  c->obs_valid = false;  // lbcad_observables forms the sums of the final state again (separate pass)
  return r;
} catch (const std::exception&) {
  return caught(c);
}

int lbcad_adjoint_fields(lbcad_ctx* c, uint32_t mask, void* dst, size_t bytes) try {
  if (!c) return LBCAD_E_INVALID_ARG;
  if (!c->adj_lam) return fail(c, LBCAD_E_INVALID_ARG, "no lbcad_adjoint has run on this context");
  if (!dst || mask == 0 || (mask & ~29u)) return fail(c, LBCAD_E_INVALID_ARG, "bad dst or mask (G, U, Q, PSI)");
  const long long N = c->inst[0].N;
  const size_t need = (size_t)ncomp_of(mask) * N * sizeof(double);
  if (bytes < need) return fail(c, LBCAD_E_INVALID_ARG, "dst too small");
  DeviceGuard dg(c->device);
  int r = ensure_staging(c, need);
  if (r) return r;
  cudaError_t e = (c->prec == LBCAD_FP64)
                      ? LaunchAdj<double, false>::export_fields(desc_now<double>(c, 0), (const double*)c->adj_lam, mask,
                                                                c->staging, c->stream)
                      : LaunchAdj<float, true>::export_fields(desc_now<float>(c, 0), (const float*)c->adj_lam, mask,
                                                              c->staging, c->stream);
  if (e != cudaSuccess) return fail(c, LBCAD_E_CUDA, std::string("adjoint export: ") + cudaGetErrorString(e));
  CK(c, cudaMemcpyAsync(dst, c->staging, need, cudaMemcpyDeviceToHost, c->stream));
  CK(c, cudaStreamSynchronize(c->stream));
  return LBCAD_OK;
} catch (const std::exception&) {
  return caught(c);
}

int lbcad_num_instances(const lbcad_ctx* c) { return c ? (int)c->inst.size() : 0; }

int lbcad_instance_grid(const lbcad_ctx* c, int32_t inst, lbcad_grid* out) {
  if (!c || !out || inst < 0 || inst >= (int)c->inst.size()) return LBCAD_E_INVALID_ARG;
  *out = c->inst[inst].g;
  return LBCAD_OK;
}

int64_t lbcad_step_count(const lbcad_ctx* c) { return c ? c->step : -1; }

void* lbcad_stream(const lbcad_ctx* c) { return c ? (void*)c->stream : nullptr; }

int lbcad_sync(lbcad_ctx* c) try {
  if (!c) return LBCAD_E_INVALID_ARG;
  DeviceGuard dg(c->device);
  CK(c, cudaStreamSynchronize(c->stream));
  CK(c, cudaGetLastError());
  return LBCAD_OK;
} catch (const std::exception&) {
  return caught(c);
}

void lbcad_destroy(lbcad_ctx* c) {
  if (!c) return;
  release(c);
  delete c;
}

const char* lbcad_last_error(const lbcad_ctx* c) { return c ? c->err.c_str() : g_create_err.c_str(); }

}  // extern "C"
