// C ABI of the library (declared in include/sem.h): mesh set-up, host-side tables and
// the orchestration of the kernels for one Laplace solve, the recovery, the Zakharov
// right-hand side and RK4 (§2–§3 of arXiv 1512.02548).
#include <algorithm>
#include <array>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <queue>
#include <mutex>
#include <tuple>
#include <memory>
#include <string>
#include <utility>
#include <vector>

#include "sem.h"
#include "mesh_index.cuh"
#include "sem_internal.cuh"
#include "tables.h"

using namespace semgb;

namespace semgb {
static std::atomic<long long> g_launches{0};
void count_launch(int k) { g_launches.fetch_add(k, std::memory_order_relaxed); }
}  // namespace semgb

namespace {

constexpr int kMaxWaveComp = 4096;
thread_local std::string t_err;

int fail(int code, const std::string& msg) {
  t_err = msg;
  return code;
}

#define CUDA_TRY(call)                                                                      \
  do {                                                                                      \
    cudaError_t e_ = (call);                                                                \
    if (e_ != cudaSuccess)                                                                  \
      return fail(SEM_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_));        \
  } while (0)

std::mutex g_tables_mu;
bool g_tables_done[64] = {false};

int ensure_device_tables(int dev) {
  std::lock_guard<std::mutex> lk(g_tables_mu);
  if (dev < 0 || dev >= 64) return fail(SEM_ERR_INVALID_ARG, "device index out of range");
  if (g_tables_done[dev]) return SEM_OK;
  std::vector<double> D(kDTotal, 0.0), w(kWTotal, 0.0);
  for (int P = 1; P <= kMaxP; ++P) {
    Line L = make_line(P);
    std::memcpy(&D[d_off(P)], L.D.data(), sizeof(double) * (P + 1) * (P + 1));
    std::memcpy(&w[w_off(P)], L.w.data(), sizeof(double) * (P + 1));
  }
  CUDA_TRY(upload_line_tables(D.data(), w.data()));
  g_tables_done[dev] = true;
  return SEM_OK;
}

// Device memory of meshes and batches comes from a per-device cache of freed blocks, so that
// a serving loop that creates and destroys meshes per request does not pay cudaMalloc and
// cudaFree for each.  A freed block is kept (up to kCacheBytes per device) and handed to a
// later request of at most its size and at least half of it.  sem_trim_cache returns the
// cached blocks to CUDA.
constexpr size_t kCacheBytes = 8ull << 30;
struct BlockCache {
  std::multimap<size_t, void*> free;          // size → block
  std::map<void*, size_t> size_of;            // every block this cache handed out or holds
  size_t cached = 0;
};
std::mutex g_cache_mu;
BlockCache g_cache[64];

cudaError_t dev_alloc(int dev, size_t bytes, void** p) {
  {
    std::lock_guard<std::mutex> lk(g_cache_mu);
    BlockCache& c = g_cache[dev];
    auto it = c.free.lower_bound(bytes);
    if (it != c.free.end() && it->first <= 2 * bytes) {
      *p = it->second;
      c.cached -= it->first;
      c.free.erase(it);
      return cudaSuccess;
    }
  }
  cudaError_t e = cudaMalloc(p, bytes);
  if (e == cudaErrorMemoryAllocation) {        // give the cached blocks back and retry once
    sem_trim_cache();
    cudaGetLastError();
    e = cudaMalloc(p, bytes);
  }
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(g_cache_mu);
  g_cache[dev].size_of[*p] = bytes;
  return cudaSuccess;
}

// The block must have no work in flight; the callers synchronise the device first.
void dev_free(int dev, void* p) {
  if (!p) return;
  std::lock_guard<std::mutex> lk(g_cache_mu);
  BlockCache& c = g_cache[dev];
  auto it = c.size_of.find(p);
  const size_t sz = it == c.size_of.end() ? 0 : it->second;
  if (sz > 0 && c.cached + sz <= kCacheBytes) {
    c.free.emplace(sz, p);
    c.cached += sz;
  } else {
    if (it != c.size_of.end()) c.size_of.erase(it);
    cudaFree(p);
  }
}

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    cudaGetDevice(&prev);
    if (prev != dev) cudaSetDevice(dev);
  }
  ~DeviceGuard() {
    int cur = -1;
    cudaGetDevice(&cur);
    if (prev >= 0 && cur != prev) cudaSetDevice(prev);
  }
};

// Bump allocator over one device allocation (256-byte aligned slices).
struct Carve {
  size_t off = 0;
  template <class T> size_t take(size_t count) {
    size_t o = (off + 255) & ~size_t(255);
    off = o + count * sizeof(T);
    return o;
  }
};

}  // namespace

struct sem_mesh {
  sem_params p{};
  int device = 0;
  int ncol = 0, nrow = 0, Pf = 0, nif = 0;
  long long n = 0;
  int grid = 0;
  unsigned char* pool = nullptr;
  size_t pool_bytes = 0;
  DevGeom g{};
  SurfTables st{};
  PcgArgs pa{};
  PrecSetup ps{};
  SolveRecord* rec = nullptr;
  // workspace
  double *Phi = nullptr, *qtmp = nullptr, *edgetmp = nullptr;
  double *wt = nullptr, *etax = nullptr, *phisx = nullptr, *R = nullptr, *R2 = nullptr, *ub = nullptr;
  double *ke = nullptr, *kp = nullptr, *ae = nullptr, *ap = nullptr, *se = nullptr, *sp = nullptr;
  double *eta_dev = nullptr, *phis_dev = nullptr;
  double *s1e = nullptr, *s1p = nullptr;   // second stage-input pair of the fused RK stage
  // kept for the stages' initial guesses (Instance), and the dt of the last fused RK call (NaN: none)
  double *Pl = nullptr, *eend = nullptr, *pend = nullptr;
  float* H = nullptr;
  int* hist_d = nullptr;
  // column positions on the host, and the cos/sin(k x) table of the left-zone columns for the
  // generated signal (its own device block, rebuilt by sem_set_wave_input)
  std::vector<double> xcol_h;
  double* wkx = nullptr;
  double hist_dt = NAN;
  unsigned int* stage_bars = nullptr;   // barrier pair of this mesh's own fused stage launch
  int stage_team = 0;
  bool solve_wide = false;       // the stand-alone solve's launch: two CTAs per SM
  size_t stage_smem = 0;         // the mesh's own fused stage launch (with the factor cache)
  size_t stage_smem_batch = 0;   // in a batch launch (no factor cache)
  int gcache = 0;                // doubles of the factor cache in the own launch (0 = none)
  int own_chunk = 0;             // element columns per pass in the own launch (g.chunk elsewhere)
  bool fused = true;
  // optional event timing of the Krylov kernel
  bool timing = false;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> events;
  std::vector<cudaEvent_t> spare;
};

// A batch: instances grouped by (order, precision) and, within a group, into launches of at
// most the co-resident capacity; each instance gets a team of CTAs sized to its work.
struct BatchLaunch {
  int P = 0, mixed = 0, wide = 1;
  int csize = 0;                     // cluster teams of csize CTAs each (0: one cooperative launch)
  std::vector<int> members;          // mesh indices
  std::vector<int> team0, nteam;
  std::vector<int> chunk;            // element columns per pass of each member
  int grid = 0;
  size_t smem = 0;
  Instance* inst_d = nullptr;
  int* cta_d = nullptr;
  unsigned int* bars_d = nullptr;
  int* status_d = nullptr;           // gathered status words of the members
  std::vector<Instance> inst_h;
  std::vector<int> status_h;
  cudaStream_t stream = nullptr;     // cluster launches: the launch's own stream
  cudaEvent_t done = nullptr;        // ... and the event that joins it back to the caller's stream
};

struct sem_batch {
  std::vector<sem_mesh*> meshes;
  std::vector<int> codes;            // per-instance error code of the last step or solve
  std::vector<BatchLaunch> launches;     // cooperative plan: one launch per RK stage and group
  std::vector<BatchLaunch> cl_launches;  // cluster plan: launches on streams of their own (empty: none)
  // the Laplace solves' plan, made by the first of them: −1 not made, 0 cooperative, 1 the steps' clusters, 2 cl_solve
  int solve_plan = -1;
  std::vector<BatchLaunch> cl_solve;
  unsigned char* solve_pool = nullptr;
  sem_batch_tuning tune{};
  int force = -1;                        // plan asked for: −1 the faster by estimate, 0 cooperative, 1 clusters
  cudaEvent_t fork = nullptr;
  int device = 0;
  unsigned char* pool = nullptr;
  // packed device copy of every member's (η, φ̃) for sem_batch_rk4_step_host: η of member i at
  // state + off[i], φ̃ at state + ncol_total + off[i]
  double* state = nullptr;
  std::vector<size_t> off;
  size_t ncol_total = 0;
  // optional event timing of the stage launches
  bool timing = false;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> events;
  std::vector<cudaEvent_t> spare;
};

namespace {

// Error code of a device status word (no message).
int status_code(int st) {
  if (st == 0) return SEM_OK;
  if (st & ST_TIMEOUT) return SEM_ERR_TIMEOUT;
  if (st & (ST_BAD_DEPTH | ST_NONFINITE)) return SEM_ERR_NONFINITE;
  if (st & ST_NOT_CONVERGED) return SEM_ERR_NOT_CONVERGED;
  return SEM_ERR_CUDA;
}

int status_error(int st) {
  if (st == 0) return SEM_OK;
  if (st & ST_TIMEOUT) return fail(SEM_ERR_TIMEOUT, "a grid barrier of the Krylov kernel timed out");
  if (st & ST_BAD_DEPTH) return fail(SEM_ERR_NONFINITE, "water depth d = eta + h is not positive and finite");
  if (st & ST_NONFINITE) return fail(SEM_ERR_NONFINITE, "non-finite residual in the Laplace solve");
  if (st & ST_NOT_CONVERGED) return fail(SEM_ERR_NOT_CONVERGED, "Laplace solve reached max_iter above tol");
  return fail(SEM_ERR_CUDA, "unknown device status");
}

// After a failed step the mesh's warm-start potential may hold non-finite values; the next
// solve on this mesh starts from zero instead.
cudaError_t reset_warm_start(sem_mesh* m, cudaStream_t s) {
  m->hist_dt = NAN;   // the stage potentials kept for initial guesses may be from a failed step
  return cudaMemsetAsync(m->Phi, 0, sizeof(double) * (size_t)m->n, s);
}

int read_status(sem_mesh* m, cudaStream_t s) {
  int st = 0;
  CUDA_TRY(cudaMemcpyAsync(&st, m->g.status, sizeof(int), cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  if (st == 0) return SEM_OK;
  CUDA_TRY(reset_warm_start(m, s));
  CUDA_TRY(cudaMemsetAsync(m->g.status, 0, sizeof(int), s));
  CUDA_TRY(cudaStreamSynchronize(s));
  return status_error(st);
}

cudaError_t take_event(sem_mesh* m, cudaEvent_t* ev) {
  if (!m->spare.empty()) { *ev = m->spare.back(); m->spare.pop_back(); return cudaSuccess; }
  return cudaEventCreate(ev);
}

int do_solve(sem_mesh* m, const double* phis, double* Phi, cudaStream_t s) {
  PcgArgs a = m->pa;
  a.x = Phi;
  a.phis = phis;
  a.start_margin = 1.0;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (m->timing) {
    CUDA_TRY(take_event(m, &e0));
    CUDA_TRY(take_event(m, &e1));
    CUDA_TRY(cudaEventRecord(e0, s));
  }
  DevGeom g = m->g;
  if (m->solve_wide) {
    CUDA_TRY(launch_pcg(g, a, 1, m->grid, m->stage_smem_batch, s));
  } else {   // the shape of the mesh's own fused stage launch: one pass over a CTA's columns, the factor cache
    g.chunk = m->own_chunk;
    g.gcache = m->gcache;
    CUDA_TRY(launch_pcg(g, a, 0, m->stage_team, m->stage_smem, s));
  }
  if (m->timing) {
    CUDA_TRY(cudaEventRecord(e1, s));
    m->events.emplace_back(e0, e1);
  }
  return SEM_OK;
}

int do_geometry(sem_mesh* m, const double* eta, cudaStream_t s) {
  const bool jacobi = m->p.precond == SEM_PRECOND_JACOBI;
  CUDA_TRY(launch_geometry(m->g, eta, jacobi, s));
  if (!jacobi) CUDA_TRY(launch_prec_setup(m->g, m->ps, s));
  return SEM_OK;
}

// Do na doubles at a and nb doubles at b share an address?
bool overlap(const double* a, size_t na, const double* b, size_t nb) {
  const uintptr_t pa = reinterpret_cast<uintptr_t>(a), pb = reinterpret_cast<uintptr_t>(b);
  return pa < pb + nb * sizeof(double) && pb < pa + na * sizeof(double);
}

bool has_zones(const sem_mesh* m) { return m->p.relax_left > 0.0 || m->p.relax_right > 0.0; }

int launch_own_stage(sem_mesh* m, const StageArgs& a, cudaStream_t s);
Instance make_instance(sem_mesh* m, double* eta, double* phis, double tstart, double dt, int team0, int nteam,
                       bool own_launch = false, int chunk = 0);

int do_rhs(sem_mesh* m, const double* eta, const double* phis, double time, double tau, double* de,
           double* dp, cudaStream_t s) {
  if (m->fused) {   // the fused stage without its RK4 update: one launch instead of seven
    StageArgs a{nullptr, nullptr, m->stage_bars, 5, 0, 0,
                make_instance(m, const_cast<double*>(eta), const_cast<double*>(phis), time, 1.0, 0, m->stage_team, true)};
    a.own.ke = de;
    a.own.kp = dp;
    a.own.tau = tau;
    return launch_own_stage(m, a, s);
  }
  int rc0 = do_geometry(m, eta, s);
  if (rc0) return rc0;
  int rc = do_solve(m, phis, m->Phi, s);
  if (rc) return rc;
  CUDA_TRY(launch_recover(m->st, m->Phi, eta, phis, m->wt, m->etax, m->phisx, s));
  CUDA_TRY(launch_zakharov(m->st, eta, m->etax, m->phisx, m->wt, m->R, s));
  CUDA_TRY(launch_mass1d(m->st, m->R, de, dp, s));
  if (has_zones(m)) CUDA_TRY(launch_relax(m->st, eta, phis, time, 1.0 / tau, de, dp, s));
  return SEM_OK;
}

// own_launch: the mesh's own fused stage launch, whose shared memory holds the factor cache.
// chunk > 0: element columns per pass in a batch launch.
Instance make_instance(sem_mesh* m, double* eta, double* phis, double tstart, double dt, int team0,
                       int nteam, bool own_launch, int chunk) {
  Instance I{};
  I.g = m->g;
  I.g.gcache = own_launch ? m->gcache : 0;
  if (own_launch) I.g.chunk = m->own_chunk;
  else if (chunk > 0) I.g.chunk = chunk;
  I.st = m->st;
  I.pa = m->pa;
  I.pa.x = m->Phi;
  I.ps = m->ps;
  I.eta = eta; I.phis = phis;
  I.s0e = m->se; I.s0p = m->sp; I.s1e = m->s1e; I.s1p = m->s1p;
  I.ke = m->ke; I.kp = m->kp; I.ae = m->ae; I.ap = m->ap;
  I.wt = m->wt; I.R = m->R; I.R2 = m->R2; I.ub = m->ub; I.ub_stride = m->p.Nx + m->grid + 1;
  I.Pl = m->Pl; I.H = m->H; I.hist_d = m->hist_d; I.eend = m->eend; I.pend = m->pend;
  I.hist = m->hist_dt == dt ? 1 : 0;
  I.tstart = tstart; I.dt = dt;
  I.tau = m->p.relax_tau > 0.0 ? m->p.relax_tau : dt;
  I.team0 = team0; I.nteam = nteam;
  I.relax = has_zones(m) ? 1 : 0;
  return I;
}

// One fused stage launch of a mesh alone (a.own filled in).
int launch_own_stage(sem_mesh* m, const StageArgs& a, cudaStream_t s) {
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (m->timing) {
    CUDA_TRY(take_event(m, &e0));
    CUDA_TRY(take_event(m, &e1));
    CUDA_TRY(cudaEventRecord(e0, s));
  }
  CUDA_TRY(launch_stage(m->p.P, m->p.precision == SEM_PREC_MIXED, 0, a, m->stage_team, m->stage_smem, s));
  if (m->timing) {
    CUDA_TRY(cudaEventRecord(e1, s));
    m->events.emplace_back(e0, e1);
  }
  return SEM_OK;
}

// nsteps RK4 steps of one mesh with the fused stage kernel: one cooperative launch per stage.
int do_rk4_fused(sem_mesh* m, double* eta, double* phis, double t0, double dt, int nsteps, cudaStream_t s) {
  StageArgs a{nullptr, nullptr, m->stage_bars, 1, 0, 0, make_instance(m, eta, phis, t0, dt, 0, m->stage_team, true)};
  for (int step = 0; step < nsteps; ++step)
    for (int stage = 1; stage <= 4; ++stage) {
      a.stage = stage;
      a.step = step;
      const int rc = launch_own_stage(m, a, s);
      if (rc) return rc;
    }
  if (nsteps > 0) m->hist_dt = dt;
  return SEM_OK;
}

int do_rk4(sem_mesh* m, double* eta, double* phis, double t0, double dt, int nsteps, cudaStream_t s) {
  if (m->fused) return do_rk4_fused(m, eta, phis, t0, dt, nsteps, s);
  const int n = m->ncol;
  const double tau = m->p.relax_tau > 0.0 ? m->p.relax_tau : dt;
  for (int step = 0; step < nsteps; ++step) {
    const double ts = t0 + step * dt;
    for (int stage = 1; stage <= 4; ++stage) {
      const double* ei = stage == 1 ? eta : m->se;
      const double* pi = stage == 1 ? phis : m->sp;
      const double tstage = ts + (stage == 1 ? 0.0 : (stage == 4 ? dt : 0.5 * dt));
      int rc = do_rhs(m, ei, pi, tstage, tau, m->ke, m->kp, s);
      if (rc) return rc;
      CUDA_TRY(launch_rk4_stage(stage, n, dt, eta, phis, m->ke, m->kp, m->ae, m->ap, m->se, m->sp, s));
    }
    CUDA_TRY(launch_filter(m->st, eta, phis, s));
  }
  return SEM_OK;
}

}  // namespace

extern "C" {

const char* sem_last_error(void) { return t_err.c_str(); }

int64_t sem_launch_count(void) { return g_launches.load(); }

// Host tables of one (P, Nz, Pf, filter) combination, shared by every mesh that has it.
struct ColumnTables {
  Line L;
  std::vector<double> SX, I, ZB, F, wrow, Z, Sg, lam, dsl, sig;
  int win = 0;
  long double S00 = 0, S01 = 0, S11 = 0;
};

static std::mutex g_ct_mu;
static std::map<std::tuple<int, int, int, double, double, int>, std::shared_ptr<const ColumnTables>> g_ct;

static int column_tables(const sem_params& p, std::shared_ptr<const ColumnTables>* out) {
  const auto key = std::make_tuple(p.P, p.Nz, p.Pf, p.filter_alpha, p.filter_s, p.filter_ic);
  {
    std::lock_guard<std::mutex> lk(g_ct_mu);
    auto it = g_ct.find(key);
    if (it != g_ct.end()) { *out = it->second; return SEM_OK; }
  }
  auto t = std::make_shared<ColumnTables>();
  const int P = p.P, Q = P + 1, Nz = p.Nz, nrow = Nz * P + 1, Qf = p.Pf + 1, Pm = P - 1;
  Line Lf;
  try {
    t->L = make_line(P);
    Lf = make_line(p.Pf);
  } catch (const std::exception& e) {
    return fail(SEM_ERR_INVALID_ARG, e.what());
  }
  const Line& L = t->L;
  t->dsl.assign(Nz, 1.0 / Nz);
  const std::vector<double>& dsl = t->dsl;
  t->sig.resize(nrow);
  for (int iz = 0; iz < nrow; ++iz) {
    int l = iz / P; if (l >= Nz) l = Nz - 1;
    const int b = iz - l * P;
    t->sig[iz] = (double)l / Nz + 0.5 * (L.r[b] + 1.0) * dsl[l];
  }
  t->sig[nrow - 1] = 1.0;
  t->I = interpolation(L, Lf);                                        // Qf×Q
  t->F = filter_matrix(L, p.filter_alpha, p.filter_s, p.filter_ic);
  // w̃ weights: v = M_σ⁻¹ e_top, c_l = (Δσ_l/2) M v|_l, contracted with the layer's σ-derivative
  // (2/Δσ_l) D into one weight per row: w̃ d = Σ_iz wrow_iz Φ_iz
  t->wrow.assign((size_t)nrow, 0.0);
  {
    std::vector<long double> wr((size_t)nrow, 0.0L);
    std::vector<long double> Ms((size_t)nrow * nrow, 0.0L);
    for (int l = 0; l < Nz; ++l)
      for (int a = 0; a < Q; ++a)
        for (int b = 0; b < Q; ++b) Ms[(size_t)(l * P + a) * nrow + l * P + b] += 0.5L * dsl[l] * L.M[a * Q + b];
    if (!invert(Ms, nrow)) return fail(SEM_ERR_INVALID_ARG, "sigma mass is singular");
    for (int l = 0; l < Nz; ++l)
      for (int b = 0; b < Q; ++b) {
        long double s = 0.0L;
        for (int c = 0; c < Q; ++c) s += 0.5L * dsl[l] * L.M[b * Q + c] * Ms[(size_t)(l * P + c) * nrow + (nrow - 1)];
        for (int c = 0; c < Q; ++c) wr[(size_t)l * P + c] += s * (2.0L / dsl[l]) * L.D[b * Q + c];
      }
    for (int iz = 0; iz < nrow; ++iz) t->wrow[iz] = (double)wr[iz];
  }
  // static condensation of M' (element scale Δx/2 · M): Z = M_bi M_ii⁻¹, the Schur complement, and the
  // element right-hand sides R = T f (T = M·D, Iᵀ M_f) condensed: boundary rows T_b − Z T_i, interior
  // rows M_ii⁻¹ T_i
  t->Z.assign((size_t)2 * Pm, 0.0);
  {
    std::vector<long double> Mii((size_t)Pm * Pm);
    for (int i = 0; i < Pm; ++i) for (int k = 0; k < Pm; ++k) Mii[i * Pm + k] = L.M[(i + 1) * Q + (k + 1)];
    if (!invert(Mii, Pm)) return fail(SEM_ERR_INVALID_ARG, "interior mass is singular");
    const int bn[2] = {0, P};
    long double Zl[2][kMaxP];
    for (int s2 = 0; s2 < 2; ++s2)
      for (int i = 0; i < Pm; ++i) {
        long double acc = 0.0L;
        for (int k = 0; k < Pm; ++k) acc += (long double)L.M[bn[s2] * Q + (k + 1)] * Mii[k * Pm + i];
        Zl[s2][i] = acc;
        t->Z[s2 * Pm + i] = (double)acc;
      }
    auto sch = [&](int s1, int s2) {
      long double acc = L.M[bn[s1] * Q + bn[s2]];
      for (int i = 0; i < Pm; ++i) acc -= Zl[s1][i] * (long double)L.M[(i + 1) * Q + bn[s2]];
      return acc;
    };
    t->S00 = sch(0, 0); t->S01 = sch(0, 1); t->S11 = sch(1, 1);
    auto condensed = [&](const std::vector<double>& Lf_, const std::vector<double>& Rt, int k, int nc) {
      // T = Lf_ (Q×k) · Rt (k×nc) in long double, then its condensed rows
      std::vector<long double> T((size_t)Q * nc, 0.0L);
      for (int a = 0; a < Q; ++a)
        for (int c = 0; c < nc; ++c)
          for (int q = 0; q < k; ++q) T[(size_t)a * nc + c] += (long double)Lf_[(size_t)a * k + q] * Rt[(size_t)q * nc + c];
      std::vector<double> out((size_t)Q * nc);
      for (int c = 0; c < nc; ++c) {
        long double b0 = T[c], b1 = T[(size_t)P * nc + c];
        for (int i = 0; i < Pm; ++i) {
          b0 -= Zl[0][i] * T[(size_t)(1 + i) * nc + c];
          b1 -= Zl[1][i] * T[(size_t)(1 + i) * nc + c];
          long double v = 0.0L;
          for (int m2 = 0; m2 < Pm; ++m2) v += Mii[i * Pm + m2] * T[(size_t)(1 + m2) * nc + c];
          out[(size_t)(1 + i) * nc + c] = (double)v;
        }
        out[c] = (double)b0;
        out[(size_t)P * nc + c] = (double)b1;
      }
      return out;
    };
    std::vector<double> It((size_t)Q * Qf);
    for (int q = 0; q < Qf; ++q) for (int c = 0; c < Q; ++c) It[(size_t)c * Qf + q] = t->I[(size_t)q * Q + c];
    t->SX = condensed(L.M, L.D, Q, Q);
    t->ZB = condensed(It, Lf.M, Qf, Qf);
    // |S01|/S00 = 1/(P+1) bounds the decay of the interface factors (surface_device.cuh)
    t->win = (int)std::ceil(18.0L * std::log(10.0L) / std::log(t->S00 / std::fabs(t->S01)));
  }
  // σ-separable preconditioner: Kσ S = Mσ S Λ on the interior rows (Dirichlet at the surface),
  // Kσ = Σ_l (2/Δσ_l) Dᵀ W D, Mσ = Σ_l (Δσ_l/2) W (GLL-lumped, as in the stiffness quadrature).
  const int nr = nrow - 1;
  t->Sg.assign((size_t)nr * nr, 0.0);
  t->lam.assign(nr, 0.0);
  {
    std::vector<long double> Ks((size_t)nrow * nrow, 0.0L), Ms(nrow, 0.0L);
    for (int l = 0; l < Nz; ++l)
      for (int a = 0; a < Q; ++a) {
        Ms[l * P + a] += 0.5L * dsl[l] * L.w[a];
        for (int b = 0; b < Q; ++b) {
          long double s2 = 0.0L;
          for (int c = 0; c < Q; ++c) s2 += (long double)L.D[c * Q + a] * L.w[c] * L.D[c * Q + b];
          Ks[(size_t)(l * P + a) * nrow + l * P + b] += (2.0L / dsl[l]) * s2;
        }
      }
    std::vector<long double> Bm((size_t)nr * nr), ev, V;
    for (int i = 0; i < nr; ++i)
      for (int j = 0; j < nr; ++j) Bm[(size_t)i * nr + j] = Ks[(size_t)i * nrow + j] / std::sqrt(Ms[i] * Ms[j]);
    sym_eig(Bm, nr, ev, V);
    for (int k = 0; k < nr; ++k) t->lam[k] = (double)ev[k];
    for (int j = 0; j < nr; ++j)
      for (int k = 0; k < nr; ++k) t->Sg[(size_t)j * nr + k] = (double)(V[(size_t)j * nr + k] / std::sqrt(Ms[j]));
  }
  std::lock_guard<std::mutex> lk(g_ct_mu);
  auto ins = g_ct.emplace(key, std::shared_ptr<const ColumnTables>(t));
  *out = ins.first->second;
  return SEM_OK;
}

static int mesh_create_impl(const sem_params* pin, const double* x_edges_h, const double* h_h, sem_mesh** out,
                            size_t* footprint_only);

int sem_mesh_create(const sem_params* pin, const double* x_edges_h, const double* h_h, sem_mesh** out) {
  if (!out) return fail(SEM_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  return mesh_create_impl(pin, x_edges_h, h_h, out, nullptr);
}

int sem_mesh_footprint(const sem_params* p, const double* x_edges_h, const double* h_h, int64_t* bytes) {
  if (!bytes) return fail(SEM_ERR_INVALID_ARG, "bytes is NULL");
  size_t b = 0;
  sem_mesh* unused = nullptr;
  const int rc = mesh_create_impl(p, x_edges_h, h_h, &unused, &b);
  *bytes = (int64_t)b;
  return rc;
}

static int mesh_create_impl(const sem_params* pin, const double* x_edges_h, const double* h_h, sem_mesh** out,
                            size_t* footprint_only) {
  if (!pin || !x_edges_h || !h_h) return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  sem_params p = *pin;
  const int Nx_in = p.Nx > 0 ? p.Nx : 0;
  if (p.P < 2 || p.P > SEM_MAX_P) return fail(SEM_ERR_INVALID_ARG, "P must be in [2, 12]");
  if (p.Nz < 1 || p.Nz > kMaxNz) return fail(SEM_ERR_INVALID_ARG, "Nz must be in [1, 16]");
  if (p.periodic ? p.Nx < 3 : p.Nx < 1) return fail(SEM_ERR_INVALID_ARG, "Nx too small (periodic needs >= 3)");
  if (p.Pf == 0) p.Pf = p.P;
  if (p.Pf < p.P || p.Pf > 3 * p.P) return fail(SEM_ERR_INVALID_ARG, "Pf must be in [P, 3P]");
  if (p.precision != SEM_PREC_FP64 && p.precision != SEM_PREC_MIXED)
    return fail(SEM_ERR_INVALID_ARG, "unknown precision");
  if (p.precond != SEM_PRECOND_SEPARABLE && p.precond != SEM_PRECOND_JACOBI)
    return fail(SEM_ERR_INVALID_ARG, "unknown preconditioner");
  if (p.relax_left < 0.0 || p.relax_right < 0.0 || p.relax_tau < 0.0 ||
      p.relax_left + p.relax_right > x_edges_h[Nx_in] - x_edges_h[0])
    return fail(SEM_ERR_INVALID_ARG, "relaxation zones must be non-negative and fit in the tank");
  if (p.tol <= 0.0) p.tol = 1e-13;
  if (p.max_iter <= 0) p.max_iter = 5000;
  const int P = p.P, Q = P + 1, Nx = p.Nx, Nz = p.Nz;
  const int ncol = p.periodic ? Nx * P : Nx * P + 1;
  const int nrow = Nz * P + 1;
  const long long n = (long long)ncol * nrow;
  for (int i = 0; i < Nx; ++i)
    if (!(x_edges_h[i + 1] > x_edges_h[i])) return fail(SEM_ERR_INVALID_ARG, "x_edges must increase");
  for (int i = 0; i < ncol; ++i)
    if (!(h_h[i] > 0.0) || !std::isfinite(h_h[i])) return fail(SEM_ERR_INVALID_ARG, "h must be positive");

  int dev = 0;
  CUDA_TRY(cudaGetDevice(&dev));
  int rc = ensure_device_tables(dev);
  if (rc) return rc;

  // ---- host tables --------------------------------------------------------------
  // Tables that depend only on (P, Nz, Pf, filter) come from a per-process cache (they are
  // built in long double, which is software-emulated on some hosts); the x-dependent ones
  // below are O(Nx) in double.
  std::shared_ptr<const ColumnTables> ct;
  rc = column_tables(p, &ct);
  if (rc) return rc;
  const Line& L = ct->L;
  const std::vector<double>& I = ct->I;
  const std::vector<double>& F = ct->F;
  const std::vector<double>& wrow = ct->wrow;
  const std::vector<double>& Z = ct->Z;
  const std::vector<double>& Sg = ct->Sg;
  const std::vector<double>& lam = ct->lam;
  const std::vector<double>& dsl = ct->dsl;
  const std::vector<double>& sig = ct->sig;
  const int Qf = p.Pf + 1, Pm = P - 1;
  std::vector<double> dxe(Nx), hx_loc((size_t)Nx * Q), se(Nx);
  for (int e = 0; e < Nx; ++e) { dxe[e] = x_edges_h[e + 1] - x_edges_h[e]; se[e] = 0.5 * dxe[e]; }
  for (int e = 0; e < Nx; ++e)
    for (int a = 0; a < Q; ++a) {
      double s = 0.0;
      for (int c = 0; c < Q; ++c) {
        int col = e * P + c; if (col >= ncol) col -= ncol;
        s = std::fma(L.D[a * Q + c], h_h[col], s);
      }
      hx_loc[(size_t)e * Q + a] = s * 2.0 / dxe[e];
    }
  // M' interface tridiagonal: pivots p_j = d_j − e²_{j−1}/p_{j−1}, around the ring until they repeat when
  // periodic (the factors of a cyclic bidiagonal LDLᵀ; their start is forgotten within ct->win steps)
  const int N = p.periodic ? Nx : Nx + 1;
  std::vector<double> th_al(N, 0.0), th_m(N, 0.0), th_cp(N, 0.0);
  {
    const double S00 = ct->S00, S01 = ct->S01, S11 = ct->S11;
    std::vector<double> d(N, 0.0), e(N, 0.0);
    for (int j = 0; j < Nx; ++j) {
      const int jr = (j + 1) % N;
      d[j] += se[j] * S00;
      d[jr] += se[j] * S11;
      e[j] = se[j] * S01;            // coupling j ↔ j+1 (periodic: e[N−1] couples N−1 and 0)
    }
    double l = 0.0;                  // multiplier e_{j−1}/p_{j−1}
    if (p.periodic)
      for (int k = ct->win; k > 0; --k) {
        const int j = ((N - k) % N + N) % N;
        l = e[j] / (d[j] - e[(j + N - 1) % N] * l);
      }
    for (int j = 0; j < N; ++j) {
      const double ep = j > 0 ? e[j - 1] : (p.periodic ? e[N - 1] : 0.0);
      th_m[j] = 1.0 / (d[j] - ep * l);
      th_al[j] = -ep * th_m[j];
      l = th_cp[j] = e[j] * th_m[j];
    }
  }
  const int nr = nrow - 1;

  // ---- device allocation -------------------------------------------------------
  sem_mesh* m = new sem_mesh;
  m->p = p; m->device = dev; m->ncol = ncol; m->nrow = nrow; m->n = n; m->Pf = p.Pf; m->nif = N;
  const int chunk = chunk_width(P, Nz);
  cudaError_t ge = pcg_grid_size(P, Nz, nrow, Nx, chunk, p.precision == SEM_PREC_MIXED, 1, &m->grid);
  if (ge != cudaSuccess) { delete m; return fail(SEM_ERR_CUDA, std::string("Krylov kernel occupancy: ") + cudaGetErrorString(ge)); }
  if (const char* lim = std::getenv("SEM_GRID_LIMIT")) {   // tuning/testing knob: cap the Krylov grid
    const int v = std::atoi(lim);
    if (v >= 1 && v < m->grid) m->grid = v;
  }

  const char* fz = std::getenv("SEM_FUSED_STAGE");
  m->fused = !(fz && fz[0] == '0') && p.precond == SEM_PRECOND_SEPARABLE;

  Carve cv;
  const size_t nE = (size_t)Nx * nrow;
  // Only what the mesh's own solves and steps use: the Krylov vectors of its precision, the inverse diagonal
  // with the Jacobi preconditioner, the guess history (72 bytes a node) with the fused stages.
  const bool mixed = p.precision == SEM_PREC_MIXED;
  const size_t n64 = mixed ? 0 : n, n32 = mixed ? n : 0, nJ = p.precond == SEM_PRECOND_JACOBI ? n : 0,
               nH = m->fused ? n : 0;
  // the arrays filled on the host come first: one copy uploads all of them ([0, up_end) of the block)
  const size_t o_cxz = cv.take<double>((size_t)Nx * Nz * 2), o_r2dx = cv.take<double>(Nx);
  const size_t o_h = cv.take<double>(ncol), o_hx = cv.take<double>((size_t)Nx * Q), o_dxe = cv.take<double>(Nx),
               o_dsl = cv.take<double>(Nz), o_sig = cv.take<double>(nrow);
  const size_t o_S32 = cv.take<float>((size_t)nr * nr), o_ST32 = cv.take<float>((size_t)nr * nr),
               o_lam = cv.take<double>(nr), o_xcol = cv.take<double>(ncol);
  // surface tables
  const size_t o_tSX = cv.take<double>(Q * Q), o_tZB = cv.take<double>((size_t)Q * Qf),
               o_tI = cv.take<double>((size_t)Qf * Q), o_tF = cv.take<double>(Q * Q), o_twr = cv.take<double>((size_t)nrow),
               o_tZ = cv.take<double>((size_t)2 * Pm + 1), o_tse = cv.take<double>(Nx), o_tal = cv.take<double>(N),
               o_tm = cv.take<double>(N), o_tcp = cv.take<double>(N);
  const size_t up_end = cv.off;
  const size_t o_geo64 = cv.take<double>((size_t)Nx * Q * 4),
               o_geo32 = cv.take<float>((size_t)Nx * Q * 4), o_id64 = cv.take<double>(nJ), o_id32 = cv.take<float>(nJ),
               o_status = cv.take<int>(4), o_rec = cv.take<SolveRecord>(1), o_bar = cv.take<unsigned>(4),
               o_part = cv.take<double>((size_t)16 * m->grid);
  const size_t o_r64 = cv.take<double>(n), o_z64 = cv.take<double>(n64), o_p64a = cv.take<double>(n64),
               o_p64b = cv.take<double>(n64), o_q64 = cv.take<double>(n), o_q64b = cv.take<double>(n),
               o_e64 = cv.take<double>(nE), o_e64b = cv.take<double>(nE);
  const size_t o_d32 = cv.take<float>(n32), o_r32 = cv.take<float>(n32), o_z32 = cv.take<float>(n32),
               o_p32a = cv.take<float>(n32), o_p32b = cv.take<float>(n32), o_q32 = cv.take<float>(n32),
               o_e32 = cv.take<float>(mixed ? nE : 0);
  const size_t o_Phi = cv.take<double>(n), o_qtmp = cv.take<double>(n), o_etmp = cv.take<double>(nE);
  const size_t o_r64b = cv.take<double>(n64), o_r32b = cv.take<float>(n32);
  const size_t o_s64b = cv.take<double>(n64), o_s32b = cv.take<float>(n32);
  const size_t o_uh64 = cv.take<double>(mixed ? 0 : (size_t)m->grid * nrow),
               o_uh32 = cv.take<float>(mixed ? (size_t)m->grid * nrow : 0);
  const size_t nEl = (size_t)nr * Nx, nIf = (size_t)nr * N;
  const size_t o_schur = cv.take<double>(nEl * 3),
               o_A32 = cv.take<float>(nEl * Pm * Pm + 1), o_Z32 = cv.take<float>(nEl * 2 * Pm + 1),
               o_te32 = cv.take<float>(nIf), o_tm32 = cv.take<float>(nIf),
               o_tcp32 = cv.take<float>(nIf), o_tz32 = cv.take<float>(nIf),
               o_tvl32 = cv.take<float>(nr), o_tfac32 = cv.take<float>(nr),
               o_gL32 = cv.take<float>(nEl), o_gR32 = cv.take<float>(nEl), o_zb32 = cv.take<float>(nIf),
               o_rh32 = cv.take<float>((size_t)ncol * nr);
  const size_t o_wave = cv.take<double>(4 * kMaxWaveComp);
  const bool zones = p.relax_left > 0.0 || p.relax_right > 0.0;
  const size_t o_wA = cv.take<double>(zones ? 4 * kMaxWaveComp : 0), o_wEP = cv.take<double>(zones ? 2 * ncol : 0);
  const size_t o_wt = cv.take<double>(ncol), o_etax = cv.take<double>(ncol), o_phisx = cv.take<double>(ncol),
               o_R = cv.take<double>((size_t)2 * Nx * Q), o_R2 = cv.take<double>((size_t)2 * Nx * Q),
               o_ub = cv.take<double>((size_t)2 * (Nx + m->grid + 1)),
               o_ke = cv.take<double>(ncol), o_kp = cv.take<double>(ncol), o_ae = cv.take<double>(ncol),
               o_ap = cv.take<double>(ncol), o_se = cv.take<double>(ncol), o_sp = cv.take<double>(ncol),
               o_etad = cv.take<double>(ncol), o_phisd = cv.take<double>(ncol),
               o_s1e = cv.take<double>(ncol), o_s1p = cv.take<double>(ncol);
  const size_t o_hist = cv.take<int>(8);
  const size_t o_sbar = cv.take<unsigned>(4);
  // written before they are read (the factor cache by every solve, the guess history by the first step of a
  // trajectory, which hist_d[0] = 0 marks): not cleared
  const size_t clear_end = cv.off;
  const size_t o_gglob = cv.take<double>((size_t)3 * Nx * Nz * Q * Q), o_Pl = cv.take<double>(nH),
               o_H = cv.take<float>((size_t)4 * kHist * nH), o_eend = cv.take<double>(ncol), o_pend = cv.take<double>(ncol);
  const size_t total = cv.off + 256;
  if (footprint_only) {
    *footprint_only = total;
    delete m;
    return SEM_OK;
  }
  m->pool_bytes = total;
  cudaError_t ae = dev_alloc(dev, total, reinterpret_cast<void**>(&m->pool));
  if (ae != cudaSuccess) { delete m; return fail(SEM_ERR_OOM, std::string("cudaMalloc: ") + cudaGetErrorString(ae)); }
  auto D_ = [&](size_t o) { return reinterpret_cast<double*>(m->pool + o); };
  auto F_ = [&](size_t o) { return reinterpret_cast<float*>(m->pool + o); };
  int code = SEM_OK;
  // host image of [0, up_end): the arrays are written into it and go up in one copy (zero padding
  // between them); the rest of the block is zeroed on the device
  std::vector<unsigned char> stage(up_end, 0);
  auto up = [&](size_t o, const std::vector<double>& v) {
    if (!v.empty()) std::memcpy(stage.data() + o, v.data(), v.size() * sizeof(double));
  };
  {
    cudaError_t e = cudaMemset(m->pool + up_end, 0, clear_end - up_end);
    if (e != cudaSuccess) code = fail(SEM_ERR_CUDA, std::string("memset: ") + cudaGetErrorString(e));
  }
  up(o_h, std::vector<double>(h_h, h_h + ncol));
  up(o_hx, hx_loc); up(o_dxe, dxe); up(o_dsl, dsl); up(o_sig, sig);
  {
    std::vector<double> cxz((size_t)Nx * Nz * 2);
    for (int e = 0; e < Nx; ++e)
      for (int l = 0; l < Nz; ++l) {
        cxz[((size_t)e * Nz + l) * 2] = dsl[l] / dxe[e];
        cxz[((size_t)e * Nz + l) * 2 + 1] = dxe[e] / dsl[l];
      }
    up(o_cxz, cxz);
    std::vector<double> r2dx(Nx);
    for (int e = 0; e < Nx; ++e) r2dx[e] = 2.0 / dxe[e];
    up(o_r2dx, r2dx);
  }
  up(o_tSX, ct->SX); up(o_tZB, ct->ZB); up(o_tI, I); up(o_tF, F); up(o_twr, wrow);
  up(o_tZ, Z); up(o_tse, se); up(o_tal, th_al); up(o_tm, th_m); up(o_tcp, th_cp);
  up(o_lam, lam);
  {
    std::vector<double> xc(ncol);
    for (int c = 0; c < ncol; ++c) {
      const int e = std::min(c / P, Nx - 1), a = c - e * P;
      xc[c] = x_edges_h[e] + 0.5 * (L.r[a] + 1.0) * dxe[e];
    }
    up(o_xcol, xc);
    m->xcol_h = xc;
  }
  {
    std::vector<float> S32(Sg.begin(), Sg.end()), ST32(S32.size());
    for (int j = 0; j < nr; ++j)
      for (int k = 0; k < nr; ++k) ST32[(size_t)k * nr + j] = S32[(size_t)j * nr + k];
    std::memcpy(stage.data() + o_S32, S32.data(), S32.size() * sizeof(float));
    std::memcpy(stage.data() + o_ST32, ST32.data(), ST32.size() * sizeof(float));
  }
  if (code == SEM_OK) {
    cudaError_t e = cudaMemcpy(m->pool, stage.data(), up_end, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) code = fail(SEM_ERR_CUDA, std::string("upload: ") + cudaGetErrorString(e));
  }
  if (code != SEM_OK) { dev_free(dev, m->pool); delete m; return code; }

  DevGeom& g = m->g;
  g.P = P; g.Nx = Nx; g.Nz = Nz; g.ncol = ncol; g.nrow = nrow; g.periodic = p.periodic ? 1 : 0; g.chunk = chunk;
  g.h = D_(o_h); g.hx_loc = D_(o_hx); g.dxe = D_(o_dxe); g.dsl = D_(o_dsl); g.sig = D_(o_sig); g.cxz = D_(o_cxz);
  g.r2dx = D_(o_r2dx);
  g.geo64 = D_(o_geo64); g.geo32 = F_(o_geo32); g.invdiag64 = D_(o_id64); g.invdiag32 = F_(o_id32);
  g.status = reinterpret_cast<int*>(m->pool + o_status);
  g.gglob = D_(o_gglob);
  g.dv_nrow = FastDiv::make(nrow);
  g.dv_nr = FastDiv::make(nrow - 1);
  g.dv_colsz = FastDiv::make(Q * nrow);
  g.dv_elsz = FastDiv::make(Nz * Q * Q);
  g.dv_qn = FastDiv::make(Q * (nrow - 1));
  g.bar_timeout_ns = kBarrierTimeoutNs;
  g.drop_rank = -1;
  g.trace = nullptr;
#ifdef SEM_TRACE
  if (cudaMalloc(reinterpret_cast<void**>(&g.trace), sizeof(unsigned long long) * (1 + 2 * kTraceMax)) != cudaSuccess ||
      cudaMemset(g.trace, 0, sizeof(unsigned long long)) != cudaSuccess)
    g.trace = nullptr;
#endif
  m->rec = reinterpret_cast<SolveRecord*>(m->pool + o_rec);

  PcgArgs& a = m->pa;
  a.r64 = D_(o_r64); a.z64 = D_(o_z64); a.p64a = D_(o_p64a); a.p64b = D_(o_p64b);
  a.q64 = D_(o_q64); a.q64b = D_(o_q64b); a.edge64 = D_(o_e64); a.edge64b = D_(o_e64b);
  a.d32 = F_(o_d32); a.r32 = F_(o_r32); a.z32 = F_(o_z32); a.p32a = F_(o_p32a); a.p32b = F_(o_p32b);
  a.q32 = F_(o_q32); a.edge32 = F_(o_e32);
  a.part = D_(o_part); a.part_stride = m->grid;
  a.bar = reinterpret_cast<unsigned int*>(m->pool + o_bar);
  a.rec = m->rec;
  a.tol = p.tol; a.inner_rtol = 1e-6; a.max_iter = p.max_iter; a.mixed = mixed;
  a.r64b = D_(o_r64b); a.r32b = F_(o_r32b);
  a.s64b = D_(o_s64b); a.s32b = F_(o_s32b);
  a.uh64 = D_(o_uh64); a.uh32 = F_(o_uh32);
  a.precond = p.precond == SEM_PRECOND_JACOBI ? PREC_JACOBI : PREC_SEPARABLE;
  PrecSetup& ps = m->ps;
  ps.nr = nr; ps.nif = N; ps.lam = D_(o_lam); ps.schur = D_(o_schur);
  ps.Aii32 = F_(o_A32); ps.Z32 = F_(o_Z32); ps.te32 = F_(o_te32); ps.tm32 = F_(o_tm32); ps.tcp32 = F_(o_tcp32);
  ps.tz32 = F_(o_tz32); ps.tvl32 = F_(o_tvl32); ps.tfac32 = F_(o_tfac32);
  ps.v32 = PrecView<float>{nr, N, F_(o_S32), F_(o_ST32), ps.Aii32, ps.Z32, ps.te32, ps.tm32, ps.tcp32, ps.tz32, ps.tvl32,
                           ps.tfac32, F_(o_gL32), F_(o_gR32), F_(o_zb32), F_(o_rh32)};
  a.pv32 = ps.v32;

  m->Phi = D_(o_Phi); m->qtmp = D_(o_qtmp); m->edgetmp = D_(o_etmp);
  m->wt = D_(o_wt); m->etax = D_(o_etax); m->phisx = D_(o_phisx); m->R = D_(o_R); m->R2 = D_(o_R2); m->ub = D_(o_ub);
  m->ke = D_(o_ke); m->kp = D_(o_kp); m->ae = D_(o_ae); m->ap = D_(o_ap); m->se = D_(o_se); m->sp = D_(o_sp);
  m->eta_dev = D_(o_etad); m->phis_dev = D_(o_phisd);
  m->s1e = D_(o_s1e); m->s1p = D_(o_s1p);
  m->Pl = D_(o_Pl); m->H = F_(o_H); m->hist_d = reinterpret_cast<int*>(m->pool + o_hist);
  m->eend = D_(o_eend); m->pend = D_(o_pend);
  m->stage_bars = reinterpret_cast<unsigned int*>(m->pool + o_sbar);

  SurfTables& t = m->st;
  t.P = P; t.Pf = p.Pf; t.Nx = Nx; t.Nz = Nz; t.ncol = ncol; t.nrow = nrow; t.periodic = g.periodic; t.g = p.g;
  t.SX = D_(o_tSX); t.ZB = D_(o_tZB); t.I = D_(o_tI); t.F = D_(o_tF); t.wrow = D_(o_twr);
  t.Z = D_(o_tZ); t.se = D_(o_tse); t.r2dx = g.r2dx; t.h = g.h;
  t.th_al = D_(o_tal); t.th_m = D_(o_tm); t.th_cp = D_(o_tcp); t.win = ct->win; t.nif = N; t.filter_on = (p.filter_ic >= 0 && p.filter_ic < P) ? 1 : 0;
  t.xcol = D_(o_xcol); t.x0 = x_edges_h[0]; t.x1 = x_edges_h[Nx];
  t.relax_left = p.relax_left; t.relax_right = p.relax_right; t.ncomp = 0; t.wave = D_(o_wave);
  t.nzl = 0; t.wkx = nullptr;
  t.wA = zones ? D_(o_wA) : nullptr;
  t.wEP = zones ? D_(o_wEP) : nullptr;
  // the fused RK stage runs this mesh with one team of CTAs (at most its Krylov grid)
  {
    m->stage_smem = stage_smem_bytes(P, nrow, Nz, chunk);
    int per_sm = 0, sms = 0;
    cudaError_t e = stage_occupancy(P, p.precision == SEM_PREC_MIXED, 0, m->stage_smem, &per_sm);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess || per_sm < 1) {
      dev_free(dev, m->pool);
      delete m;
      return fail(SEM_ERR_CUDA, "fused stage kernel does not fit on this device");
    }
    g.sms = sms;
    m->stage_team = std::min(m->grid, per_sm * sms);
    m->stage_smem_batch = m->stage_smem;
    m->own_chunk = chunk;
    // The own launch: all of a CTA's element columns in one pass (instead of passes of `chunk`,
    // each paying its own round trips to L2 and CTA barriers), and room for the solve's
    // geometric factors (3 per element-local node) after the apply's buffers, each if the
    // launch keeps its occupancy.
    {
      const int Qd = P + 1;
      const int ne_max = (Nx + m->stage_team - 1) / m->stage_team;
      int per2 = 0;
      const size_t smem_wide = stage_smem_bytes(P, nrow, Nz, ne_max);
      if (ne_max > chunk && smem_wide <= (size_t)kMaxDynSmem &&
          stage_occupancy(P, mixed, 0, smem_wide, &per2) == cudaSuccess && per2 >= per_sm) {
        m->own_chunk = ne_max;
        m->stage_smem = smem_wide;
      }
      const size_t need = (size_t)3 * ne_max * Nz * Qd * Qd;
      const size_t smem2 = m->stage_smem + need * sizeof(double);
      if (smem2 <= (size_t)kMaxDynSmem &&
          stage_occupancy(P, mixed, 0, smem2, &per2) == cudaSuccess && per2 >= per_sm) {
        m->stage_smem = smem2;
        m->gcache = (int)need;
      }
      // The stand-alone FP64 solve takes two CTAs per SM (128 registers) where that leaves a CTA one element column
      // instead of two, and where the fused launch's shape needs several passes and the element-wise work
      // outweighs the interface systems, which that shape solves faster (their ratio goes with Nz (P+1)³):
      // 5333×4, P = 6 2033 → 1618 µs, 3030×4, P = 8 1831 → 1351, 194×16, P = 8 622 → 499; below the line 10256×2,
      // P = 5 and 10667×8, P = 3 gain 4% and 38095×2, P = 3 would lose 44%.
      m->solve_wide = !mixed && m->grid > m->stage_team &&
                      (Nx <= m->grid || (m->own_chunk < ne_max && Nz * Qd * Qd * Qd >= 640));
    }
  }
  *out = m;
  return SEM_OK;
}

void sem_mesh_destroy(sem_mesh* m) {
  if (!m) return;
  DeviceGuard dg(m->device);
  for (auto& pr : m->events) { cudaEventDestroy(pr.first); cudaEventDestroy(pr.second); }
  for (auto e : m->spare) cudaEventDestroy(e);
  cudaDeviceSynchronize();   // no work of this mesh may still run when its memory is reused
  if (m->wkx) dev_free(m->device, m->wkx);
  dev_free(m->device, m->pool);
  delete m;
}

int sem_mesh_info(const sem_mesh* m, sem_info* info) {
  if (!m || !info) return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  info->n_nodes = m->n;
  info->n_unknowns = (int64_t)m->ncol * (m->nrow - 1);
  info->ncol = m->ncol; info->nrow = m->nrow;
  info->n_elements = m->p.Nx * m->p.Nz;
  info->P = m->p.P; info->Pf = m->Pf; info->Nx = m->p.Nx; info->Nz = m->p.Nz;
  info->periodic = m->p.periodic; info->precision = m->p.precision;
  info->grid_ctas = m->solve_wide ? m->grid : m->stage_team;
  info->stage_ctas = m->stage_team;
  info->device_bytes = (int64_t)m->pool_bytes;
  return SEM_OK;
}

int sem_mesh_l2g(sem_mesh* m, int32_t* l2g_d, void* stream) {
  if (!m || !l2g_d) return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  DeviceGuard dg(m->device);
  CUDA_TRY(launch_l2g(m->g, l2g_d, (cudaStream_t)stream));
  return SEM_OK;
}

int sem_update_geometry(sem_mesh* m, const double* eta_d, void* stream) {
  if (!m || !eta_d) return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  DeviceGuard dg(m->device);
  return do_geometry(m, eta_d, (cudaStream_t)stream);
}

int sem_laplace_apply(sem_mesh* m, const double* x_d, double* y_d, void* stream) {
  if (!m || !x_d || !y_d || x_d == y_d) return fail(SEM_ERR_INVALID_ARG, "bad pointer");
  DeviceGuard dg(m->device);
  const char* k = std::getenv("SEM_APPLY_KERNEL");   // "column": the element-column kernel, else tiled
  cudaError_t e = cudaErrorInvalidValue;
  if (!(k && std::strcmp(k, "column") == 0)) e = launch_apply_tile(0, m->g, x_d, y_d, (cudaStream_t)stream);
  // the element-column kernel when asked for, or when the FP64 tile does not fit in shared memory
  // (largest orders with many layers); the tile launcher checks that before launching anything
  if (e == cudaErrorInvalidValue) e = launch_apply(m->g, x_d, y_d, m->qtmp, m->edgetmp, (cudaStream_t)stream);
  if (e != cudaSuccess) return fail(SEM_ERR_CUDA, std::string("apply: ") + cudaGetErrorString(e));
  return SEM_OK;
}

int sem_laplace_apply_f32(const sem_mesh* m, const float* x_d, float* y_d, void* stream) {
  if (!m || !x_d || !y_d || x_d == y_d) return fail(SEM_ERR_INVALID_ARG, "bad pointer");
  DeviceGuard dg(m->device);
  // "tc": the tensor-core kernel for orders 4..7 (measured slower than the CUDA-core kernels on
  // GB300; kept for comparison); "line", "elem": one of the CUDA-core kernels at every size it serves, for tests
  const char* k = std::getenv("SEM_APPLY_F32");
  const int mode = !k ? 1 : std::strcmp(k, "tc") == 0 ? 3 : std::strcmp(k, "line") == 0 ? 4 : std::strcmp(k, "elem") == 0 ? 5 : 1;
  CUDA_TRY(launch_apply_tile(mode, m->g, x_d, y_d, (cudaStream_t)stream));
  return SEM_OK;
}

int sem_laplace_apply_noalloc(const sem_mesh* m, const double* x_d, double* y_d, void* stream) {
  if (!m || !x_d || !y_d || x_d == y_d) return fail(SEM_ERR_INVALID_ARG, "bad pointer");
  if ((size_t)m->p.Nx * (size_t)m->nrow > kNoAllocEdgeMax)
    return fail(SEM_ERR_INVALID_ARG, "sem_laplace_apply_noalloc: Nx*Nrow = " +
                                         std::to_string((size_t)m->p.Nx * m->nrow) + " exceeds the static scratch of " +
                                         std::to_string(kNoAllocEdgeMax) + " values");
  DeviceGuard dg(m->device);
  CUDA_TRY(launch_apply_noalloc(m->g, x_d, y_d, (cudaStream_t)stream));
  return SEM_OK;
}

int sem_laplace_solve(sem_mesh* m, const double* phis_d, double* Phi_d, sem_solve_stats* st, void* stream) {
  if (!m || !phis_d || !Phi_d) return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  DeviceGuard dg(m->device);
  cudaStream_t s = (cudaStream_t)stream;
  int rc = do_solve(m, phis_d, Phi_d, s);
  if (rc) return rc;
  if (st) {
    SolveRecord r{};
    CUDA_TRY(cudaMemcpyAsync(&r, m->rec, sizeof(r), cudaMemcpyDeviceToHost, s));
    rc = read_status(m, s);
    st->iterations = r.iterations;
    st->refinements = r.refinements;
    st->rel_residual = r.rel_residual;
    return rc;
  }
  return SEM_OK;
}

int sem_recover_gradient(sem_mesh* m, const double* Phi_d, const double* eta_d, const double* phis_d,
                         double* w_surf_d, double* etax_d, double* phisx_d, void* stream) {
  if (!m || !Phi_d || !eta_d || !phis_d || !w_surf_d || !etax_d || !phisx_d)
    return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  DeviceGuard dg(m->device);
  cudaStream_t s = (cudaStream_t)stream;
  // The kernel's blocks store while others still read the state around their own elements: where an output
  // lies over an input or another output, the results are complete before they are copied there.
  const double* in[3] = {Phi_d, eta_d, phis_d};
  const size_t n_in[3] = {(size_t)m->n, (size_t)m->ncol, (size_t)m->ncol}, nc = (size_t)m->ncol;
  double* out[3] = {w_surf_d, etax_d, phisx_d};
  double* tmp[3] = {m->wt, m->etax, m->phisx};
  bool shared = false;
  for (int i = 0; i < 3; ++i) {
    for (int j = 0; j < 3; ++j) shared = shared || overlap(out[i], nc, in[j], n_in[j]);
    for (int j = 0; j < i; ++j) shared = shared || overlap(out[i], nc, out[j], nc);
  }
  if (!shared) {
    CUDA_TRY(launch_recover(m->st, Phi_d, eta_d, phis_d, w_surf_d, etax_d, phisx_d, s));
    return SEM_OK;
  }
  CUDA_TRY(launch_recover(m->st, Phi_d, eta_d, phis_d, tmp[0], tmp[1], tmp[2], s));
  for (int i = 0; i < 3; ++i)
    CUDA_TRY(cudaMemcpyAsync(out[i], tmp[i], nc * sizeof(double), cudaMemcpyDeviceToDevice, s));
  return SEM_OK;
}

int sem_zakharov_rhs(sem_mesh* m, const double* eta_d, const double* phis_d, double t, double* deta_d,
                     double* dphis_d, void* stream) {
  if (!m || !eta_d || !phis_d || !deta_d || !dphis_d) return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  if (has_zones(m) && !(m->p.relax_tau > 0.0))
    return fail(SEM_ERR_INVALID_ARG, "relaxation zones need relax_tau > 0 outside sem_rk4_step");
  DeviceGuard dg(m->device);
  return do_rhs(m, eta_d, phis_d, t, m->p.relax_tau, deta_d, dphis_d, (cudaStream_t)stream);
}

int sem_set_wave_input(sem_mesh* m, int ncomp, const double* amp_h, const double* omega_h,
                       const double* k_h, const double* phase_h) {
  if (!m || ncomp < 0 || ncomp > kMaxWaveComp) return fail(SEM_ERR_INVALID_ARG, "ncomp must be in [0, 4096]");
  if (ncomp > 0 && (!amp_h || !omega_h || !k_h || !phase_h)) return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  for (int i = 0; i < ncomp; ++i)
    if (!(omega_h[i] > 0.0)) return fail(SEM_ERR_INVALID_ARG, "wave frequencies must be positive");
  DeviceGuard dg(m->device);
  double* w = const_cast<double*>(m->st.wave);
  const double* src[4] = {amp_h, omega_h, k_h, phase_h};
  for (int q = 0; q < 4 && ncomp > 0; ++q)
    CUDA_TRY(cudaMemcpy(w + (size_t)q * ncomp, src[q], sizeof(double) * ncomp, cudaMemcpyHostToDevice));
  m->st.ncomp = ncomp;
  // cos, sin of k x at the left-zone columns (the first nzl columns), for the fused stage's
  // angle-addition evaluation; left out when there is no left zone or the table would pass 512 MB
  CUDA_TRY(cudaDeviceSynchronize());
  if (m->wkx) { dev_free(m->device, m->wkx); m->wkx = nullptr; }
  m->st.wkx = nullptr;
  m->st.nzl = 0;
  int nzl = 0;
  if (m->p.relax_left > 0.0)
    while (nzl < m->ncol && m->xcol_h[nzl] < m->st.x0 + m->p.relax_left) ++nzl;
  const size_t entries = (size_t)nzl * (size_t)ncomp * 2;
  if (nzl > 0 && ncomp > 0 && m->st.wA && entries * sizeof(double) <= (size_t(512) << 20)) {
    std::vector<double> tab(entries);
    for (int c = 0; c < nzl; ++c)
      for (int i = 0; i < ncomp; ++i) {
        const double kx = k_h[i] * m->xcol_h[c];
        tab[((size_t)c * ncomp + i) * 2] = std::cos(kx);
        tab[((size_t)c * ncomp + i) * 2 + 1] = std::sin(kx);
      }
    void* d = nullptr;
    cudaError_t e = dev_alloc(m->device, entries * sizeof(double), &d);
    if (e != cudaSuccess) return fail(SEM_ERR_OOM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    m->wkx = static_cast<double*>(d);
    CUDA_TRY(cudaMemcpy(m->wkx, tab.data(), entries * sizeof(double), cudaMemcpyHostToDevice));
    m->st.wkx = m->wkx;
    m->st.nzl = nzl;
  }
  return SEM_OK;
}

int sem_apply_filter(sem_mesh* m, double* q_d, void* stream) {
  if (!m || !q_d) return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  DeviceGuard dg(m->device);
  CUDA_TRY(launch_filter(m->st, q_d, nullptr, (cudaStream_t)stream));
  return SEM_OK;
}

int sem_rk4_step(sem_mesh* m, double* eta_d, double* phis_d, double* t, double dt, int nsteps, void* stream) {
  if (!m || !eta_d || !phis_d || nsteps < 0 || !(dt > 0.0)) return fail(SEM_ERR_INVALID_ARG, "bad argument");
  DeviceGuard dg(m->device);
  cudaStream_t s = (cudaStream_t)stream;
  int rc = do_rk4(m, eta_d, phis_d, t ? *t : 0.0, dt, nsteps, s);
  if (rc) return rc;
  rc = read_status(m, s);
  if (t) *t += nsteps * dt;
  return rc;
}

int sem_rk4_step_host(sem_mesh* m, double* eta_h, double* phis_h, double* t, double dt, int nsteps,
                      void* stream) {
  if (!m || !eta_h || !phis_h || nsteps < 0 || !(dt > 0.0)) return fail(SEM_ERR_INVALID_ARG, "bad argument");
  DeviceGuard dg(m->device);
  cudaStream_t s = (cudaStream_t)stream;
  const size_t bytes = sizeof(double) * m->ncol;
  CUDA_TRY(cudaMemcpyAsync(m->eta_dev, eta_h, bytes, cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemcpyAsync(m->phis_dev, phis_h, bytes, cudaMemcpyHostToDevice, s));
  int rc = do_rk4(m, m->eta_dev, m->phis_dev, t ? *t : 0.0, dt, nsteps, s);
  if (rc) return rc;
  CUDA_TRY(cudaMemcpyAsync(eta_h, m->eta_dev, bytes, cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaMemcpyAsync(phis_h, m->phis_dev, bytes, cudaMemcpyDeviceToHost, s));
  rc = read_status(m, s);
  if (t) *t += nsteps * dt;
  return rc;
}

// Cost of a team's barriers and cross-CTA round trips per stage, in element-local nodes of work
// (team sizing of the cooperative plan).
constexpr double kTeamSyncNodes = 256.0;
// Batch planning parameters (sem_set_batch_tuning; the defaults are the untuned rules).
static std::mutex g_tune_mu;
static sem_batch_tuning g_tune{0.5, 16, 8, -1};

static sem_batch_tuning batch_tuning() {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  return g_tune;
}
// Dynamic shared memory per CTA up to which batch members widen their passes (two CTAs per SM,
// or one).
constexpr size_t kBatchSmemWide = 88 * 1024, kBatchSmemNarrow = 176 * 1024;
// Largest thread-block cluster (the non-portable limit of this architecture).
constexpr int kMaxCluster = 16;

int sem_set_batch_tuning(const sem_batch_tuning* t) {
  sem_batch_tuning v{0.5, 16, 8, -1};
  if (t) {
    if (!(t->cluster_share > 0.0) || t->cluster_share > 64.0 || t->max_cluster < 1 || t->max_cluster > kMaxCluster ||
        (t->max_cluster & (t->max_cluster - 1)) != 0 || t->narrow_max < 0 || t->plan < -1 || t->plan > 1)
      return fail(SEM_ERR_INVALID_ARG, "batch tuning out of range");
    v = *t;
  }
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_tune = v;
  return SEM_OK;
}

int sem_get_batch_tuning(sem_batch_tuning* t) {
  if (!t) return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  *t = batch_tuning();
  return SEM_OK;
}

int sem_set_apply_tile_width(int P, int Nz, int E) {
  if (P < 2 || P > kMaxP || Nz < 1 || Nz > kMaxNz || E < 0 || E > 16)
    return fail(SEM_ERR_INVALID_ARG, "tile width out of range");
  set_apply_tile_width(P, Nz, E);
  return SEM_OK;
}

}  // extern "C"

namespace {

int batch_wide(size_t group_size) {
  const char* wenv = std::getenv("SEM_BATCH_WIDE");
  return wenv ? (std::atoi(wenv) != 0) : (group_size > (size_t)batch_tuning().narrow_max ? 1 : 0);
}

int batch_limit(const sem_mesh* m) {   // ≤ grid: the halo and reduction buffers are sized by it
  return std::max(1, std::min(m->grid, (m->p.Nx + m->g.chunk - 1) / m->g.chunk));
}

// Each member's CTAs take their element columns in as few passes as the launch's shared memory
// allows: a budget per CTA that keeps the build's CTAs per SM.  Returns the launch's dynamic
// shared memory.
size_t widen_passes(BatchLaunch& L, sem_mesh* const* meshes, size_t smem) {
  const size_t budget = L.wide ? kBatchSmemWide : kBatchSmemNarrow;
  size_t smem_l = smem;
  L.chunk.clear();
  for (size_t k = 0; k < L.members.size(); ++k) {
    const sem_mesh* m = meshes[L.members[k]];
    const int ne = (m->p.Nx + L.nteam[k] - 1) / L.nteam[k];
    int E = m->g.chunk;
    while (E < ne && stage_smem_bytes(m->p.P, m->nrow, m->p.Nz, E + 1) <= budget) ++E;
    L.chunk.push_back(E);
    smem_l = std::max(smem_l, stage_smem_bytes(m->p.P, m->nrow, m->p.Nz, E));
  }
  return smem_l;
}

// Cooperative plan: instances grouped by (order, precision), each group split into launches of at
// most the co-resident CTA count; a launch lasts as long as its slowest team, so the CTAs go one at
// a time to the team whose estimated stage time is the largest, while that lowers it (the time of a
// team of c CTAs is taken as w/c element-local nodes per CTA, plus kTeamSyncNodes when c > 1).
int plan_cooperative(sem_batch* b, sem_mesh* const* meshes, int count, int sms) {
  std::vector<std::pair<std::pair<int, int>, std::vector<int>>> groups;
  for (int i = 0; i < count; ++i) {
    const std::pair<int, int> key(meshes[i]->p.P, meshes[i]->p.precision == SEM_PREC_MIXED ? 1 : 0);
    auto it = std::find_if(groups.begin(), groups.end(), [&](const auto& g) { return g.first == key; });
    if (it == groups.end()) groups.push_back({key, {i}});
    else it->second.push_back(i);
  }
  for (auto& grp : groups) {
    size_t smem = 0;
    for (int i : grp.second) smem = std::max(smem, meshes[i]->stage_smem_batch);
    int per_sm = 0;
    // Build of the stage kernel: two CTAs per SM (128 registers) for groups of many instances,
    // where more co-resident teams pay; one CTA per SM with the full register file (the
    // single-mesh build, faster per CTA) for a few instances.  SEM_BATCH_WIDE=0/1 forces either.
    const int wide = batch_wide(grp.second.size());
    cudaError_t e = stage_occupancy(grp.first.first, grp.first.second, wide, smem, &per_sm);
    if (e != cudaSuccess || per_sm < 1) return fail(SEM_ERR_CUDA, "fused stage kernel does not fit");
    const int cap = per_sm * sms;
    for (size_t first = 0; first < grp.second.size(); first += cap) {
      BatchLaunch L;
      L.P = grp.first.first;
      L.mixed = grp.first.second;
      L.wide = wide;
      const size_t last = std::min(grp.second.size(), first + (size_t)cap);
      L.members.assign(grp.second.begin() + first, grp.second.begin() + last);
      std::vector<double> w;
      for (int i : L.members) {
        const sem_mesh* m = meshes[i];
        w.push_back((double)m->p.Nx * m->p.Nz * (m->p.P + 1) * (m->p.P + 1));
      }
      std::vector<int> c(L.members.size(), 1), limit(L.members.size());
      for (size_t k = 0; k < L.members.size(); ++k) limit[k] = batch_limit(meshes[L.members[k]]);
      auto est = [&](size_t k, int ck) { return w[k] / ck + (ck > 1 ? kTeamSyncNodes : 0.0); };
      {
        std::priority_queue<std::pair<double, size_t>> pq;
        for (size_t k = 0; k < c.size(); ++k) pq.push({est(k, 1), k});
        int used = (int)c.size();
        while (used < cap && !pq.empty()) {
          const size_t k = pq.top().second;
          pq.pop();
          if (c[k] >= limit[k] || est(k, c[k] + 1) >= est(k, c[k])) continue;   // this team is done
          ++c[k];
          ++used;
          pq.push({est(k, c[k]), k});
        }
      }
      int acc = 0;
      for (size_t k = 0; k < c.size(); ++k) { L.team0.push_back(acc); L.nteam.push_back(c[k]); acc += c[k]; }
      L.grid = acc;
      size_t smem_l = widen_passes(L, meshes, smem);
      int per2 = 0;
      if (smem_l > smem && (stage_occupancy(L.P, L.mixed, wide, smem_l, &per2) != cudaSuccess || per2 < per_sm)) {
        for (size_t k = 0; k < L.members.size(); ++k) L.chunk[k] = meshes[L.members[k]]->g.chunk;
        smem_l = smem;
      }
      L.smem = smem_l;
      b->launches.push_back(std::move(L));
    }
  }
  return SEM_OK;
}

double member_work(const sem_mesh* m) {
  const int Q = m->p.P + 1;
  return (double)m->p.Nx * m->p.Nz * Q * Q * (8.0 * Q + 7.0);
}

// Estimated stage times of the plans, in units of work (element-local nodes × the apply's flops per node:
// about 2 ns of a CTA).  A CTA's stage costs its share of its tank's work plus its chain of phases and
// barriers, kChainWork (130 µs).  Cluster launches share the GPU: the larger of the sum of that over the CTA
// slots and of the longest team's.  Cooperative launches run one after another, each as long as its slowest
// team plus kCoopWork (80 µs: fewer, larger teams a launch, but launched once per order).  Measured RK4 steps
// of uneven tanks of five orders, ms, with cluster caps of 4 / 8 / 16 and cooperative: 8 tanks – / – / 0.75 / 2.03;
// 30: – / – / 1.65 / 2.39; 100: – / – / 3.84 / 3.24; 200: – / 4.70 / 5.65 / 4.79; 512: 9.67 / 10.27 / 10.85 /
// 10.97 (share 0.25; with the re-measured share of 0.5 the plan takes 0.75, 1.65, 2.66, 4.54 and 9.42).  24 Laplace
// solves of 1e3 to 2e5 nodes, cap 16 against cooperative: 6.69 / 5.59.
constexpr double kChainWork = 6.5e4, kCoopWork = 4.0e4;

// Cluster size of a member: the smallest power of two (≤ cap and its buffer limit) whose work per CTA is at
// most the tuned share of the batch's work per CTA slot.
int cluster_size(const sem_mesh* m, double w, double per_cta, int cap) {
  const int cmax = std::min(cap, batch_limit(m));
  const double want = per_cta > 0.0 ? w / per_cta : 1.0;
  int c = 1;
  while (c < want && 2 * c <= cmax) c *= 2;
  return c;
}

double estimate_clusters(sem_mesh* const* meshes, const std::vector<double>& w, double per_cta, int cap, double slots) {
  double total = 0.0, longest = 0.0;
  for (size_t i = 0; i < w.size(); ++i) {
    const int c = cluster_size(meshes[i], w[i], per_cta, cap);
    total += w[i] + c * kChainWork;
    longest = std::max(longest, w[i] / c + kChainWork);
  }
  return std::max(total / slots, longest);
}

double estimate_cooperative(const sem_batch* b) {
  double t = 0.0;
  for (const auto& L : b->launches) {
    double worst = 0.0;
    for (size_t k = 0; k < L.members.size(); ++k)
      worst = std::max(worst, member_work(b->meshes[L.members[k]]) / L.nteam[k]);
    t += worst + kCoopWork;
  }
  return t;
}

// Cluster plan: each member's team is one thread-block cluster, so no CTA waits on a CTA outside
// its cluster; the launches need no co-residency, the hardware starts clusters as CTA slots free
// up, and the launches of all groups run at the same time on streams of their own.  The largest
// cluster is the one of 4, 8 and 16 CTAs (at most the tuned maximum) with the best estimate: few tanks
// are bound by the longest team, many by the CTA slots, where every further CTA costs its chain.
// Members are grouped by (order, precision, c), the largest first within a launch.  Where some group's cluster
// does not fit on the device, the next best of the three is taken.  Returns false (and builds nothing) when none
// fits; *estimate: its stage time.
bool build_clusters(std::vector<BatchLaunch>* plan, sem_mesh* const* meshes, int count, const std::vector<double>& w,
                    double per_cta, int cap);

bool plan_clusters(std::vector<BatchLaunch>* plan, sem_mesh* const* meshes, int count, int sms,
                   const sem_batch_tuning& tune, double* estimate) {
  std::vector<double> w(count);
  double total = 0.0;
  for (int i = 0; i < count; ++i) {
    w[i] = member_work(meshes[i]);
    total += w[i];
  }
  const double slots = 2.0 * sms;
  const double per_cta = tune.cluster_share * total / slots;
  std::vector<std::pair<double, int>> caps;    // (estimate, cap), the best first
  for (int c = std::min(4, tune.max_cluster); c <= tune.max_cluster; c *= 2)
    caps.emplace_back(estimate_clusters(meshes, w, per_cta, c, slots), c);
  std::sort(caps.begin(), caps.end());
  for (const auto& c : caps)
    if (build_clusters(plan, meshes, count, w, per_cta, c.second)) {
      *estimate = c.first;
      return true;
    }
  return false;
}

bool build_clusters(std::vector<BatchLaunch>* plan, sem_mesh* const* meshes, int count, const std::vector<double>& w,
                    double per_cta, int cap) {
  std::vector<std::pair<std::array<int, 3>, std::vector<int>>> groups;
  for (int i = 0; i < count; ++i) {
    const int c = cluster_size(meshes[i], w[i], per_cta, cap);
    const std::array<int, 3> key{meshes[i]->p.P, meshes[i]->p.precision == SEM_PREC_MIXED ? 1 : 0, c};
    auto it = std::find_if(groups.begin(), groups.end(), [&](const auto& g) { return g.first == key; });
    if (it == groups.end()) groups.push_back({key, {i}});
    else it->second.push_back(i);
  }
  std::vector<BatchLaunch> out;
  for (auto& grp : groups) {
    BatchLaunch L;
    L.P = grp.first[0];
    L.mixed = grp.first[1];
    L.csize = grp.first[2];
    L.wide = batch_wide(grp.second.size());
    L.members = grp.second;
    std::stable_sort(L.members.begin(), L.members.end(), [&](int a, int c) { return w[a] > w[c]; });
    size_t smem = 0;
    for (int i : L.members) smem = std::max(smem, meshes[i]->stage_smem_batch);
    for (size_t k = 0; k < L.members.size(); ++k) {
      L.team0.push_back((int)k * L.csize);
      L.nteam.push_back(L.csize);
    }
    L.grid = (int)L.members.size() * L.csize;
    int fit = 0;
    if (cluster_fit(L.P, L.mixed, L.wide, L.csize, smem, &fit) != cudaSuccess || fit < 1) {
      cudaGetLastError();
      return false;
    }
    size_t smem_l = widen_passes(L, meshes, smem);
    int fit2 = 0;
    if (smem_l > smem && (cluster_fit(L.P, L.mixed, L.wide, L.csize, smem_l, &fit2) != cudaSuccess || fit2 < fit)) {
      cudaGetLastError();
      for (size_t k = 0; k < L.members.size(); ++k) L.chunk[k] = meshes[L.members[k]]->g.chunk;
      smem_l = smem;
    }
    L.smem = smem_l;
    out.push_back(std::move(L));
  }
  *plan = std::move(out);
  return true;
}

// Streams and events of cluster launches are kept per device after a batch is destroyed and
// handed to later batches (the serving loop creates batches every tick).
std::mutex g_sp_mu;
std::vector<std::pair<cudaStream_t, cudaEvent_t>> g_stream_pool[64];

cudaError_t take_stream(int dev, cudaStream_t* st, cudaEvent_t* ev) {
  {
    std::lock_guard<std::mutex> lk(g_sp_mu);
    if (dev >= 0 && dev < 64 && !g_stream_pool[dev].empty()) {
      *st = g_stream_pool[dev].back().first;
      *ev = g_stream_pool[dev].back().second;
      g_stream_pool[dev].pop_back();
      return cudaSuccess;
    }
  }
  cudaError_t e = cudaStreamCreateWithFlags(st, cudaStreamNonBlocking);
  if (e != cudaSuccess) return e;
  return cudaEventCreateWithFlags(ev, cudaEventDisableTiming);
}

void release_plan(std::vector<BatchLaunch>& plan, int dev) {
  std::lock_guard<std::mutex> lk(g_sp_mu);
  for (auto& L : plan) {
    if (L.stream && L.done && dev >= 0 && dev < 64) g_stream_pool[dev].emplace_back(L.stream, L.done);
    L.stream = nullptr;
    L.done = nullptr;
  }
}


// A plan's device arrays (CTA maps, descriptors, barrier words, gathered status) from `pool`; the maps of all
// its launches lie together and go up in one copy (a copy each had cost a server's tick 10 µs a launch).
int carve_plan(int dev, unsigned char* pool, std::vector<BatchLaunch>& plan, size_t& off) {
  const size_t first = off;
  std::vector<int> maps;
  for (auto& L : plan) {
    L.cta_d = reinterpret_cast<int*>(pool + off);
    off += (sizeof(int) * (size_t)L.grid + 255) & ~size_t(255);
    const size_t at = ((unsigned char*)L.cta_d - (pool + first)) / sizeof(int);
    maps.resize((off - first) / sizeof(int), 0);
    for (size_t k = 0; k < L.members.size(); ++k)
      for (int c = 0; c < L.nteam[k]; ++c) maps[at + L.team0[k] + c] = (int)k;
  }
  if (!maps.empty()) CUDA_TRY(cudaMemcpy(pool + first, maps.data(), sizeof(int) * maps.size(), cudaMemcpyHostToDevice));
  for (auto& L : plan) {
    L.inst_d = reinterpret_cast<Instance*>(pool + off);
    off += (sizeof(Instance) * L.members.size() + 255) & ~size_t(255);
    L.bars_d = reinterpret_cast<unsigned int*>(pool + off);
    off += (sizeof(unsigned) * 2 * L.members.size() + 255) & ~size_t(255);
    L.status_d = reinterpret_cast<int*>(pool + off);
    off += (sizeof(int) * L.members.size() + 255) & ~size_t(255);
    L.inst_h.resize(L.members.size());
    L.status_h.resize(L.members.size());
    if (L.csize > 0) CUDA_TRY(take_stream(dev, &L.stream, &L.done));
  }
  return SEM_OK;
}

size_t plan_bytes(const std::vector<BatchLaunch>& plan) {
  size_t total = 0;
  for (const auto& L : plan)
    total += ((sizeof(Instance) * L.members.size() + 255) & ~size_t(255)) +
             ((sizeof(int) * (size_t)L.grid + 255) & ~size_t(255)) +
             ((sizeof(unsigned) * 2 * L.members.size() + 255) & ~size_t(255)) +
             ((sizeof(int) * L.members.size() + 255) & ~size_t(255));
  return total;
}

// The plan of the Laplace solves of a batch whose steps run in clusters.  A solve from a caller's start takes several
// times a stage's iterations between the same fixed phases, so a CTA's chain weighs less and larger teams pay: the
// cluster plan at half the steps' share, or the cooperative one where that is estimated faster.  Solves from zero, ms, on
// the steps' plan / on this one: 512 tanks 6.25 / 5.53 FP64 and 5.48 / 4.93 mixed, 200 3.25 / 2.85, 100 2.28 / 1.74.
// (Steps at half the share: 512 tanks 9.45 → 9.65 ms.)  Without memory for it the steps' plan serves.
void plan_solves(sem_batch* b) {
  b->solve_plan = 1;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device) != cudaSuccess) return;
  sem_batch_tuning tune = b->tune;
  tune.cluster_share *= 0.5;
  std::vector<BatchLaunch> plan;
  double est = 0.0;
  const int count = (int)b->meshes.size();
  if (!plan_clusters(&plan, b->meshes.data(), count, sms, tune, &est)) return;
  if (b->force < 0 && est > estimate_cooperative(b)) {
    b->solve_plan = 0;
    return;
  }
  std::vector<int> size(count);
  for (const auto& L : b->cl_launches)
    for (int i : L.members) size[i] = L.csize;
  bool same = true;
  for (const auto& L : plan)
    for (int i : L.members) same = same && size[i] == L.csize;
  if (same) return;
  size_t off = 0;
  if (dev_alloc(b->device, plan_bytes(plan) + 256, reinterpret_cast<void**>(&b->solve_pool)) != cudaSuccess) {
    cudaGetLastError();
    b->solve_pool = nullptr;
    return;
  }
  if (carve_plan(b->device, b->solve_pool, plan, off) != SEM_OK) {
    release_plan(plan, b->device);
    dev_free(b->device, b->solve_pool);
    b->solve_pool = nullptr;
    return;
  }
  b->cl_solve = std::move(plan);
  b->solve_plan = 2;
}

}  // namespace

extern "C" {

int sem_batch_create(sem_mesh* const* meshes, int count, sem_batch** out) {
  if (!out) return fail(SEM_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (!meshes || count < 1) return fail(SEM_ERR_INVALID_ARG, "empty batch");
  for (int i = 0; i < count; ++i)
    if (!meshes[i]) return fail(SEM_ERR_INVALID_ARG, "NULL mesh in batch");
  const int dev = meshes[0]->device;
  for (int i = 0; i < count; ++i) {
    if (meshes[i]->device != dev) return fail(SEM_ERR_INVALID_ARG, "batch meshes must share one device");
    if (!meshes[i]->fused) return fail(SEM_ERR_INVALID_ARG, "batched meshes need the separable preconditioner");
    for (int j = 0; j < i; ++j)
      if (meshes[j] == meshes[i]) return fail(SEM_ERR_INVALID_ARG, "a mesh appears twice in the batch");
  }
  DeviceGuard dg(dev);
  int sms = 0;
  CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  sem_batch* b = new sem_batch;
  b->device = dev;
  b->meshes.assign(meshes, meshes + count);
  int rc = plan_cooperative(b, meshes, count, sms);
  if (rc) { delete b; return rc; }
  // The cluster plan is kept where it is estimated faster than the cooperative one (it is not
  // when a few large members would need more CTAs than a cluster holds); SEM_BATCH_CLUSTER=0 or 1
  // forces either plan.
  const char* cenv = std::getenv("SEM_BATCH_CLUSTER");
  b->tune = batch_tuning();
  const int force = b->force = cenv ? (std::atoi(cenv) != 0 ? 1 : 0) : b->tune.plan;
  double est = 0.0;
  if (force != 0 && plan_clusters(&b->cl_launches, meshes, count, sms, b->tune, &est) && force < 0 &&
      est > estimate_cooperative(b))
    b->cl_launches.clear();
  for (int i = 0; i < count; ++i) {
    b->off.push_back(b->ncol_total);
    b->ncol_total += (size_t)meshes[i]->ncol;
  }
  const size_t state_bytes = (2 * b->ncol_total * sizeof(double) + 255) & ~size_t(255);
  const size_t total = state_bytes + plan_bytes(b->launches) + plan_bytes(b->cl_launches);
  cudaError_t ae = dev_alloc(dev, total + 256, reinterpret_cast<void**>(&b->pool));
  if (ae != cudaSuccess) { delete b; return fail(SEM_ERR_OOM, std::string("cudaMalloc: ") + cudaGetErrorString(ae)); }
  b->state = reinterpret_cast<double*>(b->pool);
  size_t off = state_bytes;
  rc = carve_plan(dev, b->pool, b->launches, off);
  if (!rc) rc = carve_plan(dev, b->pool, b->cl_launches, off);
  if (!rc && !b->cl_launches.empty() && cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming) != cudaSuccess)
    rc = fail(SEM_ERR_CUDA, "event creation failed");
  if (rc) {
    release_plan(b->cl_launches, dev);
    dev_free(dev, b->pool);
    delete b;
    return rc;
  }
  *out = b;
  return SEM_OK;
}

void sem_batch_destroy(sem_batch* b) {
  if (!b) return;
  DeviceGuard dg(b->device);
  cudaDeviceSynchronize();   // no work of this batch may still run when its memory is reused
  release_plan(b->cl_launches, b->device);
  release_plan(b->cl_solve, b->device);
  if (b->fork) cudaEventDestroy(b->fork);
  for (auto& pr : b->events) { cudaEventDestroy(pr.first); cudaEventDestroy(pr.second); }
  for (cudaEvent_t e : b->spare) cudaEventDestroy(e);
  if (b->solve_pool) dev_free(b->device, b->solve_pool);
  dev_free(b->device, b->pool);
  delete b;
}

void sem_trim_cache(void) {
  std::lock_guard<std::mutex> lk(g_cache_mu);
  int prev = -1;
  cudaGetDevice(&prev);
  for (int d = 0; d < 64; ++d) {
    BlockCache& c = g_cache[d];
    if (c.free.empty()) continue;
    cudaSetDevice(d);
    for (auto& kv : c.free) {
      cudaFree(kv.second);
      c.size_of.erase(kv.second);
    }
    c.free.clear();
    c.cached = 0;
  }
  if (prev >= 0) cudaSetDevice(prev);
}

int sem_batch_info(const sem_batch* b, int* launches_per_stage, int* ctas) {
  if (!b) return fail(SEM_ERR_INVALID_ARG, "NULL batch");
  const auto& plan = b->cl_launches.empty() ? b->launches : b->cl_launches;
  int tot = 0;
  for (const auto& L : plan) tot += L.grid;
  if (launches_per_stage) *launches_per_stage = (int)plan.size();
  if (ctas) *ctas = tot;
  return SEM_OK;
}

}  // extern "C"

namespace {
int batch_status(sem_batch* b, std::vector<BatchLaunch>& plan, cudaStream_t s);

// The cluster plan serves a call unless a member carries the barrier testing hook, whose early
// CTA exit only the cooperative launches' bounded barriers turn into an error.
bool use_clusters(const sem_batch* b) {
  if (b->cl_launches.empty()) return false;
  for (const sem_mesh* m : b->meshes)
    if (m->g.drop_rank >= 0 || m->g.bar_timeout_ns != kBarrierTimeoutNs) return false;
  return true;
}

cudaError_t take_batch_event(sem_batch* b, cudaEvent_t* ev) {
  if (!b->spare.empty()) { *ev = b->spare.back(); b->spare.pop_back(); return cudaSuccess; }
  return cudaEventCreate(ev);
}

// One stage launch of a batch group on stream s, bracketed by events while timing is on.
cudaError_t batch_launch(sem_batch* b, const BatchLaunch& L, const StageArgs& a, cudaStream_t s) {
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t e;
  if (b->timing) {
    if ((e = take_batch_event(b, &e0)) != cudaSuccess) return e;
    if ((e = take_batch_event(b, &e1)) != cudaSuccess) return e;
    if ((e = cudaEventRecord(e0, s)) != cudaSuccess) return e;
  }
  if (L.csize > 0) e = launch_stage_cluster(L.P, L.mixed, L.wide, a, L.grid, L.csize, L.smem, s);
  else e = launch_stage(L.P, L.mixed, L.wide, a, L.grid, L.smem, s);
  if (e != cudaSuccess) return e;
  if (b->timing) {
    if ((e = cudaEventRecord(e1, s)) != cudaSuccess) return e;
    b->events.emplace_back(e0, e1);
  }
  return cudaSuccess;
}

// A cluster plan: each group's stage launches in order on the group's own stream, the streams
// forked from and joined back to s.  stage 0: the Laplace solve alone; else nsteps RK4 steps.
cudaError_t run_clusters(sem_batch* b, std::vector<BatchLaunch>& plan, int stage, int nsteps, cudaStream_t s) {
  cudaError_t e;
  if ((e = cudaEventRecord(b->fork, s)) != cudaSuccess) return e;
  for (auto& L : plan)
    if ((e = cudaStreamWaitEvent(L.stream, b->fork, 0)) != cudaSuccess) return e;
  for (int step = 0; step < (stage == 0 ? 1 : nsteps); ++step)
    for (int st = (stage == 0 ? 0 : 1); st <= (stage == 0 ? 0 : 4); ++st)
      for (auto& L : plan) {
        const StageArgs a{L.inst_d, L.cta_d, nullptr, st, step, 1, {}};
        if ((e = batch_launch(b, L, a, L.stream)) != cudaSuccess) return e;
      }
  for (auto& L : plan) {
    if ((e = cudaEventRecord(L.done, L.stream)) != cudaSuccess) return e;
    if ((e = cudaStreamWaitEvent(s, L.done, 0)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}
}  // namespace

extern "C" {

int sem_batch_rk4_step(sem_batch* b, double* const* eta_d, double* const* phis_d, double* t_h, const double* dt_h,
                       int nsteps, void* stream) {
  if (!b || !eta_d || !phis_d || !dt_h || nsteps < 0) return fail(SEM_ERR_INVALID_ARG, "bad argument");
  const int n = (int)b->meshes.size();
  for (int i = 0; i < n; ++i)
    if (!eta_d[i] || !phis_d[i] || !(dt_h[i] > 0.0)) return fail(SEM_ERR_INVALID_ARG, "bad instance state");
  DeviceGuard dg(b->device);
  cudaStream_t s = (cudaStream_t)stream;
  const bool cl = use_clusters(b);
  auto& plan = cl ? b->cl_launches : b->launches;
  for (auto& L : plan) {
    for (size_t k = 0; k < L.members.size(); ++k) {
      const int i = L.members[k];
      L.inst_h[k] = make_instance(b->meshes[i], eta_d[i], phis_d[i], t_h ? t_h[i] : 0.0, dt_h[i], L.team0[k],
                                  L.nteam[k], false, L.chunk[k]);
    }
    CUDA_TRY(cudaMemcpyAsync(L.inst_d, L.inst_h.data(), sizeof(Instance) * L.members.size(),
                             cudaMemcpyHostToDevice, s));
  }
  if (cl) {
    if (nsteps > 0) CUDA_TRY(run_clusters(b, plan, 1, nsteps, s));
  } else {
    for (int step = 0; step < nsteps; ++step)
      for (int stage = 1; stage <= 4; ++stage)
        for (auto& L : plan) {
          CUDA_TRY(cudaMemsetAsync(L.bars_d, 0, 2 * sizeof(unsigned int) * L.members.size(), s));
          const StageArgs a{L.inst_d, L.cta_d, L.bars_d, stage, step, 0, {}};
          CUDA_TRY(batch_launch(b, L, a, s));
        }
  }
  if (nsteps > 0)
    for (int i = 0; i < n; ++i) b->meshes[i]->hist_dt = dt_h[i];
  int rc = batch_status(b, plan, s);
  if (t_h)
    for (int i = 0; i < n; ++i) t_h[i] += nsteps * dt_h[i];
  return rc;
}

int sem_batch_laplace_solve(sem_batch* b, const double* const* eta_d, const double* const* phis_d,
                            double* const* Phi_d, void* stream) {
  if (!b || !eta_d || !phis_d || !Phi_d) return fail(SEM_ERR_INVALID_ARG, "bad argument");
  const int n = (int)b->meshes.size();
  for (int i = 0; i < n; ++i)
    if (!eta_d[i] || !phis_d[i] || !Phi_d[i]) return fail(SEM_ERR_INVALID_ARG, "bad instance state");
  DeviceGuard dg(b->device);
  cudaStream_t s = (cudaStream_t)stream;
  bool cl = use_clusters(b);
  if (cl && b->solve_plan < 0) plan_solves(b);
  cl = cl && b->solve_plan != 0;
  auto& plan = !cl ? b->launches : b->solve_plan == 2 ? b->cl_solve : b->cl_launches;
  for (auto& L : plan) {
    for (size_t k = 0; k < L.members.size(); ++k) {
      const int i = L.members[k];
      L.inst_h[k] = make_instance(b->meshes[i], const_cast<double*>(eta_d[i]), const_cast<double*>(phis_d[i]),
                                  0.0, 1.0, L.team0[k], L.nteam[k], false, L.chunk[k]);
      L.inst_h[k].pa.x = Phi_d[i];
    }
    CUDA_TRY(cudaMemcpyAsync(L.inst_d, L.inst_h.data(), sizeof(Instance) * L.members.size(),
                             cudaMemcpyHostToDevice, s));
  }
  if (cl) {
    CUDA_TRY(run_clusters(b, plan, 0, 0, s));
  } else {
    for (auto& L : plan) {
      CUDA_TRY(cudaMemsetAsync(L.bars_d, 0, 2 * sizeof(unsigned int) * L.members.size(), s));
      const StageArgs a{L.inst_d, L.cta_d, L.bars_d, 0, 0, 0, {}};
      CUDA_TRY(batch_launch(b, L, a, s));
    }
  }
  return batch_status(b, plan, s);
}

int sem_batch_rk4_step_host(sem_batch* b, double* eta_h, double* phis_h, double* t_h, const double* dt_h,
                            int nsteps, void* stream) {
  if (!b || !eta_h || !phis_h || !dt_h || nsteps < 0) return fail(SEM_ERR_INVALID_ARG, "bad argument");
  DeviceGuard dg(b->device);
  cudaStream_t s = (cudaStream_t)stream;
  const size_t n = b->meshes.size(), bytes = sizeof(double) * b->ncol_total;
  double* eta_d = b->state;
  double* phis_d = b->state + b->ncol_total;
  CUDA_TRY(cudaMemcpyAsync(eta_d, eta_h, bytes, cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemcpyAsync(phis_d, phis_h, bytes, cudaMemcpyHostToDevice, s));
  std::vector<double*> ep(n), pp(n);
  for (size_t i = 0; i < n; ++i) { ep[i] = eta_d + b->off[i]; pp[i] = phis_d + b->off[i]; }
  const int rc = sem_batch_rk4_step(b, ep.data(), pp.data(), t_h, dt_h, nsteps, stream);
  if (rc != SEM_OK && rc != SEM_ERR_NOT_CONVERGED && rc != SEM_ERR_NONFINITE && rc != SEM_ERR_TIMEOUT) return rc;
  // every member's state comes back, failed members' included (their codes say which)
  const std::string err = t_err;
  CUDA_TRY(cudaMemcpyAsync(eta_h, eta_d, bytes, cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaMemcpyAsync(phis_h, phis_d, bytes, cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  if (rc != SEM_OK) t_err = err;
  return rc;
}

int sem_batch_enable_timing(sem_batch* b, int on) {
  if (!b) return fail(SEM_ERR_INVALID_ARG, "NULL batch");
  b->timing = on != 0;
  return SEM_OK;
}

int sem_batch_get_timing(sem_batch* b, sem_timing* t) {
  if (!b || !t) return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  DeviceGuard dg(b->device);
  double total = 0.0;
  for (auto& pr : b->events) {
    CUDA_TRY(cudaEventSynchronize(pr.second));
    float ms = 0.f;
    CUDA_TRY(cudaEventElapsedTime(&ms, pr.first, pr.second));
    total += ms;
    b->spare.push_back(pr.first);
    b->spare.push_back(pr.second);
  }
  t->krylov_launches = (int64_t)b->events.size();
  t->krylov_ms = total;
  b->events.clear();
  return SEM_OK;
}

}  // extern "C"

namespace {
// One gather of every member's status word and one copy per launch group; returns the
// first failing instance's error.
int batch_status(sem_batch* b, std::vector<BatchLaunch>& plan, cudaStream_t s) {
  const int n = (int)b->meshes.size();
  for (auto& L : plan) {
    CUDA_TRY(launch_gather_status(L.inst_d, (int)L.members.size(), L.status_d, s));
    CUDA_TRY(cudaMemcpyAsync(L.status_h.data(), L.status_d, sizeof(int) * L.members.size(),
                             cudaMemcpyDeviceToHost, s));
  }
  CUDA_TRY(cudaStreamSynchronize(s));
  int rc = SEM_OK, first = n;
  b->codes.assign(n, SEM_OK);
  for (const auto& L : plan)
    for (size_t k = 0; k < L.members.size(); ++k) {
      b->codes[L.members[k]] = status_code(L.status_h[k]);
      if (L.status_h[k] && L.members[k] < first) {
        first = L.members[k];
        rc = L.status_h[k];
      }
    }
  if (rc != SEM_OK) {
    for (int i = 0; i < n; ++i)
      if (b->codes[i] != SEM_OK) CUDA_TRY(reset_warm_start(b->meshes[i], s));
    CUDA_TRY(cudaStreamSynchronize(s));
    rc = status_error(rc);
    t_err = "instance " + std::to_string(first) + ": " + t_err;
  }
  return rc;
}
}  // namespace

extern "C" {

int sem_batch_status(const sem_batch* b, int* codes_h) {
  if (!b || !codes_h) return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  for (size_t i = 0; i < b->meshes.size(); ++i) codes_h[i] = i < b->codes.size() ? b->codes[i] : SEM_OK;
  return SEM_OK;
}

int sem_get_counters(sem_mesh* m, sem_counters* c, void* stream) {
  if (!m || !c) return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  DeviceGuard dg(m->device);
  cudaStream_t s = (cudaStream_t)stream;
  SolveRecord r{};
  CUDA_TRY(cudaMemcpyAsync(&r, m->rec, sizeof(r), cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  c->solves = r.solves;
  c->iterations = r.total_iterations;
  c->refinements = r.total_refinements;
  c->max_rel_residual = r.max_rel_residual;
  return SEM_OK;
}

int sem_enable_timing(sem_mesh* m, int on) {
  if (!m) return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  m->timing = on != 0;
  return SEM_OK;
}

int sem_get_timing(sem_mesh* m, sem_timing* t) {
  if (!m || !t) return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  DeviceGuard dg(m->device);
  double total = 0.0;
  for (auto& pr : m->events) {
    CUDA_TRY(cudaEventSynchronize(pr.second));
    float ms = 0.f;
    CUDA_TRY(cudaEventElapsedTime(&ms, pr.first, pr.second));
    total += ms;
    m->spare.push_back(pr.first);
    m->spare.push_back(pr.second);
  }
  t->krylov_launches = (int64_t)m->events.size();
  t->krylov_ms = total;
  m->events.clear();
  return SEM_OK;
}

#ifdef SEM_TRACE
// Diagnostic builds only (not part of sem.h): copies the phase trace of the mesh's last launches
// ([0] = marks, then (tag, ns) pairs) to out_h and clears it.
int sem_trace_read(sem_mesh* m, unsigned long long* out_h, int max_words) {
  if (!m || !out_h || !m->g.trace) return fail(SEM_ERR_INVALID_ARG, "no trace");
  DeviceGuard dg(m->device);
  CUDA_TRY(cudaDeviceSynchronize());
  const int words = std::min(max_words, 1 + 2 * kTraceMax);
  CUDA_TRY(cudaMemcpy(out_h, m->g.trace, sizeof(unsigned long long) * words, cudaMemcpyDeviceToHost));
  CUDA_TRY(cudaMemset(m->g.trace, 0, sizeof(unsigned long long)));
  return SEM_OK;
}
#endif

int sem_set_barrier_test(sem_mesh* m, int drop_rank, double timeout_ms) {
  if (!m) return fail(SEM_ERR_INVALID_ARG, "NULL mesh");
  if (drop_rank < -1) return fail(SEM_ERR_INVALID_ARG, "drop_rank must be -1 or a team rank");
  if (!(timeout_ms >= 0.0) || timeout_ms > 1e-6 * (double)kBarrierTimeoutNs)
    return fail(SEM_ERR_INVALID_ARG, "timeout_ms must be in [0, 2000]");
  m->g.drop_rank = drop_rank;
  m->g.bar_timeout_ns = timeout_ms > 0.0 ? (unsigned long long)(timeout_ms * 1e6) : kBarrierTimeoutNs;
  return SEM_OK;
}

int sem_reset_counters(sem_mesh* m, void* stream) {
  if (!m) return fail(SEM_ERR_INVALID_ARG, "NULL argument");
  DeviceGuard dg(m->device);
  CUDA_TRY(cudaMemsetAsync(m->rec, 0, sizeof(SolveRecord), (cudaStream_t)stream));
  return SEM_OK;
}

}  // extern "C"
