// Batched ensembles of independent 2D EREM problems (declared in
// include/erem.h): member contexts, the member table the batched kernel
// reads, the divided-difference tables of every substep level, the queue
// order of a run and the cluster-size autotuner.
//
// Each member is a full context (erem_create / erem_set_state build its
// Jacobian, its Leja copy of J and its spectral interval exactly as for a
// single problem); the batched kernel (ensemble_cluster.cu) then runs every
// member on one thread-block cluster, using the member's own buffers.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <queue>
#include <string>
#include <thread>
#include <vector>

#include "erem_internal.h"

using namespace erem;

// One launch of a run: `count` members of the queue order from `first`, on
// clusters of cs CTAs, with the members' working sets in shared memory (res)
// or in L2.
struct EnsLaunch {
  bool res = false;
  int cs = 0, clusters = 0, first = 0, count = 0;
  bool operator==(const EnsLaunch& o) const {
    return res == o.res && cs == o.cs && clusters == o.clusters && first == o.first && count == o.count;
  }
};

// How a run's members are split into launches: class k (the smallest cluster a
// member fits on has 2 << k CTAs; 4: none) of [from, to) share one, and what the
// split was made for.
struct EnsPlan {
  struct Part {
    int from = 0, to = 0, cs = 0;
    bool res = false;
  };
  bool made = false;
  int max_clusters = 0;
  std::vector<int> cls;
  std::vector<double> rate;   // passes per step of each member
  std::vector<Part> parts;    // the largest classes first
};

struct erem_ens {
  int n = 0;
  erem_precision prec = EREM_FP64;
  std::vector<erem_ctx*> ctx;
  std::vector<char> ready;
  std::vector<double> dt;
  std::string err;

  // Leja options and batching configuration
  double tol_a = 1e-6, tol_r = 1e-6;
  int p_order = 2, m_max = 150, max_doublings = 6, avg_window = 5;
  erem_ens_config cfg{EREM_ENS_KEEP_SUBSTEPS, 0, 0, 0};
  int tuned_cs = 0;

  // divided differences of every member and level (host copy, reused by
  // rebuilds until a member or the options change)
  std::vector<double> dd_host;
  bool dd_valid = false;

  // batch tables (valid while built)
  bool built = false;
  int nlev = 7;
  std::vector<int> level_start;     // KEEP policy: first level of each member's next step
  std::vector<double> pass_rate;    // passes per step of each member's last run (0: none yet)
  EnsMember* mem_d = nullptr;
  EnsState* st_d = nullptr;
  EnsState* st_h = nullptr;         // pinned
  double* dd_d = nullptr;
  double* xi_d = nullptr;
  int* order_d = nullptr;
  int* order_h = nullptr;           // pinned
  unsigned* next_d = nullptr;       // queue position
  double* snap_d = nullptr;         // autotuner: saved temperatures
  double* stage_d = nullptr;        // host-pointer staging (largest member)
  cudaEvent_t ev[2] = {nullptr, nullptr};

  // the run as a CUDA graph (state and queue upload, the persistent launches,
  // state read-back), captured once per run descriptor and cluster shape
  cudaStream_t cap_stream = nullptr;
  cudaGraphExec_t run_exec = nullptr;
  EnsRun run_key{};
  std::vector<EnsLaunch> key_launches;
  std::vector<EnsLaunch> launches;   // of the next run
  EnsPlan plan;
  bool resident_ok = true;           // false: every member works from L2
  int fit_res[5] = {-1, -1, -1, -1, -1}, fit_l2[5] = {-1, -1, -1, -1, -1};   // clusters of 1 << k CTAs at once
  bool graph_ok = true;             // false after a failed capture: direct launches

  // statistics of the last run
  erem_ens_run_stats rs{};
  std::vector<EnsState> last;
};

namespace {

constexpr int kEnsLaunches = 8;   // launches of a run, at most

erem_status efail(erem_ens* E, erem_status st, const std::string& m) {
  if (E) E->err = m;
  return st;
}

#define ENS_CUDA(E, call)                                                                  \
  do {                                                                                     \
    cudaError_t e_ = (call);                                                               \
    if (e_ != cudaSuccess)                                                                 \
      return efail((E), EREM_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_));   \
  } while (0)

#define ENS_TRY(expr)               \
  do {                              \
    erem_status st_ = (expr);       \
    if (st_ != EREM_OK) return st_; \
  } while (0)

template <typename T>
erem_status ens_alloc(erem_ens* E, T** p, size_t count) {
  if (cudaMalloc((void**)p, std::max<size_t>(count, 1) * sizeof(T)) != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return efail(E, EREM_ENOMEM, "cudaMalloc of the ensemble tables failed");
  }
  ENS_CUDA(E, cudaMemset(*p, 0, std::max<size_t>(count, 1) * sizeof(T)));
  return EREM_OK;
}

void drop_graph(erem_ens* E) {
  if (E->run_exec) cudaGraphExecDestroy(E->run_exec);
  E->run_exec = nullptr;
}

void release_tables(erem_ens* E) {
  drop_graph(E);
  void* dp[] = {E->mem_d, E->st_d, E->dd_d, E->xi_d, E->order_d, E->next_d};
  for (void* p : dp)
    if (p) cudaFree(p);
  E->mem_d = nullptr;
  E->st_d = nullptr;
  E->dd_d = nullptr;
  E->xi_d = nullptr;
  E->order_d = nullptr;
  E->next_d = nullptr;
  if (E->st_h) cudaFreeHost(E->st_h);
  if (E->order_h) cudaFreeHost(E->order_h);
  E->st_h = nullptr;
  E->order_h = nullptr;
  E->built = false;
}

bool is_device(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Divided differences of every member and substep level, on host threads:
// table (e, l) holds d_0..d_mmax for the interval of dt J / 2^l.
erem_status build_dd(erem_ens* E, const std::vector<double>& xi, std::vector<double>* dd) {
  const int M = E->m_max, nl = kEnsMaxLevels;
  dd->assign((size_t)E->n * nl * (M + 1), 0.0);
  std::atomic<int> next{0}, bad{-1};
  auto work = [&]() {
    for (int job = next++; job < E->n * E->nlev; job = next++) {
      const int e = job / E->nlev, l = job % E->nlev;
      const erem_ctx* c = E->ctx[e];
      const double S = (double)(1 << l);
      double* d = dd->data() + ((size_t)e * nl + l) * (M + 1);
      if (divided_differences(M, xi.data(), c->cfoc / S, c->gam / S, d) != 0) {
        bad = e;
        continue;
      }
      for (int k = 0; k <= M; ++k)
        if (!std::isfinite(d[k])) bad = e;
    }
  };
  const int nt = std::max(1, std::min<int>(32, (int)std::thread::hardware_concurrency()));
  std::vector<std::thread> pool;
  for (int t = 1; t < nt; ++t) pool.emplace_back(work);
  work();
  for (auto& t : pool) t.join();
  if (bad >= 0)
    return efail(E, EREM_ENONFINITE,
                 "divided differences of member " + std::to_string(bad.load()) + " are not finite");
  return EREM_OK;
}

// Passes one step of a member may take at most: every level's substeps,
// each with m_max terms, the term pass that follows the decision, and its
// start and bookkeeping passes.
long long passes_per_step(const erem_ens* E) {
  long long per_step = 2;
  for (int l = 0; l < E->nlev; ++l) per_step += (1LL << l) * (E->m_max + 3) + 2;
  return per_step;
}

// Member table, divided differences and queue for the current options.
erem_status build(erem_ens* E) {
  for (int e = 0; e < E->n; ++e)
    if (!E->ready[e])
      return efail(E, EREM_EINVAL, "member " + std::to_string(e) + " has no state (erem_ensemble_set_member)");
  release_tables(E);
  E->nlev = E->max_doublings + 1;
  const int M = E->m_max;
  std::vector<double> xi;
  leja_table(M, &xi);
  if (!E->dd_valid) {
    ENS_TRY(build_dd(E, xi, &E->dd_host));
    E->dd_valid = true;
  }
  const std::vector<double>& dd = E->dd_host;

  ENS_TRY(ens_alloc(E, &E->mem_d, (size_t)E->n));
  ENS_TRY(ens_alloc(E, &E->st_d, (size_t)E->n));
  ENS_TRY(ens_alloc(E, &E->dd_d, dd.size()));
  ENS_TRY(ens_alloc(E, &E->xi_d, (size_t)M + 1));
  ENS_TRY(ens_alloc(E, &E->order_d, (size_t)E->n));
  ENS_TRY(ens_alloc(E, &E->next_d, (size_t)kEnsLaunches));
  if (cudaMallocHost((void**)&E->st_h, sizeof(EnsState) * E->n) != cudaSuccess ||
      cudaMallocHost((void**)&E->order_h, sizeof(int) * E->n) != cudaSuccess)
    return efail(E, EREM_ENOMEM, "cudaMallocHost of the ensemble tables failed");
  std::memset(E->st_h, 0, sizeof(EnsState) * E->n);

  std::vector<EnsMember> mem(E->n);
  for (int e = 0; e < E->n; ++e) {
    const erem_ctx* c = E->ctx[e];
    EnsMember& m = mem[e];
    std::memset(&m, 0, sizeof(m));
    m.nx = c->nx;
    m.ny = c->ny;
    m.px = c->px;
    m.Np = (int)c->Np;
    for (int k = 0; k < 5; ++k) m.jc[k] = c->jc[k];
    m.b0 = c->b0;
    m.jl = c->jl_all;
    m.r0 = c->jl_nodiag ? c->jl_r0 : nullptr;
    m.T = c->Tn;
    m.G = c->vrhs;
    m.w = c->w;
    m.P = c->P;
    m.q[0] = c->q[0];
    m.q[1] = c->q[1];
    m.dd = E->dd_d + (size_t)e * kEnsMaxLevels * (M + 1);
    m.sp.delta = E->dt[e];
    m.sp.ncells = (double)c->N;
    m.sp.pow10 = std::pow(10.0, E->p_order);
    m.sp.tol_a = E->tol_a;
    m.sp.tol_r = E->tol_r;
    m.sp.window = E->avg_window;
    m.sp.m_max = E->m_max;
    m.sp.replay = 0;
    m.dt = E->dt[e];
    m.cg = c->cfoc / c->gam;
    m.rsqrt_n = 1.0 / std::sqrt((double)c->N);
  }
  ENS_CUDA(E, cudaMemcpy(E->mem_d, mem.data(), sizeof(EnsMember) * E->n, cudaMemcpyHostToDevice));
  ENS_CUDA(E, cudaMemcpy(E->dd_d, dd.data(), sizeof(double) * dd.size(), cudaMemcpyHostToDevice));
  ENS_CUDA(E, cudaMemcpy(E->xi_d, xi.data(), sizeof(double) * (M + 1), cudaMemcpyHostToDevice));
  E->built = true;
  return EREM_OK;
}

// Work estimate of member e for the queue order: its passes per step (from
// its last run, else the width of its spectral interval as a proxy for the
// Leja degree) times its cells plus a latency term of a pass.
double member_weight(const erem_ens* E, int e) {
  const erem_ctx* c = E->ctx[e];
  const double rate = E->pass_rate[e] > 0.0 ? E->pass_rate[e] : 1.0 + c->gam;
  return rate * ((double)c->Np + 16384.0);
}

// Clusters of cs CTAs that run at once (0: none).
int fit_clusters(erem_ens* E, int cs, bool res) {
  int k = 0;
  while ((1 << k) < cs) ++k;
  int& f = res ? E->fit_res[k] : E->fit_l2[k];
  if (f < 0) {
    const cudaError_t e = res ? ens_res_max_clusters(E->prec, cs, E->ctx[0]->smem_optin, &f)
                              : ens_max_clusters(E->prec, cs, &f);
    if (e != cudaSuccess) {
      cudaGetLastError();
      f = 0;
    }
  }
  return E->cfg.max_clusters > 0 ? std::min(f, E->cfg.max_clusters) : f;
}

bool fits_resident(const erem_ens* E, int e, int cs) {
  const erem_ctx* c = E->ctx[e];
  return E->resident_ok && ens_res_fits(E->prec, cs, c->ny, c->px, c->jl_nodiag, c->smem_optin);
}

// Passes per step of member e: of its last run, else the width of its
// spectral interval as a proxy for the Leja degree.
double member_rate(const erem_ens* E, int e) {
  return E->pass_rate[e] > 0.0 ? E->pass_rate[e] : 1.0 + E->ctx[e]->gam;
}

// Time of one pass of member e on cs CTAs, us, measured on 64^2 to 480^2
// members and clusters of 2 to 16.  In shared memory: the barrier and the
// control step, then the band's vectors (FP64 pipe: one operation per cell in
// FP32-bulk, eight in FP64).  From L2: the same, then the load latency of the
// sweep.
double pass_time(const erem_ens* E, int e, int cs, bool res) {
  const erem_ctx* c = E->ctx[e];
  const bool f32 = E->prec == EREM_FP32_BULK;
  const double nvb = (double)((c->ny + cs - 1) / cs) * (c->px / (f32 ? 4 : 2));
  if (res) return f32 ? 2.5 + 0.00085 * nvb : 2.7 + 0.0036 * nvb;
  return f32 ? 4.0 + 0.0032 * nvb : 5.0 + 0.0043 * nvb;
}

// Time of the given members in one launch: the queue played through, heaviest
// first over the clusters that run at once, and from L2 at least the rate of
// the whole chip (110 cells per ns in FP32-bulk, 41 in FP64).
double launch_time(erem_ens* E, const std::vector<int>& who, int cs, bool res) {
  const int slots = fit_clusters(E, cs, res);
  if (slots < 1) return 1e300;
  double cells = 0.0;
  std::vector<double> t(who.size());
  for (size_t k = 0; k < who.size(); ++k) {
    const double r = member_rate(E, who[k]);
    t[k] = r * pass_time(E, who[k], cs, res);
    cells += r * (double)E->ctx[who[k]]->Np;
  }
  std::sort(t.begin(), t.end(), std::greater<double>());
  std::priority_queue<double, std::vector<double>, std::greater<double>> busy;
  double end = 0.0;
  for (size_t k = 0; k < t.size(); ++k) {
    double at = 0.0;
    if ((int)k >= slots) {
      at = busy.top();
      busy.pop();
    }
    busy.push(at + t[k]);
    end = std::max(end, at + t[k]);
  }
  return res ? end : std::max(end, cells / (E->prec == EREM_FP32_BULK ? 110e3 : 41e3));
}

// Whether the plan was made for members like these: the same classes and limit,
// and no member's passes per step off by more than a quarter (the plan has to
// promise a fifth before it is taken at all).  Playing the queues of all
// candidates takes about 1.5 us per member (0.75 ms for 512, as long as a short
// run's own work); this and the queue order take 0.05 ms.
bool plan_holds(const erem_ens* E, const std::vector<int>& cls) {
  const EnsPlan& p = E->plan;
  if (!p.made || p.max_clusters != E->cfg.max_clusters || p.cls != cls) return false;
  for (int e = 0; e < E->n; ++e) {
    const double r = member_rate(E, e);
    if (!(r <= 1.25 * p.rate[e] && p.rate[e] <= 1.25 * r)) return false;
  }
  return true;
}

// Neighbouring classes share a launch, and each launch takes the form (shared
// memory or L2) and the cluster size by which the whole run is shortest.
erem_status make_plan(erem_ens* E, const std::vector<int>& cls) {
  EnsPlan& p = E->plan;
  p.made = false;
  p.max_clusters = E->cfg.max_clusters;
  p.cls = cls;
  p.rate.resize(E->n);
  for (int e = 0; e < E->n; ++e) p.rate[e] = member_rate(E, e);
  p.parts.clear();
  // best[k]: the shortest time of classes < k, the last launch being [from, k)
  double best[6] = {0.0};
  int from[6] = {0}, size[6] = {0};
  bool resident[6] = {false};
  std::vector<int> who;
  for (int k = 1; k <= 5; ++k) {
    best[k] = 1e300;
    for (int f = 0; f < k; ++f) {
      who.clear();
      for (int e = 0; e < E->n; ++e)
        if (cls[e] >= f && cls[e] < k) who.push_back(e);
      for (int res = 0; res < 2; ++res)
        for (int c = 1; c <= 4; ++c) {
          // the largest class needs clusters of 2 << (k - 1); from L2, clusters of
          // eight, or of 16 where they all run at once
          if (res ? c < k : c < 3 || (c == 4 && (int)who.size() > fit_clusters(E, 16, false))) continue;
          const double t = best[f] + (who.empty() ? 0.0 : launch_time(E, who, 1 << c, res != 0));
          if (t < best[k]) {
            best[k] = t;
            from[k] = f;
            size[k] = 1 << c;
            resident[k] = res != 0;
          }
        }
    }
    if (best[k] >= 1e300) return efail(E, EREM_ECUDA, "no cluster size fits the device");
  }
  // one launch from L2 on clusters of eight is the rule for every ensemble: the
  // plan replaces it where it promises more than the estimates' own error
  who.resize(E->n);
  for (int e = 0; e < E->n; ++e) who[e] = e;
  if (best[5] > 0.8 * launch_time(E, who, 8, false)) {
    from[5] = 0;
    size[5] = 8;
    resident[5] = false;
  }
  for (int k = 5; k > 0; k = from[k]) {
    EnsPlan::Part t;
    t.from = from[k];
    t.to = k;
    t.cs = size[k];
    t.res = resident[k];
    p.parts.push_back(t);
  }
  p.made = true;
  return EREM_OK;
}

// The launches of the next run and its queue order.  A given (or tuned)
// cluster size takes one launch for the members that fit on such a cluster's
// shared memory and one for the rest.  Otherwise the members are split by the
// smallest cluster they fit on, as the plan says.
erem_status plan_run(erem_ens* E) {
  const int fixed = E->cfg.cluster_ctas ? E->cfg.cluster_ctas : E->tuned_cs;
  E->launches.clear();
  std::vector<std::pair<double, int>> w(E->n);
  for (int e = 0; e < E->n; ++e) w[e] = {member_weight(E, e), e};
  std::stable_sort(w.begin(), w.end(), [](const auto& a, const auto& b) { return a.first > b.first; });
  int pos = 0;
  auto add = [&](bool res, int cs, const std::vector<char>& in) -> erem_status {
    EnsLaunch L;
    L.res = res;
    L.cs = cs;
    L.first = pos;
    for (const auto& x : w)
      if (in[x.second]) E->order_h[pos++] = x.second;
    L.count = pos - L.first;
    if (L.count == 0) return EREM_OK;
    const int fit = fit_clusters(E, cs, res);
    if (fit < 1)
      return efail(E, EREM_ECUDA, "a cluster of " + std::to_string(cs) + " CTAs does not fit the device");
    L.clusters = std::min(fit, L.count);
    E->launches.push_back(L);
    return EREM_OK;
  };
  std::vector<char> in(E->n, 0), rest(E->n, 0);
  if (fixed) {
    const bool any = fit_clusters(E, fixed, true) > 0;
    for (int e = 0; e < E->n; ++e) {
      in[e] = any && fits_resident(E, e, fixed);
      rest[e] = !in[e];
    }
    ENS_TRY(add(true, fixed, in));
    return add(false, fixed, rest);
  }
  std::vector<int> cls(E->n, 4);
  for (int e = 0; e < E->n; ++e)
    for (int k = 3; k >= 0; --k)
      if (fit_clusters(E, 2 << k, true) > 0 && fits_resident(E, e, 2 << k)) cls[e] = k;
  if (!plan_holds(E, cls)) ENS_TRY(make_plan(E, cls));
  for (const EnsPlan::Part& p : E->plan.parts) {
    for (int e = 0; e < E->n; ++e) in[e] = cls[e] >= p.from && cls[e] < p.to;
    ENS_TRY(add(p.res, p.cs, in));
  }
  return EREM_OK;
}

bool same_run(const EnsRun& a, const EnsRun& b) {
  return a.mem == b.mem && a.st == b.st && a.order == b.order && a.next == b.next && a.xi == b.xi &&
         a.n == b.n && a.nlev == b.nlev && a.mmax == b.mmax && a.restart == b.restart &&
         a.passes_per_step == b.passes_per_step;
}

// The device work of a run, in stream order: the member states and the queue
// order up from pinned host memory, the queue positions reset, the persistent
// launches, the states back.  The copies read and write the pinned buffers when
// they execute, so one capture serves every run with the same descriptor.
cudaError_t enqueue_run(erem_ens* E, const EnsRun& R, cudaStream_t s) {
  cudaError_t e = cudaMemcpyAsync(E->st_d, E->st_h, sizeof(EnsState) * E->n, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(E->order_d, E->order_h, sizeof(int) * E->n, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(E->next_d, 0, sizeof(unsigned) * kEnsLaunches, s);
  for (size_t k = 0; k < E->launches.size() && e == cudaSuccess; ++k) {
    const EnsLaunch& L = E->launches[k];
    EnsRun r = R;
    r.order = R.order + L.first;
    r.n = L.count;
    r.next = R.next + k;
    e = L.res ? launch_ens_resident(r, E->prec, L.cs, L.clusters, E->ctx[0]->smem_optin, s)
              : launch_ens_cluster(r, E->prec, L.cs, L.clusters, s);
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(E->st_h, E->st_d, sizeof(EnsState) * E->n, cudaMemcpyDeviceToHost, s);
  return e;
}

// Capture the run on the ensemble's own stream (a legacy default stream
// cannot be captured) and instantiate it; on any failure the ensemble keeps
// to direct launches.
void capture_run(erem_ens* E, const EnsRun& R) {
  if (!E->cap_stream && cudaStreamCreateWithFlags(&E->cap_stream, cudaStreamNonBlocking) != cudaSuccess) {
    cudaGetLastError();
    E->cap_stream = nullptr;
    E->graph_ok = false;
    return;
  }
  cudaGraph_t g = nullptr;
  if (cudaStreamBeginCapture(E->cap_stream, cudaStreamCaptureModeRelaxed) != cudaSuccess) {
    cudaGetLastError();
    E->graph_ok = false;
    return;
  }
  const cudaError_t e = enqueue_run(E, R, E->cap_stream);
  const cudaError_t ee = cudaStreamEndCapture(E->cap_stream, &g);
  cudaGraphExec_t x = nullptr;
  if (e != cudaSuccess || ee != cudaSuccess || !g || cudaGraphInstantiate(&x, g, 0) != cudaSuccess) {
    cudaGetLastError();
    if (g) cudaGraphDestroy(g);
    E->graph_ok = false;
    return;
  }
  cudaGraphDestroy(g);
  E->run_exec = x;
  E->run_key = R;
  E->key_launches = E->launches;
}

// One run: every member advances `steps` steps, in one launch of a batched
// kernel for each part of the plan (up to five).  A member whose Leja estimate became non-finite (the Newton
// vectors or their squares left the range of the Leja precision) or whose
// interpolation did not meet the test within m_max terms takes the step again
// at twice the substeps, as erem_step splits a step whose interpolation
// failed.
erem_status run(erem_ens* E, int steps, cudaStream_t s) {
  ENS_TRY(plan_run(E));
  const bool keep = E->cfg.substep_policy == EREM_ENS_KEEP_SUBSTEPS;
  for (int e = 0; e < E->n; ++e) {
    EnsState& st = E->st_h[e];
    std::memset(&st, 0, sizeof(st));
    st.phase = ENS_INIT;
    st.level = std::min(keep ? E->level_start[e] : 0, E->nlev - 1);
    st.target = steps;
  }
  EnsRun R{};
  R.mem = E->mem_d;
  R.st = E->st_d;
  R.order = E->order_d;
  R.next = E->next_d;
  R.xi = E->xi_d;
  R.n = E->n;
  R.nlev = E->nlev;
  R.mmax = E->m_max;
  R.restart = keep ? 0 : 1;
  R.passes_per_step = passes_per_step(E);
  if (const char* v = std::getenv("EREM_ENS_PASSES_PER_STEP")) {  // test hook: a small bound
    const long long b = std::atoll(v);
    if (b >= 1) R.passes_per_step = b;
  }
  if (E->graph_ok) {
    if (E->run_exec && !(same_run(R, E->run_key) && E->launches == E->key_launches)) drop_graph(E);
    if (!E->run_exec) capture_run(E, R);
  }
  // the events bracket the whole run: copies, queue reset and the launch
  ENS_CUDA(E, cudaEventRecord(E->ev[0], s));
  if (E->run_exec)
    ENS_CUDA(E, cudaGraphLaunch(E->run_exec, s));
  else
    ENS_CUDA(E, enqueue_run(E, R, s));
  ENS_CUDA(E, cudaEventRecord(E->ev[1], s));
  ENS_CUDA(E, cudaStreamSynchronize(s));
  float t = 0.f;
  ENS_CUDA(E, cudaEventElapsedTime(&t, E->ev[0], E->ev[1]));

  erem_ens_run_stats& r = E->rs;
  std::memset(&r, 0, sizeof(r));
  r.t_ms = t;
  {  // the shape of the launch with the most work
    double most = -1.0;
    for (const EnsLaunch& L : E->launches) {
      double sum = 0.0;
      for (int k = 0; k < L.count; ++k) sum += member_weight(E, E->order_h[L.first + k]);
      if (sum > most) {
        most = sum;
        r.cluster_ctas = L.cs;
        r.clusters = L.clusters;
      }
    }
  }
  r.cta_threads = ens_cta_threads();
  r.graph = E->run_exec ? 1 : 0;
  E->last.assign(E->st_h, E->st_h + E->n);
  int first_fail = -1;
  for (int e = 0; e < E->n; ++e) {
    const EnsState& st = E->last[e];
    const long long N = E->ctx[e]->N;
    r.passes += st.terms + st.passes;
    r.cells += N;
    r.cell_terms += N * st.terms;
    r.cell_passes += N * st.passes;
    if (st.step > 0) E->pass_rate[e] = (double)(st.terms + st.passes) / st.step;
    if (st.phase == ENS_FAILED) {
      ++r.members_failed;
      if (first_fail < 0) first_fail = e;
    } else if (st.last_S > 0) {
      int l = 0;
      while ((1 << l) < st.last_S) ++l;
      E->level_start[e] = l;
    }
  }
  if (first_fail >= 0) {
    const EnsState& st = E->last[first_fail];
    const std::string who = "member " + std::to_string(first_fail);
    if (st.status == ENS_NONFINITE)
      return efail(E, EREM_ENONFINITE, who + ": non-finite value in the state or the Leja estimate");
    if (st.status == ENS_TIMEOUT)
      return efail(E, EREM_ETIMEOUT, who + ": the member reached its bound on passes");
    return efail(E, EREM_ENOTCONV,
                 who + ": Leja interpolation did not meet the stopping test within m_max terms after " +
                     std::to_string(E->max_doublings) + " substep doublings");
  }
  return EREM_OK;
}

erem_status check_member(erem_ens* E, int e) {
  if (e < 0 || e >= E->n) return efail(E, EREM_EINVAL, "member index out of range");
  return EREM_OK;
}

}  // namespace

extern "C" {

erem_status erem_ensemble_create(int n_members, const erem_grid* grids, const erem_physics* phys,
                                 erem_precision prec, erem_ens** out) {
  if (!out) return EREM_EINVAL;
  *out = nullptr;
  if (n_members < 1 || !grids || !phys) return EREM_EINVAL;
  if (prec != EREM_FP64 && prec != EREM_FP32_BULK) return EREM_EINVAL;
  for (int e = 0; e < n_members; ++e)
    if (grids[e].dim != 2 || phys[e].fluid_model != 0) return EREM_EINVAL;
  erem_ens* E = new erem_ens();
  E->n = n_members;
  E->prec = prec;
  E->ctx.assign(n_members, nullptr);
  E->ready.assign(n_members, 0);
  E->dt.assign(n_members, 0.0);
  E->level_start.assign(n_members, 0);
  E->pass_rate.assign(n_members, 0.0);
  auto bail = [&](erem_status st) {
    erem_ensemble_destroy(E);
    return st;
  };
  long long maxN = 1;
  for (int e = 0; e < n_members; ++e) {
    const erem_status st = erem_create(&grids[e], &phys[e], prec, &E->ctx[e]);
    if (st != EREM_OK) return bail(st);
    maxN = std::max(maxN, E->ctx[e]->N);
  }
  if (cudaMalloc((void**)&E->stage_d, sizeof(double) * maxN) != cudaSuccess) return bail(EREM_ENOMEM);
  if (cudaEventCreate(&E->ev[0]) != cudaSuccess || cudaEventCreate(&E->ev[1]) != cudaSuccess)
    return bail(EREM_ECUDA);
  if (const char* v = std::getenv("EREM_ENS_RESIDENT")) E->resident_ok = std::atoi(v) != 0;  // tuning override
  if (const char* v = std::getenv("EREM_ENS_GRAPH")) E->graph_ok = std::atoi(v) != 0;  // 0: direct launches
  *out = E;
  return EREM_OK;
}

erem_status erem_ensemble_destroy(erem_ens* E) {
  if (!E) return EREM_OK;
  release_tables(E);
  for (erem_ctx* c : E->ctx)
    if (c) erem_destroy(c);
  if (E->snap_d) cudaFree(E->snap_d);
  if (E->stage_d) cudaFree(E->stage_d);
  for (cudaEvent_t ev : E->ev)
    if (ev) cudaEventDestroy(ev);
  if (E->cap_stream) cudaStreamDestroy(E->cap_stream);
  delete E;
  return EREM_OK;
}

erem_status erem_ensemble_set_member(erem_ens* E, int e, const double* T, const double* p,
                                     const double* lnk, const double* phi, const double* lam,
                                     double dt, void* stream) {
  if (!E) return EREM_EINVAL;
  ENS_TRY(check_member(E, e));
  E->ready[e] = 0;
  E->built = false;
  E->dd_valid = false;
  const erem_status st = erem_set_state(E->ctx[e], T, p, lnk, phi, lam, dt, stream);
  if (st != EREM_OK) return efail(E, st, "member " + std::to_string(e) + ": " + E->ctx[e]->err);
  E->ready[e] = 1;
  E->dt[e] = dt;
  E->level_start[e] = 0;
  E->pass_rate[e] = 0.0;
  return EREM_OK;
}

erem_status erem_ensemble_set_temperature(erem_ens* E, int e, const double* T, void* stream) {
  if (!E) return EREM_EINVAL;
  ENS_TRY(check_member(E, e));
  if (!T) return efail(E, EREM_EINVAL, "T is NULL");
  if (!E->ready[e]) return efail(E, EREM_EINVAL, "member has no state");
  cudaStream_t s = (cudaStream_t)stream;
  const erem_ctx* c = E->ctx[e];
  const double* src = T;
  if (!is_device(T)) {
    ENS_CUDA(E, cudaMemcpyAsync(E->stage_d, T, sizeof(double) * c->N, cudaMemcpyHostToDevice, s));
    src = E->stage_d;
  }
  launch_pack(c, src, c->Tn, s);
  ENS_CUDA(E, cudaGetLastError());
  if (src != T) ENS_CUDA(E, cudaStreamSynchronize(s));  // the staging buffer is reused
  return EREM_OK;
}

erem_status erem_ensemble_get_member(erem_ens* E, int e, double* T, void* stream) {
  if (!E) return EREM_EINVAL;
  ENS_TRY(check_member(E, e));
  if (!T) return efail(E, EREM_EINVAL, "T is NULL");
  if (!E->ready[e]) return efail(E, EREM_EINVAL, "member has no state");
  cudaStream_t s = (cudaStream_t)stream;
  const erem_ctx* c = E->ctx[e];
  if (is_device(T)) {
    launch_unpack(c, c->Tn, T, s);
    ENS_CUDA(E, cudaGetLastError());
    return EREM_OK;
  }
  launch_unpack(c, c->Tn, E->stage_d, s);
  ENS_CUDA(E, cudaGetLastError());
  ENS_CUDA(E, cudaMemcpyAsync(T, E->stage_d, sizeof(double) * c->N, cudaMemcpyDeviceToHost, s));
  ENS_CUDA(E, cudaStreamSynchronize(s));
  return EREM_OK;
}

erem_status erem_ensemble_configure(erem_ens* E, const erem_leja_opts* o, const erem_ens_config* cfg) {
  if (!E) return EREM_EINVAL;
  double tol_a = 1e-6, tol_r = 1e-6;
  int p_order = 2, m_max = 150, max_doublings = 6, avg_window = 5;
  if (o) {
    if (o->replay || o->time_terms) return efail(E, EREM_EINVAL, "replay and time_terms are not batched");
    if (o->tol_a != 0.0) tol_a = o->tol_a;
    if (o->tol_r != 0.0) tol_r = o->tol_r;
    if (o->p_order != 0) p_order = o->p_order;
    if (o->m_max != 0) m_max = o->m_max;
    max_doublings = o->max_doublings;
    if (o->avg_window != 0) avg_window = o->avg_window;
  }
  if (!(tol_a >= 0.0) || !(tol_r >= 0.0) || tol_a + tol_r <= 0.0)
    return efail(E, EREM_EINVAL, "tolerances must be >= 0 with tol_a + tol_r > 0");
  if (m_max < 1 || m_max > kMaxTerms || avg_window < 1 || avg_window > kEnsWin || p_order < 0 ||
      p_order > 30 || max_doublings < 0 || max_doublings > kEnsMaxLevels - 1)
    return efail(E, EREM_EINVAL, "bad m_max, avg_window (1..64), p_order or max_doublings (0..6)");
  erem_ens_config c = E->cfg;
  if (cfg) {
    c = *cfg;
    if (c.substep_policy != EREM_ENS_KEEP_SUBSTEPS && c.substep_policy != EREM_ENS_RESTART_SUBSTEPS)
      return efail(E, EREM_EINVAL, "unknown substep policy");
    if (c.cluster_ctas != 0 && c.cluster_ctas != 2 && c.cluster_ctas != 4 && c.cluster_ctas != 8 &&
        c.cluster_ctas != 16)
      return efail(E, EREM_EINVAL, "cluster_ctas must be 0, 2, 4, 8 or 16");
    if (c.max_clusters < 0) return efail(E, EREM_EINVAL, "max_clusters must be >= 0");
    if (c.reserved != 0) return efail(E, EREM_EINVAL, "reserved must be 0");
  }
  E->tol_a = tol_a;
  E->tol_r = tol_r;
  E->p_order = p_order;
  E->m_max = m_max;
  E->max_doublings = max_doublings;
  E->avg_window = avg_window;
  E->cfg = c;
  E->built = false;
  E->dd_valid = false;
  std::fill(E->level_start.begin(), E->level_start.end(), 0);
  std::fill(E->pass_rate.begin(), E->pass_rate.end(), 0.0);
  return EREM_OK;
}

erem_status erem_ensemble_run(erem_ens* E, int steps, void* stream) {
  if (!E) return EREM_EINVAL;
  if (steps < 1) return efail(E, EREM_EINVAL, "steps must be >= 1");
  if (!E->built) ENS_TRY(build(E));
  return run(E, steps, (cudaStream_t)stream);
}

erem_status erem_ensemble_autotune(erem_ens* E, int probe_steps, void* stream) {
  if (!E) return EREM_EINVAL;
  if (probe_steps < 1) return efail(E, EREM_EINVAL, "probe_steps must be >= 1");
  cudaStream_t s = (cudaStream_t)stream;
  long long tot = 0;
  for (int e = 0; e < E->n; ++e) tot += E->ctx[e]->Np;
  if (!E->snap_d && cudaMalloc((void**)&E->snap_d, sizeof(double) * tot) != cudaSuccess) {
    cudaGetLastError();
    E->snap_d = nullptr;
    return efail(E, EREM_ENOMEM, "cudaMalloc of the autotuner snapshot failed");
  }
  auto copy_all = [&](bool save) -> erem_status {
    long long off = 0;
    for (int e = 0; e < E->n; ++e) {
      const erem_ctx* c = E->ctx[e];
      double* a = E->snap_d + off;
      ENS_CUDA(E, cudaMemcpyAsync(save ? a : c->Tn, save ? c->Tn : a, sizeof(double) * c->Np,
                                  cudaMemcpyDeviceToDevice, s));
      off += c->Np;
    }
    return EREM_OK;
  };
  // A first probe from the current starting levels learns each member's
  // substep level (reached by doubling, as erem_step would) and its passes
  // per step (the queue order); then every cluster size that fits is timed
  // on that schedule.
  const std::vector<int> levels0 = E->level_start;
  const std::vector<double> rates0 = E->pass_rate;
  const erem_ens_config keep = E->cfg;
  const int tuned0 = E->tuned_cs;
  const bool keep_policy = keep.substep_policy == EREM_ENS_KEEP_SUBSTEPS;
  auto restore = [&](erem_status st) {
    E->cfg = keep;
    E->level_start = levels0;
    E->pass_rate = rates0;
    E->tuned_cs = tuned0;
    copy_all(false);
    cudaStreamSynchronize(s);
    return st;
  };
  ENS_TRY(copy_all(true));
  erem_status st = E->built ? EREM_OK : build(E);
  if (st == EREM_OK) st = run(E, probe_steps, s);
  if (st != EREM_OK) return restore(st);
  const std::vector<int> learned = E->level_start;
  const std::vector<double> rates = E->pass_rate;
  if (copy_all(false) != EREM_OK) return restore(EREM_ECUDA);
  const int cand[5] = {0, 2, 4, 8, 16};   // 0: the planned launches
  E->tuned_cs = 0;
  double best = 1e300;
  int best_cs = -1;
  for (int cs : cand) {
    if (cs && fit_clusters(E, cs, false) < 1) continue;
    E->cfg.cluster_ctas = cs;
    E->level_start = keep_policy ? learned : levels0;
    E->pass_rate = rates;
    st = run(E, probe_steps, s);
    if (st != EREM_OK) return restore(st);
    if (E->rs.t_ms < best) {
      best = E->rs.t_ms;
      best_cs = cs;
    }
    if (copy_all(false) != EREM_OK) return restore(EREM_ECUDA);
  }
  ENS_CUDA(E, cudaStreamSynchronize(s));
  if (best_cs < 0) return restore(efail(E, EREM_ECUDA, "no cluster size fits the device"));
  E->cfg = keep;
  E->tuned_cs = best_cs;
  E->level_start = keep_policy ? learned : levels0;
  E->pass_rate = rates;
  return EREM_OK;
}

erem_status erem_ensemble_member_stats(const erem_ens* E, int e, erem_ens_member_stats* out) {
  if (!E || !out || e < 0 || e >= E->n) return EREM_EINVAL;
  std::memset(out, 0, sizeof(*out));
  out->alpha = E->ctx[e]->alpha;
  out->beta = E->ctx[e]->beta;
  out->leja_coefficients = erem_leja_coefficients(E->ctx[e]);
  if (E->last.empty()) return EREM_OK;
  const EnsState& st = E->last[e];
  out->status = st.phase != ENS_FAILED       ? EREM_OK
                : st.status == ENS_NONFINITE ? EREM_ENONFINITE
                : st.status == ENS_TIMEOUT   ? EREM_ETIMEOUT
                                             : EREM_ENOTCONV;
  out->steps_done = st.step;
  out->substeps = st.last_S;
  for (int k = 0; k < 64; ++k) {
    out->degrees[k] = st.last_deg[k];
    out->degree_total += st.last_deg[k];
  }
  out->terms = st.terms;
  out->passes = st.passes;
  out->attempts = st.attempts;
  return EREM_OK;
}

erem_status erem_ensemble_run_stats(const erem_ens* E, erem_ens_run_stats* out) {
  if (!E || !out) return EREM_EINVAL;
  *out = E->rs;
  return EREM_OK;
}

const char* erem_ensemble_last_error(const erem_ens* E) {
  return E ? E->err.c_str() : "erem: NULL ensemble";
}

}  // extern "C"
