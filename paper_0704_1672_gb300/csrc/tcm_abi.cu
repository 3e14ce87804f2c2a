// C ABI of libtcm.so (include/tcm.h): argument checks, the context (tables, scratch,
// descriptor staging) and the host-side planning of moment jobs and tiles.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <exception>
#include <new>
#include <vector>

#include "contract.h"

using namespace tcm;

namespace {

thread_local char g_err[512] = "";

int set_err(int code, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof g_err, fmt, ap);
  va_end(ap);
  return code;
}

#define TRY_CUDA(expr)                                                                                   \
  do {                                                                                                   \
    cudaError_t e_ = (expr);                                                                             \
    if (e_ != cudaSuccess) return set_err(TCM_ECUDA, "%s: %s", #expr, cudaGetErrorString(e_));           \
  } while (0)
#define TRY(expr)                   \
  do {                              \
    int r_ = (expr);                \
    if (r_ != TCM_OK) return r_;    \
  } while (0)
#define TRY_LAUNCH(expr)                                                                                 \
  do {                                                                                                   \
    if ((expr) != 0) {                                                                                   \
      cudaError_t e_ = cudaGetLastError();                                                               \
      return set_err(TCM_ECUDA, "%s: %s", #expr, cudaGetErrorString(e_));                                \
    }                                                                                                    \
  } while (0)

struct DevBuf {
  void* p = nullptr;
  size_t cap = 0;
};

struct Stage {  // pinned host staging slot for one call's descriptors
  void* host = nullptr;
  size_t cap = 0;
  cudaEvent_t ev = nullptr;
  bool pending = false;
};

constexpr int kStages = 4;
constexpr size_t kAlign = 256;

size_t align_up(size_t v) { return (v + kAlign - 1) & ~(kAlign - 1); }

// Layout of one call's descriptor block: add() records where each host array goes (256-byte
// aligned offsets); upload() copies the arrays straight into a pinned staging buffer and
// sends the block with a single copy.  The arrays must stay unchanged until upload().
struct Packer {
  struct Span {
    const void* p;
    size_t bytes;
    size_t off;
  };
  std::vector<Span> spans;
  size_t size = 0;
  template <typename T>
  size_t add(const std::vector<T>& v) {
    const size_t off = align_up(size);
    spans.push_back(Span{v.data(), v.size() * sizeof(T), off});
    size = off + std::max<size_t>(v.size() * sizeof(T), 1);
    return off;
  }
  // two arrays of one type back to back (one device array), without concatenating them on the host
  template <typename T>
  size_t add2(const std::vector<T>& a, const std::vector<T>& b) {
    const size_t off = align_up(size);
    spans.push_back(Span{a.data(), a.size() * sizeof(T), off});
    spans.push_back(Span{b.data(), b.size() * sizeof(T), off + a.size() * sizeof(T)});
    size = off + std::max<size_t>((a.size() + b.size()) * sizeof(T), 1);
    return off;
  }
};

// What the host arrays of a call throw stays behind the C entry.
int no_host_memory(const char* what) { return set_err(TCM_ENOMEM, "%s: host allocation failed", what); }

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace

namespace {
struct BatchScratch;
}

struct tcm_ctx {
  BatchScratch* scratch = nullptr;  // host arrays of the batched calls, kept for their capacity
  void (*free_scratch)(BatchScratch*) = nullptr;
  int device = 0;
  int num_sms = 0;
  int lmax_cap = 0;
  cudaStream_t stream = nullptr;
  // tables
  double* d_fmap = nullptr;  // F_lm of the component each (chunk, slot) holds
  ContractTables* d_ctab = nullptr;  // tables of the contraction and of the rotation of moments
  int* d_imap = nullptr;      // (chunk, slot) -> packed component, both precisions
  int* d_imap_off = nullptr;  // [precision][L] offsets into d_imap
  // scratch
  DevBuf desc, partials, gpart, systk, systiles, counters, moms, escr, dpart, tiles;
  Stage stage[kStages];
  int stage_next = 0;
  void* pinned_small = nullptr;  // 256 B for small device->host reads
  // moment-pass tiling per [TCM_FP64, TCM_MIXED][L]: atoms per lane of a warp tile, and the
  // resident CTAs per SM the persistent grid is sized for
  int atoms_per_thread[2][kLmaxMax + 1];
  int ctas_per_sm[2][kLmaxMax + 1];
  bool tiling_set[kLmaxMax + 1] = {};  // TCM_FP64: atoms per lane were set (else smaller tiles for small systems)
  int plan_l[kLmaxMax + 1];  // mixed path: the float kernel's chunk plan per degree (1 or 2)
  int64_t cfg_gen = 0;       // bumped by every tiling or chunking change (part of the graph key)
  // phase profiling
  bool prof = false;
  struct Mark {
    int phase;
    cudaEvent_t a, b;
  };
  std::vector<Mark> marks;
  std::vector<cudaEvent_t> ev_pool;
  int64_t launches[TCM_NPHASES] = {};
  double host_ms = 0.0;  // TCM_PHASE_HOST: wall time inside the batched calls while profiling
  // CUDA-graph replay of the batched launch sequence
  bool rotate_cached = false;  // rotated B sides from the moment cache by Wigner rotation
  int graphs = 1;  // 0: launch directly; 1: capture a shape seen twice in a row; 2: capture every new shape
  cudaStream_t cap_stream = nullptr;
  cudaGraphExec_t gexec = nullptr;
  std::vector<long long> gkey, gkey_seen;
  int64_t graph_captures = 0, graph_launches = 0;
};

namespace {

cudaEvent_t pool_event(tcm_ctx* c) {
  if (!c->ev_pool.empty()) {
    cudaEvent_t e = c->ev_pool.back();
    c->ev_pool.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
  return e;
}

// Records an event pair around one phase when profiling is on, and counts launches.
struct PhaseScope {
  tcm_ctx* c;
  int phase;
  cudaEvent_t a = nullptr;
  PhaseScope(tcm_ctx* c_, int ph, int nlaunch) : c(c_), phase(ph) {
    c->launches[ph] += nlaunch;
    if (c->prof && (a = pool_event(c)) != nullptr) cudaEventRecord(a, c->stream);
  }
  ~PhaseScope() {
    if (!a) return;
    cudaEvent_t b = pool_event(c);
    if (!b) {
      c->ev_pool.push_back(a);
      return;
    }
    cudaEventRecord(b, c->stream);
    c->marks.push_back({phase, a, b});
  }
};

int dev_ensure(tcm_ctx* c, DevBuf& b, size_t bytes) {
  if (bytes <= b.cap) return TCM_OK;
  size_t nc = std::max(bytes, b.cap + b.cap / 2);
  nc = align_up(std::max<size_t>(nc, kAlign));
  if (b.p) {
    TRY_CUDA(cudaStreamSynchronize(c->stream));
    TRY_CUDA(cudaFree(b.p));
    b.p = nullptr;
    b.cap = 0;
  }
  if (cudaMalloc(&b.p, nc) != cudaSuccess) {
    cudaGetLastError();
    return set_err(TCM_ENOMEM, "cudaMalloc of %zu bytes failed", nc);
  }
  b.cap = nc;
  return TCM_OK;
}

// The next pinned staging slot, free to write and at least `bytes` large; the first `keep` bytes of the
// slot survive its growth.
int stage_slot(tcm_ctx* c, size_t bytes, size_t keep, Stage** out) {
  Stage& st = c->stage[c->stage_next];
  if (st.pending) {
    TRY_CUDA(cudaEventSynchronize(st.ev));
    st.pending = false;
  }
  if (st.cap < bytes) {
    const size_t nc = align_up(std::max<size_t>(bytes + bytes / 2, 4096));
    void* p = nullptr;
    if (cudaHostAlloc(&p, nc, cudaHostAllocDefault) != cudaSuccess) {
      cudaGetLastError();
      return set_err(TCM_ENOMEM, "cudaHostAlloc of %zu bytes failed", nc);
    }
    if (st.host) {
      if (keep) std::memcpy(p, st.host, std::min(keep, st.cap));
      cudaFreeHost(st.host);
    }
    st.host = p;
    st.cap = nc;
  }
  *out = &st;
  return TCM_OK;
}

// Copy the packed descriptors to the device through a pinned slot (its first `in_place` bytes were
// written there by the caller, Packer's size began with them); returns the device base address in *dbase.
// `behind` more bytes of the device buffer follow the block (at align_up(pk.size)) for the call's kernels.
int upload(tcm_ctx* c, const Packer& pk, char** dbase, size_t in_place = 0, size_t behind = 0) {
  const size_t bytes = std::max<size_t>(pk.size, 1);
  TRY(dev_ensure(c, c->desc, align_up(bytes) + behind));
  Stage* st = nullptr;
  TRY(stage_slot(c, bytes, in_place, &st));
  c->stage_next = (c->stage_next + 1) % kStages;
  for (const Packer::Span& sp : pk.spans)
    if (sp.bytes) std::memcpy(static_cast<char*>(st->host) + sp.off, sp.p, sp.bytes);
  TRY_CUDA(cudaMemcpyAsync(c->desc.p, st->host, bytes, cudaMemcpyHostToDevice, c->stream));
  TRY_CUDA(cudaEventRecord(st->ev, c->stream));
  st->pending = true;
  *dbase = static_cast<char*>(c->desc.p);
  return TCM_OK;
}

int check_system(const tcm_system* s, const char* what) {
  if (!s) return set_err(TCM_EINVAL, "%s: null system", what);
  if (s->n < 0) return set_err(TCM_EINVAL, "%s: negative atom count", what);
  if (s->dtype != TCM_F32 && s->dtype != TCM_F64) return set_err(TCM_EINVAL, "%s: dtype must be TCM_F32 or TCM_F64", what);
  if (s->n > 0 && !s->xyzq) return set_err(TCM_EINVAL, "%s: null coordinate pointer", what);
  if (s->n > 0 && !aligned16(s->xyzq)) return set_err(TCM_EINVAL, "%s: coordinates must be 16-byte aligned", what);
  if (s->has_center && !(std::isfinite(s->center[0]) && std::isfinite(s->center[1]) && std::isfinite(s->center[2])))
    return set_err(TCM_EINVAL, "%s: non-finite centre", what);
  if (s->moments) {
    if (!s->has_center || !(s->radius >= 0.0))
      return set_err(TCM_EINVAL, "%s: a moment cache needs the centre and radius it was taken with", what);
    if (s->moments_lmax < 0 || s->moments_lmax > TCM_LMAX_MAX || !aligned16(s->moments))
      return set_err(TCM_EINVAL, "%s: bad moment cache (lmax or alignment)", what);
  }
  return TCM_OK;
}

bool geom_known(const tcm_system& s) { return s.has_center && s.radius >= 0.0; }

// Moment-job planning -------------------------------------------------------------


// Doubles of partial rows a pass of the double path may take (1 GiB).  Its tiles are small, so that one
// small system fills the GPU (2,000 atoms: 63 tiles; 315 KB of rows at degree 24), and a batch of 100,000
// would ask for 31 GB of rows at once; in passes of moments and finalisation, one behind the other, they
// reuse the same rows.  The float path's tiles are larger, its rows fewer: always one pass.
constexpr size_t kPassDoubles = size_t(1) << 27;

struct Plan {
  std::vector<MomJob> jobs;
  std::vector<MomGroup> groups;    // (job, chunk) groups, largest tiles first; expanded on the device
  int n_tiles = 0;
  // A pass: jobs [job0, job0 + n_jobs), moment launches and a finalisation.  FP64 (one launch per degree):
  // the tiles of L are [tile_begin[L], tile_begin[L+1]); mixed (one launch per chunk plan over all
  // degrees): the tiles of plan p are [tile_begin[p - 1], tile_begin[p])
  struct Pass {
    int job0, n_jobs;
    int tile_begin[kLmaxMax + 2];
  };
  std::vector<Pass> passes;
  size_t part_doubles = 0;  // partial rows, of the pass that has most
  int n_tile_ids = 0;
  struct Group {
    int job, chunk;
  };
  std::vector<Group> sort_groups;  // working arrays of build_tiles
  std::vector<uint32_t> sort_key, sort_key2, sort_order, sort_order2;
};

void plan_job(tcm_ctx* c, int precision, MomJob& j, int& next_id) {
  j.plan = precision == TCM_FP64 ? 0 : c->plan_l[j.L];
  const int nch = moments_nchunks(j.plan, j.L);
  long long apl = c->atoms_per_thread[precision == TCM_FP64 ? 0 : 1][j.L];
  if (precision == TCM_FP64 && !c->tiling_set[j.L]) apl = std::min<long long>(apl, f64_rows(j.n));
  const long long per_tile = 32 * apl;
  long long tpc = (j.n + per_tile - 1) / per_tile;
  if (tpc < 1) tpc = 1;
  j.tiles_per_chunk = (int)tpc;
  j.atoms_per_tile = (int)((j.n + tpc - 1) / tpc);
  next_id += nch * (int)tpc;
}


// Cuts the jobs into passes and places their partial rows.
void plan_passes(int precision, Plan& P) {
  P.passes.clear();
  P.part_doubles = 0;
  size_t at = 0;
  for (int ji = 0; ji < (int)P.jobs.size(); ++ji) {
    MomJob& j = P.jobs[ji];
    const size_t need = (size_t)moments_nchunks(j.plan, j.L) * j.tiles_per_chunk * plan_row(j.plan, j.L);
    if (ji == 0 || (precision == TCM_FP64 && at + need > kPassDoubles)) {
      P.passes.push_back(Plan::Pass{ji, 0, {}});
      at = 0;
    }
    ++P.passes.back().n_jobs;
    j.part = (long long)at;
    at += need;
    P.part_doubles = std::max(P.part_doubles, at);
  }
}

// The (job, chunk) groups of each pass in decreasing order of their tiles' cost (largest first, so the
// persistent warps finish together).  FP64: grouped by degree (one launch per degree); mixed:
// grouped by chunk plan (one launch per plan present, usually one), one order over all degrees.  The tiles themselves are written on the device
// (k_expand_tiles), so the host work is O(groups log groups).
void build_tiles(int precision, Plan& P) {
  // one 32-bit key per group: [degree (FP64) or chunk plan (mixed), 5 bits] [largest cost first,
  // 27 bits]; a stable sort keeps ties in their planning order, so the order is deterministic.
  // The sort is a least-significant-digit radix sort (three passes of 11 bits): for the tens of
  // thousands of groups of a large batch it takes a fraction of a comparison sort's time.
  using Group = Plan::Group;
  std::vector<Group>& g = P.sort_groups;
  std::vector<uint32_t>& key = P.sort_key;
  const bool by_degree = precision == TCM_FP64;
  plan_passes(precision, P);
  P.groups.clear();
  int first = 0;
  for (Plan::Pass& pass : P.passes) {
    g.clear();
    key.clear();
    for (int ji = pass.job0; ji < pass.job0 + pass.n_jobs; ++ji) {
      const MomJob& j = P.jobs[ji];
      const int nch = moments_nchunks(j.plan, j.L);
      const double* cc = moments_chunk_costs(j.plan, j.L);
      for (int ch = 0; ch < nch; ++ch) {
        const double cost = cc[ch] * (double)j.atoms_per_tile;
        const uint32_t cq = (uint32_t)std::min(cost, 134217727.0);  // 27 bits
        key.push_back(((uint32_t)(by_degree ? j.L : j.plan - 1) << 27) | (134217727u - cq));
        g.push_back(Group{ji, ch});
      }
    }
    const size_t n = key.size();
    const bool few = n <= 64;  // an insertion sort beats the radix sort's histograms
    std::vector<uint32_t>&order = P.sort_order, &k2 = P.sort_key2, &o2 = P.sort_order2;
    order.resize(n);
    k2.resize(n);
    o2.resize(n);
    for (size_t i = 0; i < n; ++i) order[i] = (uint32_t)i;
    for (size_t i = 1; few && i < n; ++i) {
      const uint32_t o = order[i];
      size_t j = i;
      for (; j > 0 && key[order[j - 1]] > key[o]; --j) order[j] = order[j - 1];
      order[j] = o;
    }
    for (int shift = 0; !few && shift < 32; shift += 11) {
      uint32_t count[2049] = {};
      for (size_t i = 0; i < n; ++i) ++count[((key[i] >> shift) & 2047u) + 1];
      for (int b = 0; b < 2048; ++b) count[b + 1] += count[b];
      for (size_t i = 0; i < n; ++i) {
        const uint32_t d = (key[i] >> shift) & 2047u;
        k2[count[d]] = key[i];
        o2[count[d]++] = order[i];
      }
      key.swap(k2);
      order.swap(o2);
    }
    P.groups.reserve(P.groups.size() + n);
    size_t gi = 0;
    for (int L = 0; L <= kLmaxMax; ++L) {
      pass.tile_begin[L] = first;
      for (; gi < n; ++gi) {
        const Group& gr = g[order[gi]];
        if ((by_degree ? P.jobs[gr.job].L : P.jobs[gr.job].plan - 1) != L) break;
        const int nt = P.jobs[gr.job].tiles_per_chunk;
        P.groups.push_back(MomGroup{gr.job, gr.chunk, nt, first});
        first += nt;
      }
    }
    pass.tile_begin[kLmaxMax + 1] = first;
  }
  P.n_tiles = first;
}

// Moment-phase launches of a plan (for the launch counts of a replayed graph): FP64 one per
// degree present, mixed one per chunk plan present.
int moment_launches(int precision, const Plan& P) {
  const int nb = precision == TCM_FP64 ? kLmaxMax + 1 : kNumPlans - 1;
  int n = 0;
  for (const Plan::Pass& pass : P.passes)
    for (int k = 0; k < nb; ++k) n += pass.tile_begin[k + 1] > pass.tile_begin[k];
  return n;
}

// CTAs per job of a pass's finalisation.
int split_of(const Plan& P, const Plan::Pass& pass) {
  int max_tiles = 0, max_slots = 0;
  for (int ji = pass.job0; ji < pass.job0 + pass.n_jobs; ++ji) {
    const MomJob& j = P.jobs[ji];
    max_tiles = std::max(max_tiles, j.tiles_per_chunk);
    max_slots = std::max(max_slots, moments_nchunks(j.plan, j.L) * plan_slots(j.plan, j.L));
  }
  return finalize_split(pass.n_jobs, max_tiles, max_slots);
}

// Most columns in a chunk of the jobs under one float plan (the column kernel's grid).
int max_cols_of(const Plan& P, int plan) {
  int mx = 0;
  for (const MomJob& j : P.jobs)
    if (j.plan == plan) mx = std::max(mx, moments_max_cols(plan, j.L));
  return mx;
}

// Queue the moment pass (step a2/a3) for every job of the plan.
// The moment kernels' work counters and exit tickets (counters[L], counters[32 + L]) are zero
// on entry and left zero by every launch, so they are cleared once, when allocated.
int ensure_moment_buffers(tcm_ctx* c, const Plan& P, bool tiles_on_host) {
  if (P.jobs.empty()) return TCM_OK;
  TRY(dev_ensure(c, c->partials, std::max<size_t>(P.part_doubles, 1) * sizeof(double)));
  if (!tiles_on_host) TRY(dev_ensure(c, c->tiles, (size_t)std::max(P.n_tiles, 1) * sizeof(MomTile)));
  void* before = c->counters.p;
  TRY(dev_ensure(c, c->counters, 64 * sizeof(int)));
  if (c->counters.p != before) {
    TRY_CUDA(cudaMemsetAsync(c->counters.p, 0, 64 * sizeof(int), c->stream));
  }
  return TCM_OK;
}

// Counter slots of the moment kernels (zero on entry, left zero): [L] and [32 + L] for the
// per-degree FP64 launches, [kAnyCounter + p] and [32 + kAnyCounter + p] for the mixed launch of
// chunk plan p over all degrees.
constexpr int kAnyCounter = kLmaxMax;  // + plan (1 or 2)

int run_pass(tcm_ctx* c, int precision, const Plan& P, const Plan::Pass& pass, const MomJob* d_jobs, const MomTile* tiles,
             const SysGeom* d_geoms, cudaStream_t st) {
  int* counters = static_cast<int*>(c->counters.p);
  double* parts = static_cast<double*>(c->partials.p);
  if (precision == TCM_FP64) {
    int ngroups = 0;
    for (int L = 0; L <= kLmaxMax; ++L) ngroups += pass.tile_begin[L + 1] > pass.tile_begin[L];
    PhaseScope ps(c, TCM_PHASE_MOMENTS, ngroups);
    for (int L = 0; L <= kLmaxMax; ++L) {
      const int b = pass.tile_begin[L], e = pass.tile_begin[L + 1];
      if (e == b) continue;
      const int grid = std::min(e - b, c->ctas_per_sm[0][L] * c->num_sms);  // a CTA per tile
      TRY_LAUNCH(launch_moments(0, L, d_jobs, tiles + b, e - b, counters + L, d_geoms, parts, grid, st));
    }
  } else if (P.n_tiles > 0) {
    PhaseScope ps(c, TCM_PHASE_MOMENTS, moment_launches(precision, P));
    for (int p = 1; p < kNumPlans; ++p) {
      const int b = pass.tile_begin[p - 1], e = pass.tile_begin[p];
      if (e == b) continue;
      if (moments_use_cols(P.n_tiles, c->num_sms)) {
        TRY_LAUNCH(launch_moments_cols(d_jobs, tiles + b, e - b, max_cols_of(P, p), d_geoms, parts, st));
        continue;
      }
      int cps = 1;  // the grid: the largest CTAs per SM of the plan's degrees, within its kernel's limit
      for (const MomJob& j : P.jobs)
        if (j.plan == p) cps = std::max(cps, c->ctas_per_sm[1][j.L]);
      cps = std::min(cps, moment_ctas(plan_kmax(p)));
      const int grid = std::min((e - b + kThreads / 32 - 1) / (kThreads / 32), cps * c->num_sms);
      TRY_LAUNCH(launch_moments(p, -1, d_jobs, tiles + b, e - b, counters + kAnyCounter + p, d_geoms, parts, grid,
                                st));
    }
  }
  {
    PhaseScope ps(c, TCM_PHASE_FINALIZE, 1);
    TRY_LAUNCH(launch_finalize(d_jobs + pass.job0, pass.n_jobs, parts, d_geoms, c->d_imap, c->d_fmap, c->d_imap_off,
                               static_cast<double*>(c->gpart.p), split_of(P, pass), st));
  }
  return TCM_OK;
}

// (A pass writes its rows only once the finalisation before it has read them: every moment kernel waits for
// the launch before it first.)
int run_moments(tcm_ctx* c, int precision, const Plan& P, const MomJob* d_jobs, const MomTile* tiles,
                const SysGeom* d_geoms, cudaStream_t st) {
  for (const Plan::Pass& pass : P.passes) TRY(run_pass(c, precision, P, pass, d_jobs, tiles, d_geoms, st));
  return TCM_OK;
}

// The pass over the systems' atoms before the moment pass (syspass.cu): step a1 for the systems
// whose centre or radius is not given, and the low-degree sums of the mixed path for every
// system with a computed moment job.
struct SysPlan {
  std::vector<SysJob> jobs;     // by class
  SysCount n;
  std::vector<int> of_system;   // system -> index of its SysJob, or -1
  int rows = 0;
  std::vector<SysJob> of_class[3];  // working arrays of plan_sys
};

// used[s]: system s takes part in the call; low[s]: its low-degree sums are needed.
void plan_sys(const tcm_system* systems, int n_systems, const std::vector<char>& used, const std::vector<char>& low,
              SysPlan& S) {
  S.of_system.assign(std::max(n_systems, 0), -1);
  S.jobs.clear();
  S.n = SysCount{};
  S.rows = 0;
  std::vector<SysJob>* of_class = S.of_class;
  for (int k = 0; k < 3; ++k) of_class[k].clear();
  for (int s = 0; s < n_systems; ++s) {
    if (!used[s]) continue;
    const tcm_system& sy = systems[s];
    const bool nc = !sy.has_center;
    const bool nr = nc || sy.radius < 0.0;  // a radius given without its centre is recomputed
    const bool nl = !low.empty() && low[s];
    if (!nc && !nr && !nl) continue;
    SysJob j{};
    j.xyzq = sy.xyzq;
    j.n = sy.n;
    j.dtype = sy.dtype;
    j.geom = s;
    j.need_center = nc;
    j.need_radius = nr;
    j.need_low = nl;
    j.sum_row = j.first1 = j.first2 = -1;
    const int cl = sys_class(sy.n, sy.dtype);
    if (cl == 2) {
      j.atoms_per_tile = sys_tile_atoms(sy.n);
      j.n_tiles = (int)((sy.n + j.atoms_per_tile - 1) / j.atoms_per_tile);
      j.tile_base = S.rows;
      S.rows += j.n_tiles;
      if (nc) {
        j.first1 = S.n.tiles1;
        S.n.tiles1 += j.n_tiles;
      }
      if (nr || nl) {
        j.first2 = S.n.tiles2;
        S.n.tiles2 += j.n_tiles;
      }
    }
    of_class[cl].push_back(j);
  }
  S.n.one = (int)of_class[0].size();
  S.n.cluster = (int)of_class[1].size();
  for (int k = 0; k < 3; ++k)
    for (SysJob& j : of_class[k]) {
      if (j.need_low) j.sum_row = S.rows++;  // one sum row per system after the tile rows
      S.of_system[j.geom] = (int)S.jobs.size();
      S.jobs.push_back(j);
    }
}

// Mixed path: every computed moment job takes its degrees l <= 2 from its system's low sums (the float
// kernels have no values of their own for them).
int link_low(const SysPlan& S, Plan& P) {
  for (MomJob& j : P.jobs) {
    if (j.plan == 0) continue;
    const int si = S.of_system[j.geom];
    if (si < 0 || !S.jobs[si].need_low) return set_err(TCM_ECUDA, "internal: a float moment job without its low-degree sums");
    j.low_base = S.jobs[si].sum_row;
    j.low_tiles = 1;
  }
  return TCM_OK;
}

// Partial rows and tickets of the system pass; the tickets are zeroed when allocated and every
// launch leaves them zero.
int ensure_sys_buffers(tcm_ctx* c, const SysPlan& S, bool tiles_on_host) {
  if (S.jobs.empty()) return TCM_OK;
  TRY(dev_ensure(c, c->gpart, (size_t)std::max(S.rows, 1) * kSysPart * sizeof(double)));
  if (S.n.tiles1 + S.n.tiles2 == 0) return TCM_OK;
  void* before = c->systk.p;
  TRY(dev_ensure(c, c->systk, std::max<size_t>(2 * S.jobs.size(), 64) * sizeof(int)));
  if (c->systk.p != before) TRY_CUDA(cudaMemsetAsync(c->systk.p, 0, c->systk.cap, c->stream));
  if (!tiles_on_host) TRY(dev_ensure(c, c->systiles, (size_t)std::max(S.n.tiles1 + S.n.tiles2, 1) * sizeof(SysTile)));
  return TCM_OK;
}

// The tile lists of a call: written by the host into the descriptor block when they are short (a
// launch saved: about 4 us of a small call), else on the device from the groups and system jobs (long
// lists cost more to build and upload than the launch).
constexpr int kHostTiles = 2048;
struct Lists {
  bool on_host = false;
  std::vector<MomTile> mom;
  std::vector<SysTile> sys;  // pass 1, then pass 2
  size_t o_mom = 0, o_sys = 0;
  MomTile* d_mom = nullptr;
  SysTile* d_sys = nullptr;

  void plan(const Plan* P, const SysPlan& S, Packer& pk) {
    const int nm = P ? P->n_tiles : 0, ns = S.n.tiles1 + S.n.tiles2;
    on_host = nm + ns <= kHostTiles;
    o_mom = o_sys = 0;
    if (!on_host) return;
    mom.resize(nm);
    sys.resize(ns);
    if (P)
      for (const MomGroup& g : P->groups) {
        const MomJob& j = P->jobs[g.job];
        for (int t = 0; t < g.n; ++t)
          mom[g.first + t] = MomTile{g.job, g.chunk, t, part_row(j, g.chunk, t)};
      }
    for (int ji = 0; ji < (int)S.jobs.size(); ++ji) {
      const SysJob& j = S.jobs[ji];
      for (int t = 0; t < j.n_tiles; ++t) {
        if (j.first1 >= 0) sys[j.first1 + t] = SysTile{ji, t};
        if (j.first2 >= 0) sys[S.n.tiles1 + j.first2 + t] = SysTile{ji, t};
      }
    }
    o_mom = pk.add(mom);
    o_sys = pk.add(sys);
  }
  void place(tcm_ctx* c, char* base) {
    d_mom = on_host ? reinterpret_cast<MomTile*>(base + o_mom) : static_cast<MomTile*>(c->tiles.p);
    d_sys = on_host ? reinterpret_cast<SysTile*>(base + o_sys) : static_cast<SysTile*>(c->systiles.p);
  }
};

int run_sys(tcm_ctx* c, const SysPlan& S, const Lists& T, const SysJob* d_sj, SysGeom* d_geo, cudaStream_t st) {
  if (S.jobs.empty()) return TCM_OK;
  PhaseScope ps(c, TCM_PHASE_GEOM, sys_launches(S.n));
  TRY_LAUNCH(launch_sys(d_sj, S.n, T.d_sys, T.d_sys + S.n.tiles1, static_cast<double*>(c->gpart.p),
                        static_cast<int*>(c->systk.p), d_geo, true, st));
  return TCM_OK;
}

// Long tile lists, written on the device: the first launch of a call (it depends on nothing queued
// before it).
int run_expand(tcm_ctx* c, const std::vector<MomGroup>& groups, const MomJob* d_jobs, const MomGroup* d_groups,
               const SysPlan& S, const Lists& T, const SysJob* d_sj, cudaStream_t st) {
  if (T.on_host) return TCM_OK;
  PhaseScope ps(c, TCM_PHASE_GEOM, 1);
  TRY_LAUNCH(launch_expand_tiles(d_groups, (int)groups.size(), d_jobs, T.d_mom, d_sj, (int)S.jobs.size(), T.d_sys,
                                 T.d_sys + S.n.tiles1, st));
  return TCM_OK;
}

SysGeom host_geom(const tcm_system& s) {
  SysGeom g{};
  for (int d = 0; d < 3; ++d) {
    g.c[d] = s.has_center ? s.center[d] : 0.0;
    g.chi[d] = (float)g.c[d];
    g.clo[d] = (float)(g.c[d] - (double)g.chi[d]);
  }
  g.a = s.radius >= 0.0 ? s.radius : 0.0;
  return g;
}

void identity(double* r) {
  for (int k = 0; k < 9; ++k) r[k] = (k % 4 == 0) ? 1.0 : 0.0;
}

// Whether rot is a proper rotation to the rounding of a double: |R^T R - I| <= 3e-15 in every entry
// (matrices built from unit quaternions in double are within 1.6e-15, products of two within 2e-15)
// and det R > 0.
bool is_rotation(const double* R) {
  for (int i = 0; i < 3; ++i)
    for (int j = i; j < 3; ++j) {
      const double d = R[i] * R[j] + R[3 + i] * R[3 + j] + R[6 + i] * R[6 + j] - (i == j ? 1.0 : 0.0);
      if (!(std::fabs(d) <= 3e-15)) return false;
    }
  return R[0] * (R[4] * R[8] - R[5] * R[7]) - R[1] * (R[3] * R[8] - R[5] * R[6]) + R[2] * (R[3] * R[7] - R[4] * R[6]) > 0.0;
}

// Host tables --------------------------------------------------------------------

int build_tables(tcm_ctx* c) {
  std::vector<double> fmap;
  std::vector<int> imap_off, imap;
  finalize_tables(imap_off, imap, fmap);
  TRY_CUDA(cudaMalloc(&c->d_fmap, fmap.size() * sizeof(double)));
  TRY_CUDA(cudaMalloc(&c->d_imap, imap.size() * sizeof(int)));
  TRY_CUDA(cudaMalloc(&c->d_imap_off, imap_off.size() * sizeof(int)));
  TRY_CUDA(cudaMemcpy(c->d_fmap, fmap.data(), fmap.size() * sizeof(double), cudaMemcpyHostToDevice));
  TRY_CUDA(cudaMemcpy(c->d_imap, imap.data(), imap.size() * sizeof(int), cudaMemcpyHostToDevice));
  TRY_CUDA(cudaMemcpy(c->d_imap_off, imap_off.data(), imap_off.size() * sizeof(int), cudaMemcpyHostToDevice));
  const ContractTables& t = contract_tables();
  TRY_CUDA(cudaMalloc(&c->d_ctab, sizeof t));
  TRY_CUDA(cudaMemcpy(c->d_ctab, &t, sizeof t, cudaMemcpyHostToDevice));
  return TCM_OK;
}

void free_ctx(tcm_ctx* c) {
  if (!c) return;
  if (c->scratch) c->free_scratch(c->scratch);
  cudaStreamSynchronize(c->stream);
  cudaFree(c->d_fmap);
  cudaFree(c->d_ctab);
  cudaFree(c->d_imap);
  cudaFree(c->d_imap_off);
  for (DevBuf* b : {&c->desc, &c->partials, &c->gpart, &c->systk, &c->systiles, &c->counters, &c->moms, &c->escr,
                     &c->dpart, &c->tiles})
    cudaFree(b->p);
  for (auto& st : c->stage) {
    if (st.host) cudaFreeHost(st.host);
    if (st.ev) cudaEventDestroy(st.ev);
  }
  if (c->pinned_small) cudaFreeHost(c->pinned_small);
  for (auto& m : c->marks) {
    cudaEventDestroy(m.a);
    cudaEventDestroy(m.b);
  }
  for (auto e : c->ev_pool) cudaEventDestroy(e);
  if (c->gexec) cudaGraphExecDestroy(c->gexec);
  if (c->cap_stream) cudaStreamDestroy(c->cap_stream);
  delete c;
}

int check_ctx(tcm_ctx* c) {
  if (!c) return set_err(TCM_EINVAL, "null context");
  TRY_CUDA(cudaSetDevice(c->device));
  return TCM_OK;
}

}  // namespace

int tcm::record_error(int code, const char* msg) { return set_err(code, "%s", msg); }

extern "C" {

const char* tcm_last_error(void) { return g_err; }

int tcm_ctx_create(tcm_ctx_t* out, int lmax_cap, void* cuda_stream) {
  if (!out) return set_err(TCM_EINVAL, "tcm_ctx_create: null output pointer");
  *out = nullptr;
  if (lmax_cap < 0 || lmax_cap > TCM_LMAX_MAX)
    return set_err(TCM_EINVAL, "tcm_ctx_create: lmax_cap %d outside [0, %d]", lmax_cap, TCM_LMAX_MAX);
  tcm_ctx* c = new (std::nothrow) tcm_ctx();
  if (!c) return set_err(TCM_ENOMEM, "tcm_ctx_create: host allocation failed");
  for (int L = 0; L <= kLmaxMax; ++L) {
    c->atoms_per_thread[0][L] = 32;  // FP64: 32 atoms per lane (1,024 per warp tile)
    c->atoms_per_thread[1][L] = 64;  // mixed: 64 atoms per lane (2,048 per warp tile)
    c->ctas_per_sm[0][L] = c->ctas_per_sm[1][L] = TCM_MOMENT_CTAS_PER_SM;
    c->plan_l[L] = 1;
  }
  int rc = TCM_OK;
  do {
    if (cudaGetDevice(&c->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess) {
      rc = set_err(TCM_ECUDA, "tcm_ctx_create: no usable CUDA device: %s", cudaGetErrorString(cudaGetLastError()));
      break;
    }
    c->lmax_cap = lmax_cap;
    c->stream = static_cast<cudaStream_t>(cuda_stream);
    if ((rc = build_tables(c)) != TCM_OK) break;
    for (auto& st : c->stage)
      if (cudaEventCreateWithFlags(&st.ev, cudaEventDisableTiming) != cudaSuccess) {
        rc = set_err(TCM_ECUDA, "tcm_ctx_create: cudaEventCreate failed");
        break;
      }
    if (rc != TCM_OK) break;
    if (cudaHostAlloc(&c->pinned_small, 256, cudaHostAllocDefault) != cudaSuccess) {
      rc = set_err(TCM_ENOMEM, "tcm_ctx_create: cudaHostAlloc failed");
      break;
    }
    if (cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking) != cudaSuccess) {
      cudaGetLastError();
      c->cap_stream = nullptr;  // graphs unavailable; calls launch directly
    }
  } while (0);
  if (rc != TCM_OK) {
    free_ctx(c);
    return rc;
  }
  *out = c;
  return TCM_OK;
}

void tcm_ctx_destroy(tcm_ctx_t c) { free_ctx(c); }

int tcm_ctx_set_stream(tcm_ctx_t c, void* cuda_stream) {
  TRY(check_ctx(c));
  TRY_CUDA(cudaStreamSynchronize(c->stream));
  c->stream = static_cast<cudaStream_t>(cuda_stream);
  return TCM_OK;
}

int tcm_ctx_set_tiling(tcm_ctx_t c, int precision, int atoms_per_lane) {
  TRY(check_ctx(c));
  if (precision != TCM_FP64 && precision != TCM_MIXED) return set_err(TCM_EINVAL, "tcm_ctx_set_tiling: bad precision");
  if (atoms_per_lane < 1 || atoms_per_lane > 4096)
    return set_err(TCM_EINVAL, "tcm_ctx_set_tiling: atoms_per_lane outside [1, 4096]");
  for (int L = 0; L <= kLmaxMax; ++L) {
    c->atoms_per_thread[precision == TCM_FP64 ? 0 : 1][L] = atoms_per_lane;
    if (precision == TCM_FP64) c->tiling_set[L] = true;
  }
  ++c->cfg_gen;
  return TCM_OK;
}

int tcm_ctx_set_tiling_l(tcm_ctx_t c, int precision, int lmax, int atoms_per_lane, int ctas_per_sm) {
  TRY(check_ctx(c));
  if (precision != TCM_FP64 && precision != TCM_MIXED) return set_err(TCM_EINVAL, "tcm_ctx_set_tiling_l: bad precision");
  if (lmax < 0 || lmax > kLmaxMax) return set_err(TCM_EINVAL, "tcm_ctx_set_tiling_l: lmax outside [0, %d]", kLmaxMax);
  if (atoms_per_lane < 1 || atoms_per_lane > 4096)
    return set_err(TCM_EINVAL, "tcm_ctx_set_tiling_l: atoms_per_lane outside [1, 4096]");
  const int cmax = precision == TCM_FP64 ? TCM_MOMENT_CTAS_PER_SM : moment_ctas(kKmaxF32Small);
  if (ctas_per_sm < 1 || ctas_per_sm > cmax)
    return set_err(TCM_EINVAL, "tcm_ctx_set_tiling_l: ctas_per_sm outside [1, %d]", cmax);
  c->atoms_per_thread[precision == TCM_FP64 ? 0 : 1][lmax] = atoms_per_lane;
  c->ctas_per_sm[precision == TCM_FP64 ? 0 : 1][lmax] = ctas_per_sm;
  if (precision == TCM_FP64) c->tiling_set[lmax] = true;
  ++c->cfg_gen;
  return TCM_OK;
}

int tcm_ctx_get_tiling_l(tcm_ctx_t c, int precision, int lmax, int* atoms_per_lane, int* ctas_per_sm) {
  TRY(check_ctx(c));
  if (precision != TCM_FP64 && precision != TCM_MIXED) return set_err(TCM_EINVAL, "tcm_ctx_get_tiling_l: bad precision");
  if (lmax < 0 || lmax > kLmaxMax) return set_err(TCM_EINVAL, "tcm_ctx_get_tiling_l: lmax outside [0, %d]", kLmaxMax);
  if (atoms_per_lane) *atoms_per_lane = c->atoms_per_thread[precision == TCM_FP64 ? 0 : 1][lmax];
  if (ctas_per_sm) *ctas_per_sm = c->ctas_per_sm[precision == TCM_FP64 ? 0 : 1][lmax];
  return TCM_OK;
}

int tcm_ctx_set_chunking_l(tcm_ctx_t c, int lmax, int kmax) {
  TRY(check_ctx(c));
  if (lmax < 0 || lmax > kLmaxMax) return set_err(TCM_EINVAL, "tcm_ctx_set_chunking_l: lmax outside [0, %d]", kLmaxMax);
  if (kmax != plan_kmax(1) && kmax != plan_kmax(2))
    return set_err(TCM_EINVAL, "tcm_ctx_set_chunking_l: kmax %d is not %d or %d", kmax, plan_kmax(1), plan_kmax(2));
  c->plan_l[lmax] = kmax == plan_kmax(1) ? 1 : 2;
  ++c->cfg_gen;
  return TCM_OK;
}

int tcm_ctx_get_chunking_l(tcm_ctx_t c, int lmax, int* kmax, int* n_chunks) {
  TRY(check_ctx(c));
  if (lmax < 0 || lmax > kLmaxMax) return set_err(TCM_EINVAL, "tcm_ctx_get_chunking_l: lmax outside [0, %d]", kLmaxMax);
  if (kmax) *kmax = plan_kmax(c->plan_l[lmax]);
  if (n_chunks) *n_chunks = moments_nchunks(c->plan_l[lmax], lmax);
  return TCM_OK;
}

int tcm_ctx_set_graphs(tcm_ctx_t c, int mode) {
  TRY(check_ctx(c));
  if (mode < 0 || mode > 2) return set_err(TCM_EINVAL, "tcm_ctx_set_graphs: mode %d outside [0, 2]", mode);
  c->graphs = mode;
  return TCM_OK;
}

int tcm_ctx_graph_stats(tcm_ctx_t c, int64_t* captures, int64_t* launches) {
  TRY(check_ctx(c));
  if (captures) *captures = c->graph_captures;
  if (launches) *launches = c->graph_launches;
  return TCM_OK;
}

int tcm_ctx_set_profiling(tcm_ctx_t c, int enable) {
  TRY(check_ctx(c));
  c->prof = enable != 0;
  return TCM_OK;
}

int tcm_ctx_read_profile(tcm_ctx_t c, double* ms, int64_t* launches) {
  TRY(check_ctx(c));
  TRY_CUDA(cudaStreamSynchronize(c->stream));
  double acc[TCM_NPHASES] = {};
  acc[TCM_PHASE_HOST] = c->host_ms;
  c->host_ms = 0.0;
  for (auto& m : c->marks) {
    float t = 0.0f;
    if (cudaEventElapsedTime(&t, m.a, m.b) == cudaSuccess) acc[m.phase] += t;
    c->ev_pool.push_back(m.a);
    c->ev_pool.push_back(m.b);
  }
  c->marks.clear();
  for (int k = 0; k < TCM_NPHASES; ++k) {
    if (ms) ms[k] = acc[k];
    if (launches) launches[k] = c->launches[k];
    c->launches[k] = 0;
  }
  return TCM_OK;
}

int tcm_prepare(tcm_ctx_t c, tcm_system* s) try {
  TRY(check_ctx(c));
  TRY(check_system(s, "tcm_prepare"));
  if (geom_known(*s)) return TCM_OK;
  std::vector<char> used(1, 1);
  SysPlan S;
  plan_sys(s, 1, used, {}, S);
  std::vector<SysGeom> geoms{host_geom(*s)};
  Packer pk;
  const size_t o_geo = pk.add(geoms), o_sj = pk.add(S.jobs);
  Lists T;
  T.plan(nullptr, S, pk);
  TRY(ensure_sys_buffers(c, S, T.on_host));
  char* base = nullptr;
  TRY(upload(c, pk, &base));
  SysGeom* d_geo = reinterpret_cast<SysGeom*>(base + o_geo);
  const SysJob* d_sj = reinterpret_cast<SysJob*>(base + o_sj);
  T.place(c, base);
  TRY(run_expand(c, {}, nullptr, nullptr, S, T, d_sj, c->stream));
  TRY(run_sys(c, S, T, d_sj, d_geo, c->stream));
  TRY_CUDA(cudaMemcpyAsync(c->pinned_small, d_geo, sizeof(SysGeom), cudaMemcpyDeviceToHost, c->stream));
  TRY_CUDA(cudaStreamSynchronize(c->stream));
  const SysGeom* g = static_cast<const SysGeom*>(c->pinned_small);
  for (int d = 0; d < 3; ++d) s->center[d] = g->c[d];
  s->has_center = 1;
  s->radius = g->a;
  return TCM_OK;
} catch (const std::exception&) {
  return no_host_memory("tcm_prepare");
}

int tcm_moments(tcm_ctx_t c, const tcm_system* s, const double* rot, int lmax, int precision, tcm_moments_t* out) try {
  TRY(check_ctx(c));
  TRY(check_system(s, "tcm_moments"));
  if (!out || !out->q) return set_err(TCM_EINVAL, "tcm_moments: null output");
  if (!aligned16(out->q)) return set_err(TCM_EINVAL, "tcm_moments: output must be 16-byte aligned");
  if (lmax < 0 || lmax > c->lmax_cap)
    return set_err(TCM_EINVAL, "tcm_moments: lmax %d outside [0, %d]", lmax, c->lmax_cap);
  if (precision != TCM_FP64 && precision != TCM_MIXED) return set_err(TCM_EINVAL, "tcm_moments: bad precision");
  Plan P;
  MomJob j{};
  j.xyzq = s->xyzq;
  j.n = s->n;
  j.dtype = s->dtype;
  j.L = lmax;
  j.geom = 0;
  if (rot)
    std::memcpy(j.rot, rot, 9 * sizeof(double));
  else
    identity(j.rot);
  j.out = out->q;
  int next = 0;
  plan_job(c, precision, j, next);
  P.jobs.push_back(j);
  P.n_tile_ids = next;
  build_tiles(precision, P);
  std::vector<char> used(1, 1), low(1, precision == TCM_MIXED ? 1 : 0);
  SysPlan S;
  plan_sys(s, 1, used, low, S);
  TRY(link_low(S, P));
  std::vector<SysGeom> geoms{host_geom(*s)};
  Packer pk;
  const size_t o_geo = pk.add(geoms), o_job = pk.add(P.jobs), o_tile = pk.add(P.groups), o_sj = pk.add(S.jobs);
  Lists T;
  T.plan(&P, S, pk);
  TRY(ensure_moment_buffers(c, P, T.on_host));
  TRY(ensure_sys_buffers(c, S, T.on_host));
  char* base = nullptr;
  TRY(upload(c, pk, &base));
  SysGeom* d_geo = reinterpret_cast<SysGeom*>(base + o_geo);
  const SysJob* d_sj = reinterpret_cast<SysJob*>(base + o_sj);
  T.place(c, base);
  TRY(run_expand(c, P.groups, reinterpret_cast<MomJob*>(base + o_job), reinterpret_cast<MomGroup*>(base + o_tile), S, T,
                 d_sj, c->stream));
  TRY(run_sys(c, S, T, d_sj, d_geo, c->stream));
  TRY(run_moments(c, precision, P, reinterpret_cast<MomJob*>(base + o_job), T.d_mom, d_geo, c->stream));
  out->lmax = lmax;
  if (!geom_known(*s)) {
    TRY_CUDA(cudaMemcpyAsync(c->pinned_small, d_geo, sizeof(SysGeom), cudaMemcpyDeviceToHost, c->stream));
    TRY_CUDA(cudaStreamSynchronize(c->stream));
    const SysGeom* g = static_cast<const SysGeom*>(c->pinned_small);
    for (int d = 0; d < 3; ++d) out->center[d] = g->c[d];
    out->radius = g->a;
  } else {
    for (int d = 0; d < 3; ++d) out->center[d] = s->center[d];
    out->radius = s->radius;
  }
  return TCM_OK;
} catch (const std::exception&) {
  return no_host_memory("tcm_moments");
}

int tcm_energy(tcm_ctx_t c, const tcm_moments_t* A, const tcm_moments_t* B, const double* R0, int lmax, double* E) try {
  TRY(check_ctx(c));
  if (!A || !B || !R0 || !E || !A->q || !B->q) return set_err(TCM_EINVAL, "tcm_energy: null argument");
  if (lmax < 0 || lmax > c->lmax_cap || lmax > A->lmax || lmax > B->lmax)
    return set_err(TCM_EINVAL, "tcm_energy: lmax %d exceeds the moments' lmax or the context cap", lmax);
  const double R = std::sqrt(R0[0] * R0[0] + R0[1] * R0[1] + R0[2] * R0[2]);
  if (!(R > A->radius + B->radius))
    return set_err(TCM_ENOTCONV, "tcm_energy: |R0| = %.17g <= a_A + a_B = %.17g (Eq. (mainCond))", R,
                   A->radius + B->radius);
  std::vector<MomJob> jobs(2);
  std::memset(jobs.data(), 0, 2 * sizeof(MomJob));
  jobs[0].out = A->q;
  jobs[0].L = A->lmax;
  jobs[1].out = B->q;
  jobs[1].L = B->lmax;
  std::vector<SysGeom> geoms(2);
  std::memset(geoms.data(), 0, 2 * sizeof(SysGeom));
  geoms[0].a = A->radius;
  geoms[1].a = B->radius;
  std::vector<PairDesc> items(1);
  make_pair(PairRun{0, 0, 1, 0, 1, (short)lmax, kBLab, 0}, 0, R0, 2, nullptr, items[0], nullptr);
  TRY(dev_ensure(c, c->escr, 64));
  double* dE = static_cast<double*>(c->escr.p);
  std::vector<PairOut> out{PairOut{dE, nullptr, nullptr}};
  std::vector<ContractPlan> plan(1);
  for (int L = 0; L <= kLmaxMax + 1; ++L) plan[0].first[L] = plan[0].gfirst[L] = L > lmax;
  Packer pk;
  const size_t o_job = pk.add(jobs), o_geo = pk.add(geoms), o_it = pk.add(items), o_out = pk.add(out), o_plan = pk.add(plan);
  char* base = nullptr;
  TRY(upload(c, pk, &base));
  {
    PhaseScope ps(c, TCM_PHASE_CONTRACT, 1);
    TRY_LAUNCH(launch_contract(reinterpret_cast<PairDesc*>(base + o_it), nullptr,
                               reinterpret_cast<ContractPlan*>(base + o_plan), 1, lmax,
                               reinterpret_cast<MomJob*>(base + o_job), reinterpret_cast<SysGeom*>(base + o_geo),
                               c->d_ctab, nullptr, reinterpret_cast<PairOut*>(base + o_out), false, true, c->num_sms,
                               c->stream));
  }
  TRY_CUDA(cudaMemcpyAsync(c->pinned_small, dE, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  TRY_CUDA(cudaStreamSynchronize(c->stream));
  *E = *static_cast<const double*>(c->pinned_small);
  return TCM_OK;
} catch (const std::exception&) {
  return no_host_memory("tcm_energy");
}

int tcm_rotate_moments(tcm_ctx_t c, int64_t n, const tcm_moments_t* in, const double* rot, tcm_moments_t* out) try {
  TRY(check_ctx(c));
  if (n < 0) return set_err(TCM_EINVAL, "tcm_rotate_moments: negative count");
  if (n == 0) return TCM_OK;
  if (!in || !rot || !out) return set_err(TCM_EINVAL, "tcm_rotate_moments: null argument");
  if (n > (1LL << 30)) return set_err(TCM_EINVAL, "tcm_rotate_moments: too many sets");
  std::vector<RotDesc> sets(n);
  int Lmax = 0;
  for (int64_t i = 0; i < n; ++i) {
    if (!in[i].q || !out[i].q) return set_err(TCM_EINVAL, "tcm_rotate_moments: set %lld has a null moment pointer", (long long)i);
    if (out[i].lmax < 0 || out[i].lmax > c->lmax_cap || out[i].lmax > in[i].lmax)
      return set_err(TCM_EINVAL, "tcm_rotate_moments: set %lld: output lmax %d outside [0, min(input lmax %d, cap %d)]",
                     (long long)i, out[i].lmax, in[i].lmax, c->lmax_cap);
    for (int k = 0; k < 9; ++k)
      if (!std::isfinite(rot[9 * i + k])) return set_err(TCM_EINVAL, "tcm_rotate_moments: set %lld: non-finite rotation", (long long)i);
    sets[i].in = in[i].q;
    sets[i].out = out[i].q;
    sets[i].L = out[i].lmax;
    std::memcpy(sets[i].M, rot + 9 * i, 9 * sizeof(double));
    Lmax = std::max(Lmax, out[i].lmax);
    for (int d = 0; d < 3; ++d) out[i].center[d] = in[i].center[d];
    out[i].radius = in[i].radius;
  }
  Packer pk;
  const size_t o_set = pk.add(sets);
  char* base = nullptr;
  TRY(upload(c, pk, &base));
  PhaseScope ps(c, TCM_PHASE_CONTRACT, 1);
  TRY_LAUNCH(launch_rotate_moments(reinterpret_cast<RotDesc*>(base + o_set), (int)n, Lmax, c->d_ctab->dpi2, c->stream));
  return TCM_OK;
} catch (const std::exception&) {
  return no_host_memory("tcm_rotate_moments");
}

int tcm_ctx_set_rotate_cached(tcm_ctx_t c, int enable) {
  TRY(check_ctx(c));
  c->rotate_cached = enable != 0;
  return TCM_OK;
}

namespace {
int energy_batch(tcm_ctx_t c, int n_systems, const tcm_system* systems, int64_t n_items, const tcm_pair_item* items,
                 int precision, double* E, int32_t* status, double* G);
}

namespace {
// The batched call, with its host wall time added to TCM_PHASE_HOST while profiling is on.
int timed_batch(tcm_ctx_t c, int n_systems, const tcm_system* systems, int64_t n_items, const tcm_pair_item* items,
                int precision, double* E, int32_t* status, double* G) {
  const auto t0 = std::chrono::steady_clock::now();
  int rc;
  try {
    rc = energy_batch(c, n_systems, systems, n_items, items, precision, E, status, G);
  } catch (const std::exception&) {
    rc = no_host_memory("tcm_energy_batch");
  }
  if (c && c->prof) c->host_ms += std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  return rc;
}
}  // namespace

int tcm_energy_batch(tcm_ctx_t c, int n_systems, const tcm_system* systems, int64_t n_items, const tcm_pair_item* items,
                     int precision, double* E, int32_t* status) {
  return timed_batch(c, n_systems, systems, n_items, items, precision, E, status, nullptr);
}

int tcm_gradients_batch(tcm_ctx_t c, int n_systems, const tcm_system* systems, int64_t n_items,
                        const tcm_pair_item* items, int precision, double* E, double* G, int32_t* status) {
  if (n_items > 0 && !G) return set_err(TCM_EINVAL, "tcm_gradients_batch: null gradient output");
  return timed_batch(c, n_systems, systems, n_items, items, precision, E, status, G);
}

namespace {
// Items from which their descriptors are made on the device.
constexpr int64_t kDeviceFrames = 128;

// Host arrays of the batched calls (one context, one thread at a time): cleared, not freed, between calls,
// and lookups stamped with the call's epoch instead of being cleared.
struct BatchScratch {
  Plan P;
  SysPlan S;
  Lists T;
  std::vector<PairRun> runs;
  std::vector<double> R0;
  std::vector<PairDesc> pd;
  std::vector<EulerZYZ> rots;
  std::vector<double> rotB;
  std::vector<MomJob> cached;
  std::vector<size_t> job_moff;
  std::vector<SysGeom> geoms;
  std::vector<PairOut> out;
  std::vector<ContractPlan> plan;
  std::vector<int> order;
  int count[kLmaxMax + 1];  // items per degree
  std::vector<char> used, low;
  std::vector<uint64_t> job_of, cached_of;  // epoch << 32 | index, by (system, degree) and by system
  uint32_t epoch = 0;
  std::vector<long long> key;

  void begin(int n_systems) {
    if (++epoch == 0) {  // wrapped: no stamp of the past may match
      std::fill(job_of.begin(), job_of.end(), 0);
      std::fill(cached_of.begin(), cached_of.end(), 0);
      epoch = 1;
    }
    if (job_of.size() < (size_t)n_systems * (kLmaxMax + 1)) job_of.resize((size_t)n_systems * (kLmaxMax + 1), 0);
    if (cached_of.size() < (size_t)n_systems) cached_of.resize(n_systems, 0);
    used.assign(n_systems, 0);
    low.assign(n_systems, 0);
    P.jobs.clear();
    rotB.clear();
    runs.clear();
    cached.clear();
    job_moff.clear();
  }
};

int energy_batch(tcm_ctx_t c, int n_systems, const tcm_system* systems, int64_t n_items, const tcm_pair_item* items,
                 int precision, double* E, int32_t* status, double* G) {
  TRY(check_ctx(c));
  if (n_items < 0 || n_systems < 0) return set_err(TCM_EINVAL, "tcm_energy_batch: negative count");
  if (n_items == 0) return TCM_OK;
  if (!systems || !items || !E) return set_err(TCM_EINVAL, "tcm_energy_batch: null argument");
  if (n_items > (1LL << 30)) return set_err(TCM_EINVAL, "tcm_energy_batch: too many items");
  if (precision != TCM_FP64 && precision != TCM_MIXED) return set_err(TCM_EINVAL, "tcm_energy_batch: bad precision");
  if (!c->scratch) {
    c->scratch = new BatchScratch;
    c->free_scratch = [](BatchScratch* s) { delete s; };
  }
  BatchScratch& B = *c->scratch;
  B.begin(n_systems);
  Plan& P = B.P;
  // Large batches: the items' descriptors are made on the device (k_frames) from runs of items and the
  // separations, which are written straight into the staging slot; small ones on the host (a launch costs
  // more than their square roots).
  const bool on_device = n_items >= kDeviceFrames;
  double* R0s = nullptr;
  size_t in_place = 0;
  if (on_device) {
    in_place = (size_t)n_items * 3 * sizeof(double);
    Stage* st = nullptr;
    TRY(stage_slot(c, in_place + in_place / 4 + 65536, 0, &st));
    R0s = static_cast<double*>(st->host);
  } else {
    B.R0.resize(3 * n_items);
    R0s = B.R0.data();
  }
  // One pass over the items: checks, moment jobs (A sides and unrotated B sides shared), records.
  int next_id = 0, Lmax_items = 0;
  std::fill(B.count, B.count + kLmaxMax + 1, 0);
  bool sorted = true;  // degrees never fall from item to item
  size_t moff = 0;
  auto new_job = [&](int sys, int L, const double* rot) {
    P.jobs.emplace_back();
    MomJob& j = P.jobs.back();
    j = MomJob{};
    j.xyzq = systems[sys].xyzq;
    j.n = systems[sys].n;
    j.dtype = systems[sys].dtype;
    j.L = L;
    j.geom = sys;
    if (rot)
      std::memcpy(j.rot, rot, 9 * sizeof(double));
    else
      identity(j.rot);
    plan_job(c, precision, j, next_id);
    B.job_moff.push_back(moff);
    moff += (size_t)(L + 1) * (L + 1);
    return (int)P.jobs.size() - 1;
  };
  // the unrotated set of (system, L): from the system's moment cache (~index) or computed (index)
  auto unrotated = [&](int sys, int L, bool use_cache) {
    const tcm_system& sy = systems[sys];
    if (use_cache && sy.moments && L <= sy.moments_lmax) {
      uint64_t& e = B.cached_of[sys];
      if ((e >> 32) != B.epoch) {
        MomJob j{};
        j.L = sy.moments_lmax;
        j.geom = sys;
        j.out = const_cast<double*>(sy.moments);
        e = (uint64_t)B.epoch << 32 | (uint32_t)B.cached.size();
        B.cached.push_back(j);
      }
      return ~(int)(uint32_t)e;
    }
    uint64_t& e = B.job_of[(size_t)sys * (kLmaxMax + 1) + L];
    if ((e >> 32) != B.epoch) e = (uint64_t)B.epoch << 32 | (uint32_t)new_job(sys, L, nullptr);
    return (int)(uint32_t)e;
  };
  int64_t nc_item = -1;  // first item that a host-known radius shows not to converge
  double nc_R = 0.0, nc_a = 0.0;
  // B's moments of a rotated item, in its frame, in the contraction:
  //   from_cache  the caller asked for it and B carries its moments: the cached set, rotated by W rotB;
  //   from_lab    double path: B's lab-frame set, computed once per (system, degree) from B's atoms and
  //               shared by all items and by unrotated sides, rotated by W rotB.  The moments of a rotated
  //               system are those of the system, rotated degree by degree (exact; O(L^3) operations
  //               against O(atoms L^2)): 256 orientations of 20,000 atoms at degree 20 take 0.16 ms
  //               instead of 13 ms, at the same error.  Only for matrices that are rotations to rounding;
  //   else        a set of the item's own, the frame rotation W folded into its atom transform: any other
  //               matrix of the double path, and the mixed path, which keeps each item's own float sums
  //               over the rotated atoms, whose rounding errors are independent.
  int last_L = 0;
  for (int64_t k = 0; k < n_items;) {
    const tcm_pair_item& it = items[k];
    if (it.a < 0 || it.a >= n_systems || it.b < 0 || it.b >= n_systems)
      return set_err(TCM_EINVAL, "tcm_energy_batch: item %lld refers to a system outside [0, %d)", (long long)k, n_systems);
    if (it.lmax < 0 || it.lmax > c->lmax_cap)
      return set_err(TCM_EINVAL, "tcm_energy_batch: item %lld lmax %d outside [0, %d]", (long long)k, it.lmax, c->lmax_cap);
    const int ia = it.a, ib = it.b, L = it.lmax, has_rot = it.has_rot != 0;
    const tcm_system &sa = systems[ia], &sb = systems[ib];
    B.used[ia] = B.used[ib] = 1;
    const bool known = geom_known(sa) && geom_known(sb);  // both radii known on the host
    const double aa = sa.radius + sb.radius, near2 = aa * aa * (1.0 + 1e-12);
    const bool from_cache = has_rot && c->rotate_cached && sb.moments && L <= sb.moments_lmax;
    const bool lab = has_rot && !from_cache && precision == TCM_FP64;
    auto mode_of = [&](const tcm_pair_item& x) {
      return !has_rot ? kBLab : (from_cache || (lab && is_rotation(x.rotB)) ? kBRotate : kBInFrame);
    };
    const int mode = mode_of(it);
    PairRun r{(int)k, unrotated(ia, L, true), 0, ia, ib, (short)L, (short)mode, (int)(B.rotB.size() / 9)};
    if (mode != kBInFrame) r.jobB = unrotated(ib, L, mode == kBLab || from_cache);
    else r.jobB = (int)P.jobs.size();
    int64_t e = k;
    for (; e < n_items; ++e) {
      const tcm_pair_item& x = items[e];
      if (x.a != ia || x.b != ib || x.lmax != L || (x.has_rot != 0) != (has_rot != 0)) break;
      if (lab && e > k && mode_of(x) != mode) break;
      const double x0 = x.R0[0], x1 = x.R0[1], x2 = x.R0[2];
      R0s[3 * e] = x0;
      R0s[3 * e + 1] = x1;
      R0s[3 * e + 2] = x2;
      if (known) {
        const double R2 = x0 * x0 + x1 * x1 + x2 * x2;
        if (!(R2 > near2) && nc_item < 0) {  // (the square root only near the limit)
          const double R = std::sqrt(R2);
          if (!(R > aa)) {
            nc_item = e;
            nc_R = R;
            nc_a = aa;
          }
        }
      }
      if (mode == kBRotate) {
        B.rotB.insert(B.rotB.end(), x.rotB, x.rotB + 9);
      } else if (mode == kBInFrame) {
        double fr[6], M[9];
        r0_frame(x.R0, fr);
        frame_times(fr, x.rotB, M);
        new_job(ib, L, M);
      }
    }
    B.runs.push_back(r);
    B.count[L] += (int)(e - k);
    sorted = sorted && L >= last_L;
    last_L = L;
    Lmax_items = std::max(Lmax_items, L);
    k = e;
  }
  for (int s = 0; s < n_systems; ++s)
    if (B.used[s]) TRY(check_system(&systems[s], "tcm_energy_batch"));
  if (nc_item >= 0)  // rejected before any work is queued
    return set_err(TCM_ENOTCONV, "tcm_energy_batch: item %lld: |R0| = %.17g <= a_A + a_B = %.17g (Eq. (mainCond))",
                   (long long)nc_item, nc_R, nc_a);
  P.n_tile_ids = next_id;
  TRY(dev_ensure(c, c->moms, std::max<size_t>(moff, 1) * sizeof(double)));
  for (size_t ji = 0; ji < P.jobs.size(); ++ji) P.jobs[ji].out = static_cast<double*>(c->moms.p) + B.job_moff[ji];
  build_tiles(precision, P);
  if (precision == TCM_MIXED)
    for (const MomJob& j : P.jobs) B.low[j.geom] = 1;
  SysPlan& S = B.S;
  plan_sys(systems, n_systems, B.used, B.low, S);
  TRY(link_low(S, P));
  const int n_computed = (int)P.jobs.size();  // cached sides follow them in the descriptor array (not finalised)
  const int n_rot = (int)(B.rotB.size() / 9);
  B.geoms.resize(std::max(n_systems, 1));
  for (int s = 0; s < n_systems; ++s) B.geoms[s] = host_geom(systems[s]);
  B.out.assign(1, PairOut{E, status, G});
  // the contraction's order: items by degree, in place when there is one degree only
  B.plan.resize(1);
  ContractPlan& cp = B.plan[0];
  int n_groups = 0, at = 0;
  for (int L = 0; L <= kLmaxMax + 1; ++L) {
    cp.first[L] = at;
    cp.gfirst[L] = n_groups;
    if (L > kLmaxMax) break;
    at += B.count[L];
    n_groups += (B.count[L] + contract_group(L) - 1) / contract_group(L);
  }
  const bool ordered = !sorted;
  B.order.clear();
  if (ordered) {
    int next[kLmaxMax + 1];
    std::copy(cp.first, cp.first + kLmaxMax + 1, next);
    B.order.resize(n_items);
    for (size_t r = 0; r < B.runs.size(); ++r) {
      const int end = r + 1 < B.runs.size() ? B.runs[r + 1].first : (int)n_items;
      for (int k = B.runs[r].first; k < end; ++k) B.order[next[B.runs[r].L]++] = k;
    }
  }
  Packer pk;
  pk.size = in_place;
  const size_t o_geo = pk.add(B.geoms), o_job = pk.add2(P.jobs, B.cached), o_tile = pk.add(P.groups),
               o_sj = pk.add(S.jobs), o_out = pk.add(B.out), o_plan = pk.add(B.plan), o_ord = pk.add(B.order);
  size_t o_it = 0, o_rot = 0, o_run = 0;
  const int n_runs = (int)B.runs.size();
  if (on_device) {
    o_run = pk.add(B.runs);
    o_rot = pk.add(B.rotB);
  } else {
    B.pd.resize(n_items);
    B.rots.resize(n_rot);
    for (int r = 0; r < n_runs; ++r) {
      const int end = r + 1 < n_runs ? B.runs[r + 1].first : (int)n_items;
      for (int k = B.runs[r].first; k < end; ++k)
        make_pair(B.runs[r], k, R0s + 3 * k, n_computed, B.rotB.data(), B.pd[k], B.rots.data());
    }
    o_it = pk.add(B.pd);
    o_rot = pk.add(B.rots);
  }
  Lists& T = B.T;
  T.plan(&P, S, pk);
  // every buffer the launches touch is sized before anything is queued (no reallocation
  // may happen while a graph is being captured)
  TRY(ensure_sys_buffers(c, S, T.on_host));
  TRY(ensure_moment_buffers(c, P, T.on_host));
  char* base = nullptr;
  TRY(upload(c, pk, &base, in_place,
             on_device ? (size_t)n_items * sizeof(PairDesc) + (size_t)n_rot * sizeof(EulerZYZ) : 0));
  SysGeom* d_geo = reinterpret_cast<SysGeom*>(base + o_geo);
  const MomJob* d_jobs = reinterpret_cast<MomJob*>(base + o_job);
  T.place(c, base);
  PairDesc* d_items = reinterpret_cast<PairDesc*>(base + (on_device ? align_up(pk.size) : o_it));
  EulerZYZ* d_rots = on_device ? reinterpret_cast<EulerZYZ*>(d_items + n_items) : reinterpret_cast<EulerZYZ*>(base + o_rot);
  const bool no_moments = P.jobs.empty() && S.jobs.empty();
  auto enqueue = [&](cudaStream_t st) -> int {
    const SysJob* d_sj = reinterpret_cast<SysJob*>(base + o_sj);
    TRY(run_expand(c, P.groups, d_jobs, reinterpret_cast<MomGroup*>(base + o_tile), S, T, d_sj, st));
    if (on_device) {
      PhaseScope ps(c, TCM_PHASE_GEOM, 1);
      TRY_LAUNCH(launch_frames(reinterpret_cast<PairRun*>(base + o_run), n_runs, reinterpret_cast<double*>(base),
                               (int)n_items, n_computed, reinterpret_cast<double*>(base + o_rot), d_items, d_rots, st));
    }
    TRY(run_sys(c, S, T, d_sj, d_geo, st));
    TRY(run_moments(c, precision, P, d_jobs, T.d_mom, d_geo, st));
    PhaseScope ps(c, TCM_PHASE_CONTRACT, 1);
    // (directly behind k_frames the contraction must not read the descriptors ahead of its end)
    TRY_LAUNCH(launch_contract(d_items, ordered ? reinterpret_cast<int*>(base + o_ord) : nullptr,
                               reinterpret_cast<ContractPlan*>(base + o_plan), n_groups, Lmax_items, d_jobs, d_geo,
                               c->d_ctab, n_rot ? d_rots : nullptr, reinterpret_cast<PairOut*>(base + o_out),
                               G != nullptr, !(on_device && no_moments), c->num_sms, st));
    return TCM_OK;
  };
  if (!c->graphs || c->prof || !c->cap_stream) return enqueue(c->stream);
  // Replay a captured graph of the launch sequence when this call has the same shape and
  // buffers as the captured one (only the uploaded descriptor contents differ).
  const bool cols = precision == TCM_MIXED && moments_use_cols(P.n_tiles, c->num_sms);
  std::vector<long long>& key = B.key;
  key = {precision, (long long)P.passes.size(), cols ? max_cols_of(P, 1) : 0, cols ? max_cols_of(P, 2) : 0, G != nullptr, S.n.one,
         S.n.cluster, S.n.tiles1, S.n.tiles2, (long long)S.jobs.size(), (long long)T.o_mom, (long long)T.o_sys, T.on_host,
         (long long)P.jobs.size(), P.n_tile_ids, (long long)n_items, n_rot, Lmax_items, (long long)o_geo, (long long)o_job,
         (long long)o_tile, (long long)o_sj, (long long)o_it, (long long)o_rot, (long long)o_out,
         n_groups, ordered, (long long)o_ord, (long long)o_run, n_runs,
         (long long)pk.size, (long long)(uintptr_t)c->systiles.p, (long long)(uintptr_t)base,
         (long long)(uintptr_t)c->gpart.p, (long long)(uintptr_t)c->systk.p, (long long)(uintptr_t)c->partials.p,
         (long long)(uintptr_t)c->counters.p, (long long)P.groups.size(), (long long)P.n_tiles,
         (long long)(uintptr_t)c->tiles.p, (long long)c->cfg_gen};
  for (const Plan::Pass& pass : P.passes) {
    key.push_back(pass.job0);
    key.push_back(split_of(P, pass));
    key.insert(key.end(), pass.tile_begin, pass.tile_begin + kLmaxMax + 2);
  }
  if (!c->gexec || key != c->gkey) {
    // by default capture only a shape seen twice in a row: a stream of changing shapes
    // (continuous batching) launches directly instead of paying a capture per call
    if (c->graphs == 1 && key != c->gkey_seen) {
      c->gkey_seen = key;
      return enqueue(c->stream);
    }
    if (c->gexec) {
      cudaGraphExecDestroy(c->gexec);
      c->gexec = nullptr;
    }
    TRY_CUDA(cudaStreamBeginCapture(c->cap_stream, cudaStreamCaptureModeThreadLocal));
    int64_t saved[TCM_NPHASES];
    std::copy(c->launches, c->launches + TCM_NPHASES, saved);
    const int rc = enqueue(c->cap_stream);
    for (int k = 0; k < TCM_NPHASES; ++k) c->launches[k] = saved[k];
    cudaGraph_t g = nullptr;
    const cudaError_t ec = cudaStreamEndCapture(c->cap_stream, &g);
    if (rc != TCM_OK || ec != cudaSuccess) {
      if (g) cudaGraphDestroy(g);
      cudaGetLastError();
      return rc != TCM_OK ? rc : set_err(TCM_ECUDA, "graph capture failed: %s", cudaGetErrorString(ec));
    }
    const cudaError_t ei = cudaGraphInstantiate(&c->gexec, g, 0);
    cudaGraphDestroy(g);
    if (ei != cudaSuccess) {
      c->gexec = nullptr;
      return set_err(TCM_ECUDA, "cudaGraphInstantiate: %s", cudaGetErrorString(ei));
    }
    c->gkey = key;
    ++c->graph_captures;
  }
  TRY_CUDA(cudaGraphLaunch(c->gexec, c->stream));
  ++c->graph_launches;
  c->launches[TCM_PHASE_GEOM] += sys_launches(S.n) + !T.on_host + on_device;
  c->launches[TCM_PHASE_MOMENTS] += moment_launches(precision, P);
  c->launches[TCM_PHASE_FINALIZE] += (int64_t)P.passes.size();
  c->launches[TCM_PHASE_CONTRACT] += 1;
  return TCM_OK;
}
}  // namespace

namespace {
// Eq. (Coulomb) for n items (B rotated by rotB[9 k] about its centre, at separation R0[3 k]);
// energies to the device array dE.  Asynchronous.
int direct_items(tcm_ctx_t c, const tcm_system* A, const tcm_system* B, int64_t n, const double* rotB,
                 const double* R0, double* dE) {
  // the radii choose the form of the pair loop and its scales (direct.cu): computed unless given
  tcm_system sys[2] = {*A, *B};
  std::vector<char> used(2, 1);
  SysPlan S;
  plan_sys(sys, 2, used, {}, S);
  std::vector<SysGeom> geoms{host_geom(sys[0]), host_geom(sys[1])};
  std::vector<double> xf(12 * (size_t)n);
  for (int64_t k = 0; k < n; ++k) {
    if (rotB)
      std::memcpy(&xf[12 * k], rotB + 9 * k, 9 * sizeof(double));
    else
      identity(&xf[12 * k]);
    for (int d = 0; d < 3; ++d) xf[12 * k + 9 + d] = R0[3 * k + d];
  }
  Packer pk;
  const size_t o_geo = pk.add(geoms), o_xf = pk.add(xf), o_sj = pk.add(S.jobs);
  Lists T;
  T.plan(nullptr, S, pk);
  const DirectSplit split = direct_split(A->n, B->n);
  TRY(ensure_sys_buffers(c, S, T.on_host));
  TRY(dev_ensure(c, c->dpart, (size_t)std::max<int64_t>((int64_t)split.parts * std::min<int64_t>(n, split.slab), 1) * sizeof(double)));
  char* base = nullptr;
  TRY(upload(c, pk, &base));
  SysGeom* d_geo = reinterpret_cast<SysGeom*>(base + o_geo);
  const SysJob* d_sj = reinterpret_cast<SysJob*>(base + o_sj);
  T.place(c, base);
  TRY(run_expand(c, {}, nullptr, nullptr, S, T, d_sj, c->stream));
  TRY(run_sys(c, S, T, d_sj, d_geo, c->stream));
  const int nlaunch = (int)((n + split.slab - 1) / split.slab) * (split.parts > 0 ? 2 : 1);
  PhaseScope ps(c, TCM_PHASE_DIRECT, nlaunch);
  TRY_LAUNCH(launch_direct(A->xyzq, A->n, A->dtype, B->xyzq, B->n, B->dtype, d_geo,
                           reinterpret_cast<double*>(base + o_xf), (int)n, static_cast<double*>(c->dpart.p), split, dE,
                           c->stream));
  return TCM_OK;
}
}  // namespace

int tcm_direct(tcm_ctx_t c, const tcm_system* A, const tcm_system* B, const double* rotB, const double* R0, double* E) try {
  TRY(check_ctx(c));
  TRY(check_system(A, "tcm_direct A"));
  TRY(check_system(B, "tcm_direct B"));
  if (!R0 || !E) return set_err(TCM_EINVAL, "tcm_direct: null argument");
  TRY(dev_ensure(c, c->escr, 64));
  double* dE = static_cast<double*>(c->escr.p);
  TRY(direct_items(c, A, B, 1, rotB, R0, dE));
  TRY_CUDA(cudaMemcpyAsync(c->pinned_small, dE, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  TRY_CUDA(cudaStreamSynchronize(c->stream));
  *E = *static_cast<const double*>(c->pinned_small);
  return TCM_OK;
} catch (const std::exception&) {
  return no_host_memory("tcm_direct");
}

int tcm_direct_batch(tcm_ctx_t c, const tcm_system* A, const tcm_system* B, int64_t n_items, const double* rotB,
                     const double* R0, double* E) try {
  TRY(check_ctx(c));
  TRY(check_system(A, "tcm_direct_batch A"));
  TRY(check_system(B, "tcm_direct_batch B"));
  if (n_items < 0) return set_err(TCM_EINVAL, "tcm_direct_batch: negative count");
  if (n_items == 0) return TCM_OK;
  if (!R0 || !E) return set_err(TCM_EINVAL, "tcm_direct_batch: null argument");
  if (n_items > (1LL << 30)) return set_err(TCM_EINVAL, "tcm_direct_batch: too many items");
  if ((A->n + 255) / 256 * n_items > (1LL << 34))
    return set_err(TCM_EINVAL, "tcm_direct_batch: A's blocks x items exceeds the partial-sum buffer limit");
  return direct_items(c, A, B, n_items, rotB, R0, E);
} catch (const std::exception&) {
  return no_host_memory("tcm_direct_batch");
}

}  // extern "C"
