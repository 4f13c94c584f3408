// pft_batch.cu -- many independent systems of uneven grid and contour sizes advanced
// together.  Instances are grouped into classes of equal field kind and grid; within a
// class the members are sorted by contour length, so at contour step s the instances
// still marching are a prefix of the class and one launch per pass covers all of them
// (blockIdx.y = instance).  One field update of every instance -- both marches of all
// classes, each instance's reductions and its field step -- is captured once as a CUDA
// graph and replayed.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <string>
#include <tuple>
#include <vector>

#include "pft_batch.cuh"
#include "pft_engine.h"

namespace {

// The plans the batch autotuner times, in the order of BatchClass::tuned_ms.
const int kBatchPlans[PFT_BATCH_PLANS] = {0, 1, 2, 3, 19, 35, 51};
int batch_plan_index(int plan) {
  for (int k = 0; k < PFT_BATCH_PLANS; k++)
    if (kBatchPlans[k] == plan) return k;
  return -1;
}

struct BatchClass {
  pft::BatchGeom g;
  pft_kind kind;
  std::vector<int> members;   // instance indices, Ns descending
  int maxNs = 0;
  std::vector<int> active;    // active[s-1]: members with Ns >= s
  pft::BatchStep* d_fwd = nullptr;  // [maxNs][K]
  pft::BatchStep* d_bwd = nullptr;
  // plan 0: one march after the other, the quadrature fused into the conjugate march;
  // plan 1: both marches in the same launches (entries 2k / 2k+1 of a step), the z passes
  // of consecutive steps fused, the quadrature after the marches over both histories;
  // plan 2: the separable march on the plane and x kernels (FP32 real, ny = nz = nx in
  // {64, 128}); plan 3: the separable march on pencils -- both marches per launch, the
  // quadrature after them, as plan 1; plans 19, 35, 51: plan 3 with line variant 1, 2, 3
  // (register lines; 32-line tiles; twice the elements a thread in 32-line tiles)
  int plan = 3;
  pft::BatchStep* d_conc = nullptr;  // [maxNs][2K]
  pft::BatchStep* d_sep = nullptr;   // the same entries with the per-axis factors of plans 2, 3
  float tuned_ms[PFT_BATCH_PLANS] = {-1.f, -1.f, -1.f, -1.f, -1.f, -1.f, -1.f};  // autotuner timings of kBatchPlans
};

// A stream of the update besides the batch stream, with the event that joins it.
struct BatchLane {
  cudaStream_t stream = nullptr;
  cudaEvent_t event = nullptr;
  int load = 0;  // contour steps recorded on it
};

// Members k0 <= k < k1 of a class that march together; whole: all of them.
struct BatchGroup {
  int cls, k0, k1;
  bool whole;
  double work;
};

__global__ void k_batch_increment(unsigned long long* __restrict__ c, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) c[i] += 1ull;
}

pft_status bfail(pft_status s, const std::string& m) {
  pft::set_error(m);
  return s;
}

pft_status bcuda(cudaError_t e, const char* what) {
  pft::set_error(std::string(what) + ": " + cudaGetErrorString(e));
  (void)cudaGetLastError();
  return e == cudaErrorMemoryAllocation ? PFT_ERR_OOM : PFT_ERR_CUDA;
}

}  // namespace

struct pft_batch {
  std::vector<pft_ctx*> inst;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  std::vector<BatchClass> classes;
  unsigned long long* d_steps = nullptr;
  int* d_err = nullptr;  // error word of the kernels' bounded waits
  cudaEvent_t fork = nullptr;
  std::vector<BatchLane> march, finish;
  cudaGraphExec_t graph = nullptr;
  double g_lam = -1.0, g_dt = -1.0;
  long long launches = 0;
  double units = 0.0;
};

namespace {

// The update's streams and the working set of a group.  A march is a chain of dependent launches,
// so the chains of different classes run beside one another, a march stream each (six at least, for
// the groups of few classes), the next group going to the stream with the fewest steps so far.
//
// Groups: a class marched whole keeps every member's field, factors and newest slices in turn, and
// where they pass the 129 MB L2 each launch finds the last one's field evicted; groups of at most
// 16 MB on six streams stay in L2 together.  But groups are more chains of smaller launches: where
// the whole batch nearly fits (three classes or more, together below 175 MB and none above 90) its
// classes march whole.  ms an update of 32^3 to 64^3 members with fields in and out, one stream a
// class and its finishes behind it / groups always / this rule: 15 members 6.9 / 9.0 / 6.8, 18 6.5 /
// 7.3 / 6.5, 22 9.6 / 11.1 / 9.4, 38 16.7 / 15.5 / 15.6, 64 27.4 / 25.1 / 24.5; a total of 120, 150 or 200 MB
// for 175 loses up to 4 % at 28 to 31 members or gives up to 7 % away at 35 to 39.  One class: 12
// members of 64^3 (complex, 151 MB) 17.1 / 13.6 / 13.6; FP64, 24 members 144 / 50.5 / 51.4, 16 64.2 / 23.5 /
// 23.9.
//
// Finishes: a member's quadrature and field step, a few small launches, on one of the march
// stream's own finish streams, a group's as soon as its member is done, a whole class's when the
// class is.  Streams shared by all classes held the early ones' finishes up behind the late ones':
// 101 members in ten classes 4.0 one stream a class, 5.2 shared, 3.7 now; 200 of one class 28.7, 11.5, 7.5.
constexpr int kMarchLanes = 6, kMaxMarchLanes = 24, kFinishLanes = 24;
constexpr double kBatchBytes = 175e6, kClassBytes = 90e6, kGroupBytes = 16e6;
constexpr double kGroupSlices = 6.0;  // a member's slices: both fields, both newest slices, B_A, B_B

double member_bytes(const pft_batch* b, const BatchClass& c) {
  const pft::CtxData& d = b->inst[c.members[0]]->d;
  return kGroupSlices * (double)d.M * (d.prec == PFT_FP64 ? 8 : 4) * (d.kind == PFT_SCFT_REAL ? 1 : 2);
}

// cls: one class (-1: all); whole: one group a class.
std::vector<BatchGroup> batch_groups(const pft_batch* b, int cls, bool whole) {
  std::vector<BatchGroup> out;
  double total = 0.0;
  for (const BatchClass& c : b->classes) total += member_bytes(b, c) * (double)c.members.size();
  for (size_t i = 0; i < b->classes.size(); i++) {
    if (cls >= 0 && (int)i != cls) continue;
    const BatchClass& c = b->classes[i];
    const double bytes = member_bytes(b, c);
    const int K = (int)c.members.size();
    const bool all = whole || (b->classes.size() > 2 && total <= kBatchBytes && bytes * K <= kClassBytes);
    const int per = all ? K : std::max(1, (int)(kGroupBytes / bytes));
    const int ng = (K + per - 1) / per;
    for (int q = 0; q < ng; q++) {
      BatchGroup g{(int)i, (int)((long long)K * q / ng), (int)((long long)K * (q + 1) / ng), all, 0.0};
      for (int k = g.k0; k < g.k1; k++) g.work += bytes * b->inst[c.members[k]]->d.Ns;
      out.push_back(g);
    }
  }
  std::stable_sort(out.begin(), out.end(), [](const BatchGroup& x, const BatchGroup& y) { return x.work > y.work; });
  return out;
}

void batch_free(pft_batch* b) {
  if (!b) return;
  if (b->graph) cudaGraphExecDestroy(b->graph);
  for (auto& c : b->classes) {
    if (c.d_fwd) cudaFree(c.d_fwd);
    if (c.d_bwd) cudaFree(c.d_bwd);
    if (c.d_conc) cudaFree(c.d_conc);
    if (c.d_sep) cudaFree(c.d_sep);
  }
  for (auto* lanes : {&b->march, &b->finish})
    for (auto& l : *lanes) {
      if (l.stream) cudaStreamDestroy(l.stream);
      if (l.event) cudaEventDestroy(l.event);
    }
  if (b->fork) cudaEventDestroy(b->fork);
  if (b->d_steps) cudaFree(b->d_steps);
  if (b->d_err) cudaFree(b->d_err);
  for (pft_ctx* c : b->inst)
    if (c) pft_destroy(c);
  if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
  delete b;
}

// Per-instance step arguments of both marches.
void fill_steps(const pft_ctx* c, int s, bool bwd, pft::BatchStep* st) {
  const pft::CtxData& d = c->d;
  const size_t we = (d.prec == PFT_FP64 ? 8 : 4) * (d.kind == PFT_SCFT_REAL ? 1 : 2);
  const size_t slice = (size_t)d.M * we;
  const char* hist = (const char*)d.hist;
  memset(st, 0, sizeof(*st));
  if (!bwd) {
    st->in = hist + (size_t)(s - 1) * slice;
    st->B = (s <= d.NsA) ? d.BA : d.BB;
    st->out = (void*)(hist + (size_t)s * slice);
  } else {
    const int nb = d.Ns + 1 - s;
    st->B = (nb <= d.NsA) ? d.BA : d.BB;
    st->in = (s == 1) ? d.qd0 : d.qd[(s - 1) & 1];
    st->out = d.qd[s & 1];
    const int pn = d.Ns - s;
    st->partner = hist + (size_t)pn * slice;
    double cA = 0.0, cB = 0.0;
    if (d.NsA > 0 && pn <= d.NsA) cA = (pn == 0 || pn == d.NsA) ? 0.5 : 1.0;
    if (d.NsA < d.Ns && pn >= d.NsA) cB = (pn == d.NsA || pn == d.Ns) ? 0.5 : 1.0;
    st->cA = cA;
    st->cB = cB;
    st->accA = d.accA;
    st->accB = d.accB;
  }
  st->spec = d.spec;
  const char* t = (const char*)d.tables;
  for (int a = 0; a < 4; a++) st->tw[a] = t + d.tw_off[a];
  for (int a = 0; a < 3; a++) st->d[a] = t + d.d_off[a];
}

// Entries of step s of both marches of one instance (plan 1): forward into the q history,
// conjugate into the qd history, each with the factor of its next step for the fused z
// passes (none at the instance's last step).
void fill_pair(const pft_ctx* c, int s, pft::BatchStep* f, pft::BatchStep* b) {
  const pft::CtxData& d = c->d;
  const size_t we = (d.prec == PFT_FP64 ? 8 : 4) * (d.kind == PFT_SCFT_REAL ? 1 : 2);
  const size_t slice = (size_t)d.M * we;
  const char* hist = (const char*)d.hist;
  char* qdh = (char*)d.qdh;
  memset(f, 0, sizeof(*f));
  memset(b, 0, sizeof(*b));
  const int nb = d.Ns + 1 - s;
  f->in = hist + (size_t)(s - 1) * slice;
  f->B = (s <= d.NsA) ? d.BA : d.BB;
  f->out = (void*)(hist + (size_t)s * slice);
  f->spec = d.spec;
  b->in = (s == 1) ? d.qd0 : (const void*)(qdh + (size_t)(s - 1) * slice);
  b->B = (nb <= d.NsA) ? d.BA : d.BB;
  b->out = qdh + (size_t)s * slice;
  b->spec = d.spec2;
  if (s < d.Ns) {
    f->Bnext = (s + 1 <= d.NsA) ? d.BA : d.BB;
    b->Bnext = (nb - 1 <= d.NsA) ? d.BA : d.BB;
  }
  const char* t = (const char*)d.tables;
  for (int a = 0; a < 4; a++) f->tw[a] = b->tw[a] = t + d.tw_off[a];
  for (int a = 0; a < 3; a++) f->d[a] = b->d[a] = t + d.d_off[a];
}

// qd histories and the pair-step table of a class (plan 1), once.
pft_status prepare_pairs(pft_batch* b, BatchClass& c) {
  if (c.d_conc) return PFT_OK;
  for (int i : c.members) {
    pft::CtxData& d = b->inst[i]->d;
    if (d.qdh) continue;
    const size_t we = (d.prec == PFT_FP64 ? 8 : 4) * (d.kind == PFT_SCFT_REAL ? 1 : 2);
    const size_t bytes = (size_t)(d.Ns + 1) * d.M * we;
    cudaError_t e = cudaMalloc(&d.qdh, bytes);
    if (e != cudaSuccess) return bcuda(e, "batch qd history");
    d.bytes += bytes;
  }
  const int K = (int)c.members.size();
  std::vector<pft::BatchStep> h((size_t)c.maxNs * 2 * K);
  for (int s = 1; s <= c.maxNs; s++)
    for (int k = 0; k < c.active[s - 1]; k++)
      fill_pair(b->inst[c.members[k]], s, &h[((size_t)(s - 1) * K + k) * 2], &h[((size_t)(s - 1) * K + k) * 2 + 1]);
  const size_t bytes = h.size() * sizeof(pft::BatchStep);
  cudaError_t e = cudaMalloc(&c.d_conc, bytes);
  if (e == cudaSuccess) e = cudaMemcpy(c.d_conc, h.data(), bytes, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return bcuda(e, "batch pair-step table");
  // the separable plans: the same entries with each member's full-axis factors
  for (int s = 1; s <= c.maxNs; s++)
    for (int k = 0; k < c.active[s - 1]; k++) {
      const pft::CtxData& d = b->inst[c.members[k]]->d;
      const char* t = (const char*)d.tables;
      for (int m = 0; m < 2; m++) {
        pft::BatchStep& x = h[((size_t)(s - 1) * K + k) * 2 + m];
        for (int a = 0; a < 3; a++) x.d[a] = t + d.sd_off[a];
      }
    }
  e = cudaMalloc(&c.d_sep, bytes);
  if (e == cudaSuccess) e = cudaMemcpy(c.d_sep, h.data(), bytes, cudaMemcpyHostToDevice);
  return e == cudaSuccess ? PFT_OK : bcuda(e, "batch separable step table");
}

// The marches of the members k0 <= k < k1 of one class under its plan, on `sm` (the members'
// context streams must be `sm` too); done(k) records what follows member k's marches.
template <typename F>
pft_status record_marches(pft_batch* b, BatchClass& c, int k0, int k1, long long* launches, cudaStream_t sm, F done) {
  const int K = (int)c.members.size();
  pft::Engine* eng = b->inst[c.members[0]]->eng;
  const int maxNs = b->inst[c.members[k0]]->d.Ns;
  auto active = [&](int s) { return std::min(c.active[s - 1], k1) - k0; };
  pft_status st = PFT_OK;
  if (c.plan == 2 || (c.plan & 15) == 3) {
    int left = k1;  // members without a recorded end: [k0, left)
    for (int j = 0; j <= maxNs; j++) {
      const int s = j == 0 ? 1 : j;
      cudaError_t e = eng->batch_sep_launch(c.g, c.d_sep + ((size_t)(s - 1) * K + k0) * 2, j, 2 * active(s), c.plan,
                                            b->d_err, sm);
      if (e != cudaSuccess) return bcuda(e, "batched separable step");
      *launches += (c.plan != 2 && j > 0) ? 2 : 1;
      for (; st == PFT_OK && j > 0 && left > k0 && b->inst[c.members[left - 1]]->d.Ns == j; left--) st = done(left - 1);
      if (st != PFT_OK) return st;
    }
    return PFT_OK;
  }
  if (c.plan == 1) {
    for (int s = 1; s <= maxNs; s++) {
      cudaError_t e = eng->batch_pair_step(c.g, c.d_conc + ((size_t)(s - 1) * K + k0) * 2, 2 * active(s), s == 1, sm);
      if (e != cudaSuccess) return bcuda(e, "batched pair step");
      *launches += eng->batch_pair_launches(c.g, s == 1);
    }
  } else {
    for (int march = 0; march < 2; march++) {
      for (int s = 1; s <= maxNs; s++) {
        cudaError_t e = eng->batch_contour_step(c.g, (march ? c.d_bwd : c.d_fwd) + (size_t)(s - 1) * K + k0, active(s),
                                                march, sm);
        if (e != cudaSuccess) return bcuda(e, "batched contour step");
        *launches += 5;
      }
      for (int k = k0; k < k1 && march == 0; k++) {
        pft_ctx* x = b->inst[c.members[k]];
        cudaError_t e = x->eng->solve_mid(x->d);
        if (e != cudaSuccess) return bcuda(e, "batched reductions");
        *launches += 3;
      }
    }
  }
  for (int k = k0; k < k1 && st == PFT_OK; k++) st = done(k);
  return st;
}

// Q, the quadrature and the densities of one member after its marches, on its context's stream.
pft_status record_finish(pft_batch* b, const BatchClass& c, int k, long long* launches) {
  pft_ctx* x = b->inst[c.members[k]];
  cudaError_t e = cudaSuccess;
  if (c.plan == 0) {
    e = x->eng->solve_tail(x->d);
    *launches += 2;
  } else if (c.plan == 1) {
    e = x->eng->solve_mid(x->d);
    if (e == cudaSuccess) e = x->eng->quadrature(x->d);
    if (e == cudaSuccess) e = x->eng->solve_tail(x->d);
    *launches += 6;
  } else {
    e = x->eng->finish_both(x->d);
    *launches += 4;
  }
  return e == cudaSuccess ? PFT_OK : bcuda(e, "batched quadrature");
}

// The solves of class `cls` (-1: every instance): the groups of members spread over the march
// streams (each forked from and joined back into b->stream), each member's quadrature, and what
// after(member) records, on a finish stream of its march stream.  `direct`: enqueued, not captured;
// then whole classes (half the launches, 2 us of the host each) on the march streams alone, the
// finishes on those without a class (streams beyond the device's eight hardware queues share one
// and wait for one another).
template <typename F>
pft_status record_solves(pft_batch* b, int cls, bool direct, long long* launches, F after) {
  cudaError_t e = cudaEventRecord(b->fork, b->stream);
  for (auto& l : b->march) {
    if (e == cudaSuccess) e = cudaStreamWaitEvent(l.stream, b->fork, 0);
    l.load = 0;
  }
  for (auto& l : b->finish)
    if (e == cudaSuccess && !direct) e = cudaStreamWaitEvent(l.stream, b->fork, 0);
  if (e != cudaSuccess) return bcuda(e, "batch fork");
  const size_t nfin = b->finish.size() / b->march.size();  // finish streams of a march stream
  size_t nf = 0;
  const std::vector<BatchGroup> groups = batch_groups(b, cls, direct);
  // direct: the groups take a march stream each, the finishes those that are left, if they are
  // enough of them (100 members of 24^3 11.8 ms against 19.9 with the finishes behind the march)
  size_t idle = b->march.size() > groups.size() ? b->march.size() - groups.size() : 0;
  if (idle < 3) idle = 0;
  pft_status st = PFT_OK;
  for (const BatchGroup& g : groups) {
    BatchClass& c = b->classes[g.cls];
    const size_t li = std::min_element(b->march.begin(), b->march.end(),
                                       [](const BatchLane& x, const BatchLane& y) { return x.load < y.load; }) -
                      b->march.begin();
    BatchLane& l = b->march[li];
    l.load += b->inst[c.members[g.k0]]->d.Ns;
    for (int k = g.k0; k < g.k1; k++) b->inst[c.members[k]]->d.stream = l.stream;
    auto finish = [&](int k) {
      pft_ctx* x = b->inst[c.members[k]];
      cudaError_t e = cudaSuccess;
      if (!direct || idle > 0) {
        const BatchLane& f = direct ? b->march[groups.size() + nf++ % idle] : b->finish[li * nfin + nf++ % nfin];
        e = cudaEventRecord(l.event, l.stream);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(f.stream, l.event, 0);
        if (e != cudaSuccess) return bcuda(e, "member fork");
        x->d.stream = f.stream;
      }
      pft_status s = record_finish(b, c, k, launches);
      if (s != PFT_OK) return s;
      e = after(x);
      return e == cudaSuccess ? PFT_OK : bcuda(e, "batched field step");
    };
    st = record_marches(b, c, g.k0, g.k1, launches, l.stream,
                        [&](int k) { return g.whole ? PFT_OK : finish(k); });
    for (int k = g.k0; k < g.k1 && st == PFT_OK && g.whole; k++) st = finish(k);
    for (int k = g.k0; k < g.k1; k++) b->inst[c.members[k]]->d.stream = b->stream;
    if (st != PFT_OK) break;
  }
  for (auto* lanes : {&b->march, &b->finish})  // after an error too: what was launched is joined
    for (auto& l : *lanes) {
      if (direct && lanes == &b->finish) break;
      if (e == cudaSuccess) e = cudaEventRecord(l.event, l.stream);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(b->stream, l.event, 0);
    }
  if (st != PFT_OK) return st;
  return e == cudaSuccess ? PFT_OK : bcuda(e, "batch join");
}

// One field update of every instance: the solves, each with its field step, then the step
// counters on b->stream.
pft_status record_update(pft_batch* b, double lam, double dt, bool direct) {
  long long launches = 0;
  pft_status s = record_solves(b, -1, direct, &launches, [&](pft_ctx* x) {
    const bool scft = (x->d.kind == PFT_SCFT_REAL);
    launches += 2;
    return x->eng->field_step(x->d, scft ? PFT_STEP_SCFT_EULER : PFT_STEP_CL_EULER_MARUYAMA, scft ? lam : dt, nullptr,
                              nullptr);
  });
  if (s != PFT_OK) return s;
  const int n = (int)b->inst.size();
  k_batch_increment<<<(n + 255) / 256, 256, 0, b->stream>>>(b->d_steps, n);
  launches += 1;
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return bcuda(e, "batched step counter");
  b->launches = launches;
  return PFT_OK;
}

// What record() enqueues from and to b->stream, as a graph.
template <typename F> pft_status capture(pft_batch* b, cudaGraphExec_t* out, F record) {
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return bcuda(e, "batch capture");
  pft_status s = record();
  e = cudaStreamEndCapture(b->stream, &g);
  if (s != PFT_OK) {
    if (g) cudaGraphDestroy(g);
    return s;
  }
  if (e != cudaSuccess) return bcuda(e, "batch capture end");
  e = cudaGraphInstantiate(out, g, 0);
  cudaGraphDestroy(g);
  return e == cudaSuccess ? PFT_OK : bcuda(e, "batch graph instantiate");
}

// The graph of one update.
pft_status make_graph(pft_batch* b, double lam, double dt) {
  pft_status s = capture(b, &b->graph, [&] { return record_update(b, lam, dt, false); });
  if (s != PFT_OK) return s;
  b->g_lam = lam;
  b->g_dt = dt;
  return PFT_OK;
}

// Can the batch stream be captured (a legacy stream, or one being captured, cannot)?
cudaError_t try_capture(pft_batch* b) {
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) e = cudaStreamEndCapture(b->stream, &g);
  if (e == cudaSuccess) e = cudaGraphDestroy(g);
  return e;
}

// Time of one solve of class `cls` under its plan, as the update runs it: its groups on the march
// streams, captured (launch by launch where the stream allows no capture).  The class whole on one
// stream orders the plans otherwise: 200 members of 16^3, complex FP64, plans 0 / 3, ms: 40.4 / 41.4
// against 31.7 / 26.1 in the update.
pft_status time_class(pft_batch* b, int cls, cudaEvent_t e0, cudaEvent_t e1, float* ms) {
  long long n = 0;
  cudaGraphExec_t graph = nullptr;
  auto solves = [&](bool direct) {
    return record_solves(b, cls, direct, &n, [](pft_ctx*) { return cudaSuccess; });
  };
  const bool direct = try_capture(b) != cudaSuccess;
  if (direct) (void)cudaGetLastError();
  pft_status s = direct ? PFT_OK : capture(b, &graph, [&] { return solves(false); });
  cudaError_t e = cudaSuccess;
  auto solve = [&] {
    if (direct) s = solves(true);
    else e = cudaGraphLaunch(graph, b->stream);
  };
  if (s == PFT_OK) solve();  // warm-up
  if (s == PFT_OK && e == cudaSuccess) e = cudaEventRecord(e0, b->stream);
  if (s == PFT_OK && e == cudaSuccess) solve();
  if (s == PFT_OK && e == cudaSuccess) e = cudaEventRecord(e1, b->stream);
  if (s == PFT_OK && e == cudaSuccess) e = cudaEventSynchronize(e1);
  if (s == PFT_OK && e == cudaSuccess) e = cudaEventElapsedTime(ms, e0, e1);
  if (graph) cudaGraphExecDestroy(graph);
  if (s != PFT_OK) return s;
  return e == cudaSuccess ? PFT_OK : bcuda(e, "autotune timing");
}

}  // namespace

extern "C" {

pft_status pft_batch_create(pft_batch** out, int count, const pft_instance_desc* descs, pft_precision precision,
                            void* stream) {
  if (!out) return bfail(PFT_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (count < 1 || !descs) return bfail(PFT_ERR_ARG, "need at least one instance description");
  for (int i = 0; i < count; i++)
    if (descs[i].model.arch != PFT_ARCH_DIBLOCK)
      return bfail(PFT_ERR_UNSUPPORTED, "batch instance " + std::to_string(i) + ": batches hold diblock systems");
  for (int i = 0; i < count; i++)
    for (int a = 0; a < 3; a++)
      if (!pft::batch_axis_supported(descs[i].grid.n[a]))
        return bfail(PFT_ERR_SHAPE, "batch instance " + std::to_string(i) + ": grid sizes must be one of " +
                                        "4,6,8,12,16,24,32,48,64");
  pft_batch* b = new pft_batch();
  if (stream) {
    b->stream = (cudaStream_t)stream;
  } else {
    cudaError_t e = cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
      delete b;
      return bcuda(e, "cudaStreamCreate");
    }
    b->own_stream = true;
  }
  b->inst.assign(count, nullptr);
  for (int i = 0; i < count; i++) {
    pft_opts o;
    memset(&o, 0, sizeof(o));
    o.precision = precision;
    o.use_graph = 1;
    o.stream = b->stream;
    o.seed = descs[i].seed;
    o.instance = (unsigned long long)i;
    o.march = PFT_MARCH_PASSES;
    o.checkpoint = 1;
    pft_status s = pft_create(&b->inst[i], &descs[i].grid, &descs[i].chain, &descs[i].model, &o);
    if (s != PFT_OK) {
      std::string msg = pft_last_error();
      batch_free(b);
      return bfail(s, "batch instance " + std::to_string(i) + ": " + msg);
    }
    b->units += 2.0 * (double)b->inst[i]->d.M * b->inst[i]->d.Ns;
    // members march one propagator at a time with the quadrature inside the conjugate
    // march (the batched launches already fill the GPU), in both batch modes
    b->inst[i]->d.concurrent = false;
  }
  cudaError_t e = cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming);
  if (e != cudaSuccess) {
    batch_free(b);
    return bcuda(e, "batch fork event");
  }
  e = cudaMalloc(&b->d_err, 4 * sizeof(int));
  if (e == cudaSuccess) e = cudaMemsetAsync(b->d_err, 0, 4 * sizeof(int), b->stream);
  if (e != cudaSuccess) {
    batch_free(b);
    return bcuda(e, "batch error word");
  }
  e = cudaMalloc(&b->d_steps, sizeof(unsigned long long) * count);
  if (e == cudaSuccess) e = cudaMemsetAsync(b->d_steps, 0, sizeof(unsigned long long) * count, b->stream);
  if (e != cudaSuccess) {
    batch_free(b);
    return bcuda(e, "batch step counters");
  }
  for (int i = 0; i < count; i++) b->inst[i]->d.step_dev = b->d_steps + i;
  // classes of equal kind and grid, members by descending contour length
  std::map<std::tuple<int, int, int, int>, int> index;
  for (int i = 0; i < count; i++) {
    const pft::CtxData& d = b->inst[i]->d;
    auto key = std::make_tuple((int)d.kind, d.n[0], d.n[1], d.n[2]);
    auto it = index.find(key);
    if (it == index.end()) {
      BatchClass c;
      for (int a = 0; a < 3; a++) c.g.n[a] = d.n[a];
      c.g.kind = d.kind;
      c.g.nzh = d.nzh;
      c.kind = d.kind;
      // the default plan (measured on GB300 with the 256-instance batch): the separable
      // march on the plane kernel where it applies, else on pencils
      pft::Engine* eng = b->inst[i]->eng;
      c.plan = eng->batch_plan_ok(c.g, 2) ? 2 : (eng->batch_plan_ok(c.g, 3) ? 3 : 1);
      index[key] = (int)b->classes.size();
      b->classes.push_back(c);
      it = index.find(key);
    }
    b->classes[it->second].members.push_back(i);
  }
  const int lanes = std::min(count, std::min(kMaxMarchLanes, std::max(kMarchLanes, (int)b->classes.size())));
  b->march.resize(lanes);
  b->finish.resize((size_t)lanes * std::max(1, std::min(4, kFinishLanes / lanes)));
  for (auto* v : {&b->march, &b->finish})
    for (auto& l : *v) {
      if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&l.stream, cudaStreamNonBlocking);
      if (e == cudaSuccess) e = cudaEventCreateWithFlags(&l.event, cudaEventDisableTiming);
    }
  if (e != cudaSuccess) {
    batch_free(b);
    return bcuda(e, "batch streams");
  }
  for (auto& c : b->classes) {
    std::stable_sort(c.members.begin(), c.members.end(),
                     [&](int x, int y) { return b->inst[x]->d.Ns > b->inst[y]->d.Ns; });
    const int K = (int)c.members.size();
    c.maxNs = b->inst[c.members[0]]->d.Ns;
    c.active.assign(c.maxNs, 0);
    for (int s = 1; s <= c.maxNs; s++)
      for (int k = 0; k < K; k++)
        if (b->inst[c.members[k]]->d.Ns >= s) c.active[s - 1] = k + 1;
    std::vector<pft::BatchStep> hf((size_t)c.maxNs * K), hb((size_t)c.maxNs * K);
    for (int s = 1; s <= c.maxNs; s++)
      for (int k = 0; k < c.active[s - 1]; k++) {
        fill_steps(b->inst[c.members[k]], s, false, &hf[(size_t)(s - 1) * K + k]);
        fill_steps(b->inst[c.members[k]], s, true, &hb[(size_t)(s - 1) * K + k]);
      }
    const size_t bytes = hf.size() * sizeof(pft::BatchStep);
    e = cudaMalloc(&c.d_fwd, bytes);
    if (e == cudaSuccess) e = cudaMalloc(&c.d_bwd, bytes);
    if (e == cudaSuccess) e = cudaMemcpy(c.d_fwd, hf.data(), bytes, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(c.d_bwd, hb.data(), bytes, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
      batch_free(b);
      return bcuda(e, "batch step tables");
    }
  }
  *out = b;
  return PFT_OK;
}

pft_status pft_batch_destroy(pft_batch* b) {
  if (!b) return PFT_OK;
  if (b->stream) cudaStreamSynchronize(b->stream);
  batch_free(b);
  return PFT_OK;
}

pft_status pft_batch_set_fields(pft_batch* b, int i, const void* wp, const void* wm, pft_mem where) {
  if (!b || i < 0 || i >= (int)b->inst.size()) return bfail(PFT_ERR_ARG, "bad batch or instance index");
  pft_status s = pft_set_fields(b->inst[i], wp, wm, where);
  if (s != PFT_OK) return s;
  cudaError_t e = cudaMemsetAsync(b->d_steps + i, 0, sizeof(unsigned long long), b->stream);
  return e == cudaSuccess ? PFT_OK : bcuda(e, "reset step counter");
}

pft_status pft_batch_get_fields(pft_batch* b, int i, void* wp, void* wm, pft_mem where) {
  if (!b || i < 0 || i >= (int)b->inst.size()) return bfail(PFT_ERR_ARG, "bad batch or instance index");
  return pft_get_fields(b->inst[i], wp, wm, where);
}

pft_status pft_batch_get_densities(pft_batch* b, int i, void* phiA, void* phiB, pft_mem where) {
  if (!b || i < 0 || i >= (int)b->inst.size()) return bfail(PFT_ERR_ARG, "bad batch or instance index");
  return pft_get_densities(b->inst[i], phiA, phiB, where);
}

pft_status pft_batch_get_observables(pft_batch* b, int i, pft_obs* obs) {
  if (!b || i < 0 || i >= (int)b->inst.size()) return bfail(PFT_ERR_ARG, "bad batch or instance index");
  return pft_get_observables(b->inst[i], obs);
}

pft_status pft_batch_run(pft_batch* b, int updates, double lam, double dt, pft_batch_mode mode) {
  if (!b || updates < 0) return bfail(PFT_ERR_ARG, "bad argument");
  if (!(lam > 0.0) || !(dt > 0.0) || !isfinite(lam) || !isfinite(dt))
    return bfail(PFT_ERR_ARG, "lam and dt must be positive");
  for (pft_ctx* x : b->inst)
    if (!x->d.fields_set) return bfail(PFT_ERR_STATE, "every batch instance needs pft_batch_set_fields first");
  for (auto& c : b->classes) {  // allocations and table uploads happen outside any capture
    if (c.plan == 0) continue;
    pft_status s = prepare_pairs(b, c);
    if (s != PFT_OK) return s;
  }
  int run = 0;  // updates enqueued
  pft_status s = PFT_OK;
  if (mode == PFT_BATCH_GRAPHED) {
    if (!b->graph || lam != b->g_lam || dt != b->g_dt) {
      if (b->graph) {
        cudaGraphExecDestroy(b->graph);
        b->graph = nullptr;
      }
      // a stream that cannot be captured is refused before anything runs on it
      const cudaError_t e = try_capture(b);
      if (e != cudaSuccess) return bcuda(e, "batch capture");
      // The first update runs launch by launch, and while the GPU works on it the host makes the
      // graph of the later ones (2.5 us a launch; 64 members of 32^3 to 64^3, 5064 launches: 13
      // ms), which a first update, or one with another lam or dt, would else wait for.
      if (updates > 0) {
        if ((s = record_update(b, lam, dt, true)) != PFT_OK) return s;
        run = 1;
      }
      s = make_graph(b, lam, dt);
    }
    for (; s == PFT_OK && run < updates; run++) {
      cudaError_t e = cudaGraphLaunch(b->graph, b->stream);
      if (e != cudaSuccess) s = bcuda(e, "batch graph launch");
    }
  } else if (mode == PFT_BATCH_PER_INSTANCE) {
    const int n = (int)b->inst.size();
    for (; s == PFT_OK && run < updates; run++) {
      for (pft_ctx* x : b->inst) {
        const bool scft = (x->d.kind == PFT_SCFT_REAL);
        cudaError_t e = x->eng->enqueue_solve(x->d);
        if (e == cudaSuccess)
          e = x->eng->field_step(x->d, scft ? PFT_STEP_SCFT_EULER : PFT_STEP_CL_EULER_MARUYAMA, scft ? lam : dt,
                                 nullptr, nullptr);
        if (e != cudaSuccess) return bcuda(e, "per-instance update");
      }
      k_batch_increment<<<(n + 255) / 256, 256, 0, b->stream>>>(b->d_steps, n);
      cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return bcuda(e, "step counter");
    }
  } else {
    return bfail(PFT_ERR_ARG, "unknown batch mode");
  }
  for (pft_ctx* x : b->inst) {
    x->d.step += run;
    x->d.solved = false;
    if (run > 0) x->have_obs = true;
  }
  return s;
}

pft_status pft_batch_autotune(pft_batch* b) {
  if (!b) return bfail(PFT_ERR_ARG, "NULL batch");
  for (pft_ctx* x : b->inst)
    if (!x->d.fields_set) return bfail(PFT_ERR_STATE, "every batch instance needs pft_batch_set_fields first");
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  if (e != cudaSuccess) return bcuda(e, "autotune events");
  pft_status st = PFT_OK;
  for (auto& c : b->classes) {
    float best = -1.f;
    int bplan = c.plan;
    pft::Engine* eng = b->inst[c.members[0]]->eng;
    for (int pi = 0; pi < PFT_BATCH_PLANS && st == PFT_OK; pi++) {
      const int plan = kBatchPlans[pi];
      if (!eng->batch_plan_ok(c.g, plan)) continue;
      c.plan = plan;
      if (plan >= 1 && (st = prepare_pairs(b, c)) != PFT_OK) break;
      float ms = 0.f;
      if ((st = time_class(b, (int)(&c - b->classes.data()), e0, e1, &ms)) != PFT_OK) break;
      c.tuned_ms[pi] = ms;
      if (best < 0.f || ms < best) {
        best = ms;
        bplan = plan;
      }
    }
    c.plan = bplan;
    if (st != PFT_OK) break;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (b->graph) {  // the next graphed run captures the chosen plans
    cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
  }
  return st;
}

pft_status pft_batch_set_plan(pft_batch* b, int cls, int plan) {
  if (!b || cls < -1 || cls >= (int)b->classes.size()) return bfail(PFT_ERR_ARG, "bad batch or class index");
  if (batch_plan_index(plan) < 0) return bfail(PFT_ERR_ARG, "plan must be 0, 1, 2, 3, 19, 35 or 51");
  if (cls >= 0 && !b->inst[b->classes[cls].members[0]]->eng->batch_plan_ok(b->classes[cls].g, plan))
    return bfail(PFT_ERR_UNSUPPORTED, "plan " + std::to_string(plan) + " does not apply to class " + std::to_string(cls));
  for (int k = 0; k < (int)b->classes.size(); k++) {
    BatchClass& c = b->classes[k];
    // all classes (cls = -1): the classes the plan applies to
    if ((cls < 0 || k == cls) && b->inst[c.members[0]]->eng->batch_plan_ok(c.g, plan)) c.plan = plan;
  }
  if (b->graph) {
    cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
  }
  return PFT_OK;
}

pft_status pft_batch_class_info(const pft_batch* b, int cls, int n[3], int* kind, int* members, int* plan,
                                float tuned_ms[PFT_BATCH_PLANS]) {
  if (!b || cls < 0 || cls >= (int)b->classes.size()) return bfail(PFT_ERR_ARG, "bad batch or class index");
  const BatchClass& c = b->classes[cls];
  if (n)
    for (int a = 0; a < 3; a++) n[a] = c.g.n[a];
  if (kind) *kind = (int)c.kind;
  if (members) *members = (int)c.members.size();
  if (plan) *plan = c.plan;
  if (tuned_ms)
    for (int k = 0; k < PFT_BATCH_PLANS; k++) tuned_ms[k] = c.tuned_ms[k];
  return PFT_OK;
}

pft_status pft_batch_synchronize(pft_batch* b) {
  if (!b) return bfail(PFT_ERR_ARG, "NULL batch");
  int err = 0;
  cudaError_t e = cudaMemcpyAsync(&err, b->d_err, sizeof(int), cudaMemcpyDeviceToHost, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) return bcuda(e, "batch synchronize");
  if (err != 0) {
    cudaMemsetAsync(b->d_err, 0, sizeof(int), b->stream);
    cudaStreamSynchronize(b->stream);
    return bfail(PFT_ERR_TIMEOUT, "a bounded wait in a kernel of the last updates ran out (their results are invalid)");
  }
  return PFT_OK;
}

pft_status pft_batch_info(const pft_batch* b, double* units_per_update, int* nclasses, long long* launches) {
  if (!b) return bfail(PFT_ERR_ARG, "NULL batch");
  if (units_per_update) *units_per_update = b->units;
  if (nclasses) *nclasses = (int)b->classes.size();
  if (launches) *launches = b->launches;
  return PFT_OK;
}

pft_status pft_batch_get_stream(const pft_batch* b, void** stream) {
  if (!b || !stream) return bfail(PFT_ERR_ARG, "NULL argument");
  *stream = (void*)b->stream;
  return PFT_OK;
}

}  // extern "C"
