// C ABI of the batched evolution (include/floquet_sv.h, "batch" section):
// many independent chains on one device, each in its own slice of one
// caller-owned buffer.
//
// Every chain gets a context (sv_ctx) on its slice for initialisation and,
// for the plain, block and multi-gate forms, for its evolution graph.  Chains of at most
// 14 sites may instead run the resident form: one launch per length advances them,
// each in the shared memory of one CTA or of a cluster (k_resident.cu; up to ten sites
// k_batch.cu, one launch for up to nine and one for ten).  An evolution is
// one CUDA graph per run of M periods: the resident launches; one branch per
// group of tensor-core chains whose plans share their structure (same L; one
// branch for all groups where their tiles are few), each pass of all its chains
// one launch over all their tiles and each period's reduces one launch; and, for every other chain, its run of M
// periods captured from its context.  A block plan whose periods start off
// site 0 relabels into its period layout at the start of the run and hands
// back the natural layout at its end.
//
// The autotuner (form SV_BATCH_AUTO) times every form that fits a distinct
// L, run together for four periods through the same kind of graph (the
// CUDA-core block form at widths n = 5, 6 and 7, the tensor-core block form
// as a group, the plain, multi-gate and resident forms), and keeps the
// fastest (most chain-periods per second) for all chains of that L.  The resident form is
// timed on all chains of that L (one or a few CTAs each, so its rate grows with
// their number), the tensor-core form on a group that fills the device, the
// others, which fill it with one chain, on up to eight.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <new>
#include <string>
#include <vector>

#include "sv_batch.h"
#include "sv_block.h"

// The resident chains' device tables: descriptors, gates, rounds (or the
// short chains' bonds), energy rings and the shared period counter; the launches, one
// per chain length (shape.L = 0: the chains of up to kShortMaxL sites).
struct ResidentSet {
  struct Class {
    fsv::ResidentShape shape;
    int first = 0, count = 0, ngates = 0;
    Class() { shape.L = 0; }
  };
  fsv::ChainArgs* d_res = nullptr;
  float2* d_gates = nullptr;
  fsv::ResidentRound* d_rounds = nullptr;
  double* d_ring = nullptr;
  long long* d_count = nullptr;
  int count = 0;
  std::vector<Class> classes;
  std::vector<int> place;  // ring of the k-th chain of the set
  void release() {
    cudaFree(d_res);
    cudaFree(d_gates);
    cudaFree(d_rounds);
    cudaFree(d_ring);
    cudaFree(d_count);
    *this = ResidentSet();
  }
};

struct sv_batch {
  int device = 0;
  int n = 0;
  cudaStream_t stream = nullptr;      // caller's stream
  cudaStream_t cap_stream = nullptr;  // capture of the resident launch
  char* base = nullptr;
  std::vector<int> L;
  std::vector<size_t> off;
  std::vector<int> form;
  std::vector<int> width;      // block forms: window width n
  std::vector<sv_floquet_params> params;
  std::vector<const double*> spinors;  // caller's arrays, valid during create only
  std::vector<sv_ctx*> ctx;
  // resident chains
  std::vector<int> res;
  ResidentSet rset;
  // graphs of one period and of M periods of every chain
  cudaGraphExec_t g1 = nullptr, gm = nullptr;
  // of a batch whose chains all are resident: d_count[1] (run) periods
  cudaGraphExec_t gr = nullptr;
  int64_t run = 0;
  std::vector<fsv::BlockSet*> groups;  // chain groups the two graphs launch
  // energies of the graph-form chains: their rings, and a buffer that a run's
  // slots are gathered into for one copy
  fsv::RingSource* d_rings = nullptr;
  double* d_gather = nullptr;
  int M = 16;
  int64_t counter = 0;
  std::string err;
};

namespace {

constexpr size_t kAlign = 256;
// CUDA-core block passes of a batch share the device with other chains'
// passes: each CTA keeps a run of at least this many tiles.
constexpr int kDefaultTileRun = 8;
constexpr int kSimtWidths[3] = {5, 6, 7};
constexpr int kDefaultWidth = 6;

int bfail(sv_batch* b, int code, const char* fmt, ...) {
  if (b) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    b->err = buf;
  }
  if (code == SV_ECUDA) cudaGetLastError();  // reported here, not again by the next call
  return code;
}

#define BCUDA(call, what)                                                        \
  do {                                                                           \
    cudaError_t e_ = (call);                                                     \
    if (e_ != cudaSuccess) return bfail(b, SV_ECUDA, "%s: %s", what, cudaGetErrorString(e_)); \
  } while (0)

bool form_fits(int form, int L) {
  switch (form) {
    case SV_BATCH_PLAIN: return true;
    case SV_BATCH_BLOCK_SIMT: return L >= 6;
    case SV_BATCH_BLOCK_TC: return L >= 13;
    case SV_BATCH_RESIDENT: return L <= fsv::kResidentMaxL;
    case SV_BATCH_MULTIGATE: return true;
    default: return false;
  }
}

int build_resident(sv_batch* b, const std::vector<int>& chains, ResidentSet* rs) {
  *rs = ResidentSet();
  if (chains.empty()) return SV_OK;
  const int ring = fsv::ctx_ring_len();
  // chains of one length together, each length one launch; set order: by length,
  // then as given
  std::vector<int> order(chains.size());
  for (size_t k = 0; k < order.size(); ++k) order[k] = (int)k;
  std::stable_sort(order.begin(), order.end(),
                   [&](int x, int y) { return b->L[chains[x]] > b->L[chains[y]]; });
  // a chain takes several blocks where the device has SMs left over
  int sms = 0;
  BCUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device), "SM count");
  std::map<int, int> count, blocks;
  for (int c : chains) ++count[b->L[c]];
  int used = (int)chains.size();
  for (auto& kv : count) blocks[kv.first] = 1;
  for (bool grew = true; grew;) {
    grew = false;
    for (auto it = count.rbegin(); it != count.rend(); ++it) {  // the longest chains first
      const int L = it->first, n = it->second, now = blocks[L];
      if (now >= 8 || used + n * now > sms) continue;
      if (fsv::resident_shape(false, L, 2 * now).kbits == fsv::resident_shape(false, L, now).kbits) continue;
      blocks[L] = 2 * now;
      used += n * now;
      grew = true;
      break;
    }
  }
  std::vector<fsv::ChainArgs> hd(chains.size());
  std::vector<float2> gates;
  std::vector<fsv::ResidentRound> rounds;
  std::vector<int> bonds;
  std::vector<size_t> goff(chains.size()), roff(chains.size()), boff(chains.size());
  for (size_t k = 0; k < chains.size(); ++k) {
    const int c = chains[order[k]];
    const int L = b->L[c];
    const sv_floquet_params& p = b->params[c];
    auto pg = fsv::period_gates(L, p, p.theta, p.hx);
    goff[k] = gates.size();
    gates.resize(gates.size() + pg.size() * fsv::kGateEntries);
    fsv::gate_tables(pg, &gates[goff[k]]);
    fsv::ChainArgs& r = hd[k];
    r.L = L;
    r.ngates = (int)pg.size();
    fsv::Observable o = fsv::observable(L, p);
    r.Jf = (float)o.J;
    for (int i = 0; i < L; ++i) {
      r.cx[i] = (float)o.cx[i];
      r.cz[i] = (float)o.cz[i];
    }
    boff[k] = bonds.size();
    roff[k] = rounds.size();
    if (L <= fsv::kShortMaxL) {
      for (auto& g : pg) bonds.push_back(g.bond);
      const int threads = fsv::short_threads(L);
      if (rs->classes.empty() || rs->classes.back().shape.L != 0 ||
          rs->classes.back().shape.threads != threads) {
        rs->classes.push_back({});
        rs->classes.back().shape.threads = threads;
      }
    } else {
      const fsv::ResidentShape sh = fsv::resident_shape(false, L, blocks[L]);
      auto rr = fsv::resident_rounds(pg, sh);
      if (rr.empty()) return bfail(b, SV_EINVAL, "chain %d: no plan for a chain in shared memory", c);
      r.nrounds = (int)rr.size();
      rounds.insert(rounds.end(), rr.begin(), rr.end());
      if (rs->classes.empty() || rs->classes.back().shape.L != L) {
        rs->classes.push_back({});
        rs->classes.back().shape = sh;
      }
      ResidentSet::Class& cl = rs->classes.back();
      cl.ngates = std::max(cl.ngates, r.ngates);
    }
    if (rs->classes.back().count++ == 0) rs->classes.back().first = (int)k;
  }
  for (const auto& cl : rs->classes)
    BCUDA(cl.shape.L ? fsv::resident_prepare(false, cl.shape, cl.ngates, nullptr) : fsv::short_prepare(),
          "resident attributes");
  rs->count = (int)chains.size();
  rs->place.resize(chains.size());
  for (size_t k = 0; k < chains.size(); ++k) rs->place[order[k]] = (int)k;
  const size_t round_b = sizeof(fsv::ResidentRound) * rounds.size(), bond_b = sizeof(int) * bonds.size();
  if (cudaMalloc(&rs->d_res, sizeof(fsv::ChainArgs) * hd.size()) != cudaSuccess ||
      cudaMalloc(&rs->d_gates, sizeof(float2) * gates.size()) != cudaSuccess ||
      cudaMalloc(&rs->d_rounds, round_b + bond_b + 16) != cudaSuccess ||
      cudaMalloc(&rs->d_ring, sizeof(double) * 2 * ring * hd.size()) != cudaSuccess ||
      cudaMalloc(&rs->d_count, 2 * sizeof(long long)) != cudaSuccess) {
    cudaGetLastError();
    rs->release();
    return bfail(b, SV_ENOMEM, "resident tables");
  }
  int* d_bonds = reinterpret_cast<int*>(reinterpret_cast<char*>(rs->d_rounds) + round_b);
  for (size_t k = 0; k < chains.size(); ++k) {
    fsv::ChainArgs& r = hd[k];
    r.psi = reinterpret_cast<float2*>(b->base + b->off[chains[order[k]]]);
    r.gates = rs->d_gates + goff[k];
    r.rounds = rs->d_rounds + roff[k];
    r.bonds = d_bonds + boff[k];
    r.ring = rs->d_ring + 2 * k;
    r.ring_stride = (long long)chains.size();
  }
  BCUDA(cudaMemcpyAsync(rs->d_res, hd.data(), sizeof(fsv::ChainArgs) * hd.size(),
                        cudaMemcpyHostToDevice, b->stream),
        "upload resident descriptors");
  BCUDA(cudaMemcpyAsync(rs->d_gates, gates.data(), sizeof(float2) * gates.size(),
                        cudaMemcpyHostToDevice, b->stream),
        "upload resident gates");
  if (round_b)
    BCUDA(cudaMemcpyAsync(rs->d_rounds, rounds.data(), round_b, cudaMemcpyHostToDevice, b->stream),
          "upload resident rounds");
  if (bond_b)
    BCUDA(cudaMemcpyAsync(d_bonds, bonds.data(), bond_b, cudaMemcpyHostToDevice, b->stream),
          "upload resident bonds");
  BCUDA(cudaMemsetAsync(rs->d_count, 0, 2 * sizeof(long long), b->stream), "reset counter");
  BCUDA(cudaStreamSynchronize(b->stream), "synchronize");
  return SV_OK;
}

// Build the period evolution of chain c in its context for a graph form
// (block forms: window width n; CUDA-core passes keep kDefaultTileRun tiles
// per CTA at least).
int build_graph_form(sv_batch* b, int c, int form, int n) {
  fsv::ctx_set_min_tiles(b->ctx[c], kDefaultTileRun);
  sv_floquet_params p = b->params[c];
  p.theta_p = nullptr;
  p.hx_p = nullptr;
  p.n_period_params = 0;
  p.renorm_every = 0;
  if (form == SV_BATCH_PLAIN) {
    p.mode = SV_MODE_PLAIN;
  } else if (form == SV_BATCH_MULTIGATE) {
    p.mode = SV_MODE_MULTIGATE;
  } else {
    p.mode = SV_MODE_BLOCK;
    p.block_n = form == SV_BATCH_BLOCK_TC ? 6 : n;
    p.split = form == SV_BATCH_BLOCK_TC ? SV_SPLIT_BF16X3 : SV_SPLIT_FP32;
  }
  int rc = sv_build_floquet(b->ctx[c], &p);
  if (rc) return bfail(b, rc, "chain %d build: %s", c, sv_last_error(b->ctx[c]));
  return SV_OK;
}

// Tensor-core chains grouped by plan structure, the groups in sets; the other chains
// are returned in `rest`.
int make_groups(sv_batch* b, const std::vector<int>& chains, std::vector<int>* rest,
                std::vector<fsv::BlockSet*>* sets) {
  std::vector<std::vector<fsv::GroupMember>> parts;
  for (int c : chains) {
    fsv::GroupMember m;
    if (fsv::ctx_block_member(b->ctx[c], &m.plan, &m.psi, &m.counter, &m.ring) != SV_OK) {
      rest->push_back(c);
      continue;
    }
    bool placed = false;
    for (auto& p : parts)
      if (fsv::block_same_structure(p[0].plan, m.plan)) {
        p.push_back(m);
        placed = true;
        break;
      }
    if (!placed) parts.push_back({m});
  }
  if (parts.empty()) return SV_OK;
  const fsv::LaunchCfg& cfg = parts[0][0].plan->cfg;
  const bool together = fsv::block_groups_together(parts, cfg);
  for (size_t k = 0; k < (together ? 1 : parts.size()); ++k) {
    fsv::BlockSet* set = nullptr;
    std::string msg;
    int rc = fsv::block_set_build(together ? parts : std::vector<std::vector<fsv::GroupMember>>{parts[k]},
                                  together, fsv::ctx_ring_len(), cfg, b->stream, &set, &msg);
    if (rc) return bfail(b, rc, "chain groups: %s", msg.c_str());
    sets->push_back(set);
  }
  return SV_OK;
}

void free_groups(std::vector<fsv::BlockSet*>* sets) {
  for (fsv::BlockSet* s : *sets) fsv::block_set_free(s);
  sets->clear();
}

// One graph advancing `periods` periods of the given graph-form chains and
// of the resident set (if any); 0 (a resident set alone): d_count[1] periods.
// Tensor-core chains run in groups, built on the first call (groups empty) and
// reused by later ones; the caller frees them after the graphs.
int make_graph(sv_batch* b, const std::vector<int>& chains, const ResidentSet* rs, int periods,
               cudaGraphExec_t* out, std::vector<fsv::BlockSet*>* groups) {
  *out = nullptr;
  cudaGraph_t g = nullptr;
  BCUDA(cudaGraphCreate(&g, 0), "graph create");
  auto fail_g = [&](int rc) {
    cudaGraphDestroy(g);
    return rc;
  };
  if (rs && rs->count > 0) {
    // each length's launch is a branch of its own; the counter advances after
    // all of them
    std::vector<cudaGraphNode_t> runs;
    const int ring = fsv::ctx_ring_len();
    for (size_t k = 0; k <= rs->classes.size(); ++k) {
      cudaGraph_t rg = nullptr;
      cudaError_t e = cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeRelaxed);
      if (e == cudaSuccess) {
        cudaError_t le;
        if (k == rs->classes.size()) {
          le = fsv::launch_advance(rs->d_count, periods, b->cap_stream);
        } else {
          const ResidentSet::Class& c = rs->classes[k];
          le = c.shape.L ? fsv::launch_resident_batch(rs->d_res + c.first, c.count, c.shape,
                                                      c.ngates, rs->d_count, periods, ring, b->cap_stream)
                         : fsv::launch_chain_short(rs->d_res + c.first, c.count, c.shape.threads,
                                                   rs->d_count, periods, ring, b->cap_stream);
        }
        e = cudaStreamEndCapture(b->cap_stream, &rg);
        if (le != cudaSuccess) e = le;
      }
      if (e != cudaSuccess) {
        if (rg) cudaGraphDestroy(rg);
        return fail_g(bfail(b, SV_ECUDA, "resident capture: %s", cudaGetErrorString(e)));
      }
      cudaGraphNode_t node;
      const bool last = k == rs->classes.size();
      e = cudaGraphAddChildGraphNode(&node, g, last ? runs.data() : nullptr, last ? runs.size() : 0, rg);
      cudaGraphDestroy(rg);
      if (e != cudaSuccess)
        return fail_g(bfail(b, SV_ECUDA, "resident node: %s", cudaGetErrorString(e)));
      runs.push_back(node);
    }
  }
  std::vector<int> rest;
  if (groups->empty()) {
    int rc = make_groups(b, chains, &rest, groups);
    if (rc) return fail_g(rc);
  } else {
    // the groups were built for these chains by an earlier call
    size_t grouped = 0;
    for (int c : chains) {
      fsv::GroupMember m;
      if (fsv::ctx_block_member(b->ctx[c], &m.plan, &m.psi, &m.counter, &m.ring) != SV_OK)
        rest.push_back(c);
      else
        ++grouped;
    }
    size_t members = 0;
    for (const fsv::BlockSet* set : *groups) members += fsv::block_set_size(set);
    if (members != grouped)
      return fail_g(bfail(b, SV_ESTATE, "chain groups built for another set of chains"));
  }
  for (fsv::BlockSet* set : *groups) {
    // Passes of a set that has the device to itself start under the one before, at every
    // size (a CTA's tiles are contiguous, so the order in which CTAs start does not
    // scatter L2 as it does for a single chain): 32 periods of 48 chains of 15 sites 3.05
    // ms, in turn 3.32, of 20 sites (400 MB) 49.4 and 49.8, 2 chains of 24 sites 39.4 and 39.9.
    const bool alone = groups->size() == 1 && rest.empty() && (!rs || rs->count == 0);
    cudaGraph_t pg = nullptr;
    cudaError_t e = cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeRelaxed);
    cudaError_t le = cudaSuccess;
    if (e == cudaSuccess) {
      le = fsv::block_set_enqueue(set, periods, alone, b->cap_stream);
      e = cudaStreamEndCapture(b->cap_stream, &pg);
      if (le != cudaSuccess) e = le;
    }
    if (e != cudaSuccess) {
      if (pg) cudaGraphDestroy(pg);
      return fail_g(bfail(b, SV_ECUDA, "group capture: %s", cudaGetErrorString(e)));
    }
    cudaGraphNode_t node;
    e = cudaGraphAddChildGraphNode(&node, g, nullptr, 0, pg);
    cudaGraphDestroy(pg);
    if (e != cudaSuccess)
      return fail_g(bfail(b, SV_ECUDA, "group node: %s", cudaGetErrorString(e)));
  }
  for (int c : rest) {
    cudaGraph_t pg = nullptr;
    int rc = fsv::ctx_capture_run(b->ctx[c], periods, &pg);
    if (rc) return fail_g(bfail(b, rc, "chain %d capture: %s", c, sv_last_error(b->ctx[c])));
    cudaGraphNode_t node;
    cudaError_t e = cudaGraphAddChildGraphNode(&node, g, nullptr, 0, pg);
    cudaGraphDestroy(pg);
    if (e != cudaSuccess)
      return fail_g(bfail(b, SV_ECUDA, "chain node: %s", cudaGetErrorString(e)));
  }
  cudaError_t e = cudaGraphInstantiate(out, g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) {
    *out = nullptr;
    return bfail(b, SV_ECUDA, "graph instantiate: %s", cudaGetErrorString(e));
  }
  return SV_OK;
}

// Bytes that the energies of `count` periods of `chains` chains are gathered into,
// and their flags behind them.
size_t gather_bytes(size_t chains, int64_t count) {
  return (2 * sizeof(double) * (size_t)count + sizeof(int)) * chains;
}

// The rings of the graph-form chains, and the buffer for a ring's length of periods.
int make_gather(sv_batch* b, const std::vector<int>& chains) {
  if (chains.empty()) return SV_OK;
  std::vector<fsv::RingSource> src;
  for (int c : chains) src.push_back(fsv::ctx_ring(b->ctx[c]));
  const size_t bytes = sizeof(fsv::RingSource) * src.size();
  if (cudaMalloc(&b->d_rings, bytes) != cudaSuccess ||
      cudaMalloc(&b->d_gather, gather_bytes(src.size(), fsv::ctx_ring_len())) != cudaSuccess) {
    cudaGetLastError();
    return bfail(b, SV_ENOMEM, "energy readback buffer");
  }
  BCUDA(cudaMemcpyAsync(b->d_rings, src.data(), bytes, cudaMemcpyHostToDevice, b->stream),
        "upload ring list");
  BCUDA(cudaStreamSynchronize(b->stream), "synchronize");
  return SV_OK;
}

// Energies and norms of the graph-form chains' last `count` periods (one copy for
// all chains, rows of `periods` from column `done`).
int read_graph_chains(sv_batch* b, const std::vector<int>& chains, int64_t count, int64_t periods,
                      int64_t done, double* energy_out, double* norm_out) {
  const size_t C = chains.size(), pairs = C * (size_t)count;
  std::vector<char> host(gather_bytes(C, count));
  BCUDA(fsv::launch_gather_rings(b->d_rings, (int)C, b->counter, (int)count, fsv::ctx_ring_len(),
                                 b->d_gather, reinterpret_cast<int*>(b->d_gather + 2 * pairs), b->stream),
        "energy gather launch");
  BCUDA(cudaMemcpyAsync(host.data(), b->d_gather, host.size(), cudaMemcpyDeviceToHost, b->stream),
        "energy readback");
  BCUDA(cudaStreamSynchronize(b->stream), "synchronize");
  const double* p = reinterpret_cast<const double*>(host.data());
  const int* status = reinterpret_cast<const int*>(p + 2 * pairs);
  for (size_t k = 0; k < C; ++k) {
    if (status[k])
      return bfail(b, SV_ETIMEOUT, "chain %d: a tensor-core block pass gave up a bounded wait", chains[k]);
    for (int64_t q = 0; q < count; ++q, p += 2) {
      if (energy_out) energy_out[(size_t)chains[k] * periods + done + q] = p[0];
      if (norm_out) norm_out[(size_t)chains[k] * periods + done + q] = p[1];
    }
  }
  return SV_OK;
}

int reinit(sv_batch* b, int c) {
  int rc = sv_init(b->ctx[c], b->L[c], b->spinors[c]);
  if (rc) return bfail(b, rc, "chain %d init: %s", c, sv_last_error(b->ctx[c]));
  return SV_OK;
}

// Chain-periods per second of the chains `sample` run together, chain
// sample[i] in form forms[i] (the CUDA-core block form at width n).  The
// trial moves the states; they are initialised again after it.
int time_forms(sv_batch* b, const std::vector<int>& sample, const std::vector<int>& forms, int n,
               double* rate) {
  *rate = 0.0;
  constexpr int kPeriods = 4;
  ResidentSet rs;
  std::vector<int> graph_chains, res_chains;
  int rc = SV_OK;
  for (size_t i = 0; i < sample.size() && rc == SV_OK; ++i) {
    if (forms[i] == SV_BATCH_RESIDENT) {
      res_chains.push_back(sample[i]);
    } else {
      rc = build_graph_form(b, sample[i], forms[i], n);
      graph_chains.push_back(sample[i]);
    }
  }
  if (rc == SV_OK) rc = build_resident(b, res_chains, &rs);
  cudaGraphExec_t ge = nullptr;
  std::vector<fsv::BlockSet*> groups;
  if (rc == SV_OK) rc = make_graph(b, graph_chains, &rs, kPeriods, &ge, &groups);
  if (rc == SV_OK) {
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    bool ok = cudaEventCreate(&e0) == cudaSuccess && cudaEventCreate(&e1) == cudaSuccess &&
              cudaGraphLaunch(ge, b->stream) == cudaSuccess &&  // warm-up
              cudaEventRecord(e0, b->stream) == cudaSuccess &&
              cudaGraphLaunch(ge, b->stream) == cudaSuccess &&
              cudaEventRecord(e1, b->stream) == cudaSuccess &&
              cudaEventSynchronize(e1) == cudaSuccess;
    float ms = 0.f;
    if (ok && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess && ms > 0.f)
      *rate = (double)sample.size() * kPeriods / (ms * 1e-3);
    if (!ok) rc = bfail(b, SV_ECUDA, "autotune run: %s", cudaGetErrorString(cudaGetLastError()));
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
  }
  if (ge) cudaGraphExecDestroy(ge);
  free_groups(&groups);
  rs.release();
  for (int c : sample) {
    int r2 = reinit(b, c);
    if (rc == SV_OK) rc = r2;
  }
  return rc;
}

int time_form(sv_batch* b, const std::vector<int>& sample, int form, int n, double* rate) {
  return time_forms(b, sample, std::vector<int>(sample.size(), form), n, rate);
}

int autotune(sv_batch* b) {
  std::map<int, std::vector<int>> byL;
  for (int c = 0; c < b->n; ++c) byL[b->L[c]].push_back(c);
  for (auto& kv : byL) {
    const int L = kv.first;
    auto first = [&](size_t n) {
      return std::vector<int>(kv.second.begin(), kv.second.begin() + std::min(n, kv.second.size()));
    };
    const std::vector<int> sample = first(8);
    // enough chains that their tiles fill the device (2^21 amplitudes): a group
    // of eight at L = 15 leaves half of the SMs without a tile
    const std::vector<int> group = first(std::max<size_t>(8, L < 21 ? (size_t)1 << (21 - L) : 1));
    int best = SV_BATCH_PLAIN, best_n = 0;
    double best_rate = -1.0;
    for (int f : {SV_BATCH_RESIDENT, SV_BATCH_BLOCK_TC, SV_BATCH_BLOCK_SIMT, SV_BATCH_PLAIN,
                  SV_BATCH_MULTIGATE}) {
      if (!form_fits(f, L)) continue;
      for (int n : kSimtWidths) {
        // widths for the CUDA-core form
        if (f != SV_BATCH_BLOCK_SIMT && n != kDefaultWidth) continue;
        if (f == SV_BATCH_BLOCK_SIMT && n > L) continue;
        // a resident chain uses one CTA or a few, so its form scales with the
        // chain count up to the SM count: it is timed on every chain of this L;
        // the tensor-core form as one group; the other forms fill the device with
        // one chain's passes
        double rate = 0.0;
        int rc = time_form(b, f == SV_BATCH_RESIDENT ? kv.second : f == SV_BATCH_BLOCK_TC ? group : sample,
                           f, n, &rate);
        if (rc) return rc;
        if (rate > best_rate) {
          best_rate = rate;
          best = f;
          best_n = f == SV_BATCH_BLOCK_TC ? 6 : (f == SV_BATCH_BLOCK_SIMT ? n : 0);
        }
      }
    }
    for (int c : kv.second) {
      b->form[c] = best;
      b->width[c] = best_n;
    }
  }
  return SV_OK;
}

int setup(sv_batch* b) {
  std::vector<int> graph_chains;
  for (int c = 0; c < b->n; ++c) {
    if (b->form[c] == SV_BATCH_RESIDENT) {
      b->res.push_back(c);
    } else {
      int rc = build_graph_form(b, c, b->form[c],
                                b->width[c] > 0 ? b->width[c] : kDefaultWidth);
      if (rc) return rc;
      graph_chains.push_back(c);
    }
  }
  int rc = make_gather(b, graph_chains);
  if (rc) return rc;
  return build_resident(b, b->res, &b->rset);
}

void destroy(sv_batch* b) {
  if (!b) return;
  if (b->g1) cudaGraphExecDestroy(b->g1);
  if (b->gm) cudaGraphExecDestroy(b->gm);
  if (b->gr) cudaGraphExecDestroy(b->gr);
  free_groups(&b->groups);
  b->rset.release();
  cudaFree(b->d_rings);
  cudaFree(b->d_gather);
  for (sv_ctx* c : b->ctx)
    if (c) sv_destroy(c);
  if (b->cap_stream) cudaStreamDestroy(b->cap_stream);
  delete b;
}

}  // namespace

extern "C" {

size_t sv_batch_state_bytes(int n_chains, const int* L) {
  if (n_chains <= 0 || !L) return 0;
  size_t total = 0;
  for (int c = 0; c < n_chains; ++c) {
    if (L[c] < 2 || L[c] > 34) return 0;
    total = (total + kAlign - 1) / kAlign * kAlign;
    total += sizeof(float2) << L[c];
  }
  return total;
}

int sv_batch_create(sv_batch** out, int device, int n_chains, const int* L,
                    const sv_floquet_params* params, const double* product_states,
                    void* state_dev, size_t bytes, int form, void* cuda_stream) {
  if (!out) return SV_EINVAL;
  *out = nullptr;
  if (n_chains <= 0 || !L || !params || !product_states || !state_dev) return SV_EINVAL;
  if (form < SV_BATCH_AUTO || form > SV_BATCH_MULTIGATE) return SV_EINVAL;
  const size_t need = sv_batch_state_bytes(n_chains, L);
  if (need == 0 || bytes < need) return SV_EINVAL;
  if (reinterpret_cast<uintptr_t>(state_dev) % kAlign != 0) return SV_EINVAL;
  for (int c = 0; c < n_chains; ++c) {
    if (!fsv::params_valid(L[c], params[c], nullptr)) return SV_EINVAL;
    if (params[c].n_period_params != 0) return SV_EINVAL;
    if (params[c].h_bonds || params[c].inverse) return SV_EUNSUPPORTED;
  }
  sv_batch* b = new (std::nothrow) sv_batch();
  if (!b) return SV_ENOMEM;
  b->device = device;
  b->n = n_chains;
  b->stream = static_cast<cudaStream_t>(cuda_stream);
  b->base = static_cast<char*>(state_dev);
  b->L.assign(L, L + n_chains);
  b->params.assign(params, params + n_chains);
  b->ctx.assign(n_chains, nullptr);
  size_t off = 0, sp = 0;
  for (int c = 0; c < n_chains; ++c) {
    off = (off + kAlign - 1) / kAlign * kAlign;
    b->off.push_back(off);
    off += sizeof(float2) << L[c];
    b->spinors.push_back(product_states + sp);
    sp += 4 * (size_t)L[c];
  }
  int prev = -1;
  cudaGetDevice(&prev);
  int rc = SV_OK;
  if (cudaSetDevice(device) != cudaSuccess ||
      cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking) != cudaSuccess) {
    cudaGetLastError();
    rc = SV_ECUDA;
  }
  for (int c = 0; c < n_chains && rc == SV_OK; ++c) {
    rc = sv_create(&b->ctx[c], device, SV_C64, cuda_stream);
    if (rc == SV_OK) rc = sv_attach_state(b->ctx[c], b->base + b->off[c], sizeof(float2) << L[c]);
    if (rc == SV_OK) rc = reinit(b, c);
  }
  if (rc == SV_OK) {
    b->form.assign(n_chains, SV_BATCH_PLAIN);
    b->width.assign(n_chains, 0);
    if (form == SV_BATCH_AUTO) {
      rc = autotune(b);
    } else {
      for (int c = 0; c < n_chains; ++c) {
        b->form[c] = form_fits(form, L[c]) ? form : SV_BATCH_PLAIN;
        if (b->form[c] == SV_BATCH_BLOCK_TC || b->form[c] == SV_BATCH_BLOCK_SIMT)
          b->width[c] = kDefaultWidth;
      }
    }
  }
  if (rc == SV_OK) rc = setup(b);
  b->spinors.clear();
  if (prev >= 0) cudaSetDevice(prev);
  if (rc != SV_OK) {
    destroy(b);
    return rc;
  }
  *out = b;
  return SV_OK;
}

int sv_batch_evolve(sv_batch* b, int64_t periods, double* energy_out, double* norm_out) {
  if (!b) return SV_EINVAL;
  if (periods < 0) return bfail(b, SV_EINVAL, "periods must be >= 0");
  int prev = -1;
  cudaGetDevice(&prev);
  cudaSetDevice(b->device);
  struct Restore {
    int d;
    ~Restore() {
      if (d >= 0) cudaSetDevice(d);
    }
  } restore{prev};
  std::vector<int> graph_chains;
  for (int c = 0; c < b->n; ++c)
    if (b->form[c] != SV_BATCH_RESIDENT) graph_chains.push_back(c);
  const bool all_resident = graph_chains.empty();
  if (!b->g1 && !all_resident) {
    int rc = make_graph(b, graph_chains, &b->rset, 1, &b->g1, &b->groups);
    if (rc) return rc;
  }
  if (!b->gm && !all_resident && periods >= b->M) {
    int rc = make_graph(b, graph_chains, &b->rset, b->M, &b->gm, &b->groups);
    if (rc) return rc;
  }
  if (!b->gr && all_resident && periods > 0) {
    int rc = make_graph(b, graph_chains, &b->rset, 0, &b->gr, &b->groups);
    if (rc) return rc;
  }
  const int ring = fsv::ctx_ring_len();
  int64_t done = 0;
  std::vector<double> rbuf;
  // a call that ends early may not have run the copy of its run length
  struct Forget {
    int64_t* run;
    ~Forget() {
      if (run) *run = 0;
    }
  } forget{&b->run};
  while (done < periods) {
    const int64_t chunk = std::min<int64_t>(periods - done, ring);
    int64_t k = 0;
    while (all_resident && k < chunk) {
      // a run of any length is one launch per chain length
      const int64_t n = std::min<int64_t>(chunk - k, 128);
      if (b->run != n) {
        b->run = n;
        BCUDA(cudaMemcpyAsync(b->rset.d_count + 1, &b->run, sizeof(b->run), cudaMemcpyHostToDevice,
                              b->stream),
              "run length");
      }
      BCUDA(cudaGraphLaunch(b->gr, b->stream), "graph launch");
      k += n;
    }
    for (; b->gm && k + b->M <= chunk; k += b->M)
      BCUDA(cudaGraphLaunch(b->gm, b->stream), "graph launch");
    for (; k < chunk; ++k) BCUDA(cudaGraphLaunch(b->g1, b->stream), "graph launch");
    if (!graph_chains.empty() && (energy_out || norm_out)) {
      int rc = read_graph_chains(b, graph_chains, chunk, periods, done, energy_out, norm_out);
      if (rc) return rc;
    }
    for (int c : graph_chains) fsv::ctx_advance(b->ctx[c], chunk);
    if (!b->res.empty() && (energy_out || norm_out)) {
      // the slots written, every chain's pair of a slot together
      const size_t row = 2 * b->res.size(), at = (size_t)(b->counter % ring);
      const size_t head = std::min<size_t>(chunk, ring - at);
      rbuf.resize(row * chunk);
      BCUDA(cudaMemcpyAsync(rbuf.data(), b->rset.d_ring + row * at, sizeof(double) * row * head,
                            cudaMemcpyDeviceToHost, b->stream),
            "resident ring readback");
      if (head < (size_t)chunk)
        BCUDA(cudaMemcpyAsync(rbuf.data() + row * head, b->rset.d_ring,
                              sizeof(double) * row * (chunk - head), cudaMemcpyDeviceToHost, b->stream),
              "resident ring readback");
      BCUDA(cudaStreamSynchronize(b->stream), "synchronize");
      for (size_t r = 0; r < b->res.size(); ++r) {
        const int c = b->res[r];
        const double* src = rbuf.data() + 2 * b->rset.place[r];
        for (int64_t q = 0; q < chunk; ++q, src += row) {
          if (energy_out) energy_out[(size_t)c * periods + done + q] = src[0];
          if (norm_out) norm_out[(size_t)c * periods + done + q] = src[1];
        }
      }
    }
    b->counter += chunk;
    done += chunk;
  }
  BCUDA(cudaStreamSynchronize(b->stream), "synchronize");
  forget.run = nullptr;
  return SV_OK;
}

int sv_batch_forms(const sv_batch* b, int* form_out) {
  if (!b || !form_out) return SV_EINVAL;
  for (int c = 0; c < b->n; ++c) form_out[c] = b->form[c];
  return SV_OK;
}

int sv_batch_widths(const sv_batch* b, int* n_out) {
  if (!b || !n_out) return SV_EINVAL;
  for (int c = 0; c < b->n; ++c) n_out[c] = b->width[c];
  return SV_OK;
}

const char* sv_batch_last_error(const sv_batch* b) { return b ? b->err.c_str() : ""; }

void sv_batch_destroy(sv_batch* b) { destroy(b); }

}  // extern "C"
