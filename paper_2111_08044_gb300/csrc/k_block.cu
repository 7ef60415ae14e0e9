// Block form: host construction of the pass descriptors and the CUDA-core
// FP32 block pass.  The CUDA-core pass applies any window width n <= 7 and
// any tile height; it serves chains too short for 128-row tensor-core tiles
// and is the reference form the tensor-core pass is checked against.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <map>

#include "sv_block.h"
#include "sv_device.cuh"

namespace fsv {

namespace {

using namespace dev;

constexpr int kSimtThreads = 512;

// position of site s while the window starts at lo (see sv_block.h)
int pos_of(int L, int n, int lo, int s) {
  (void)L;
  if (s >= lo && s < lo + n) return s - lo;
  if (s < lo) return n + s;
  return s;
}

// site held at position p while the window starts at lo
int site_at(int L, int n, int lo, int p) {
  (void)L;
  if (p < n) return lo + p;
  if (p < n + lo) return p - n;
  return p;
}

template <int N>
__global__ void __launch_bounds__(kSimtThreads) k_block_simt(float2* __restrict__ psi,
                                                             PassArgs pa) {
  constexpr int D = 1 << N;
  constexpr int DP = D + 1;  // padded row stride (bank spread)
  constexpr int CH = D < 16 ? D : 16;
  extern __shared__ float2 tile[];
  const int R = pa.R, rows = 1 << R, a = pa.a, L = pa.L;
  const int nel = rows * D;
  const int nitems = rows * (D / CH);
  const int nbits = N + R;
  Diag<float> dg;
  if (pa.diag) dg.init(pa.ep, L);
  const float sc = (float)renorm_scale(pa.ep.rn);
  double eacc = 0.0, nacc = 0.0;
  for (long long t = blockIdx.x; t < pa.ntiles; t += gridDim.x) {
    const uint64_t tlo = (uint64_t)t & ((1ull << (a - N)) - 1);
    const uint64_t thi = (uint64_t)t >> (a - N);
    const uint64_t base = (tlo << N) | (thi << (a + R));
    for (int e = threadIdx.x; e < nel; e += blockDim.x) {
      const int r = e >> N, c = e & (D - 1);
      tile[r * DP + c] = psi[base + ((uint64_t)r << a) + c];
    }
    __syncthreads();
    float2 acc[2][CH];
    int rr[2], cb[2];
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      const int item = threadIdx.x + it * blockDim.x;
      rr[it] = item % rows;
      cb[it] = item / rows;
      // each output starts from its row's largest entry's FP32 residual
      // times that entry's amplitude: a sum started from a bare product
      // with a fixed entry rounds with an error that correlates with the
      // result (for passes of few gates, with one dominant entry per row,
      // it biased the norm by 1e-8 per period); the residual term varies
      // independently of that rounding grid and takes the bias out
#pragma unroll
      for (int j = 0; j < CH; ++j) acc[it][j] = make_float2(0.f, 0.f);
      if (item < nitems) {
#pragma unroll
        for (int j = 0; j < CH; ++j) {
          const float4 ld = __ldg(&pa.Ulead[cb[it] * CH + j]);
          acc[it][j] = cmac(acc[it][j], make_float2(ld.x, ld.y), tile[rr[it] * DP + (int)ld.z]);
        }
        for (int k = 0; k < D; ++k) {
          const float2 v = tile[rr[it] * DP + k];
#pragma unroll
          for (int j = 0; j < CH; ++j)
            acc[it][j] = cmac(acc[it][j], __ldg(&pa.U[(cb[it] * CH + j) * D + k]), v);
        }
      }
    }
    __syncthreads();
    // write the result at its place in the next window's layout
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      const int item = threadIdx.x + it * blockDim.x;
      if (item >= nitems) continue;
#pragma unroll
      for (int j = 0; j < CH; ++j) {
        const int y = (rr[it] << N) | (cb[it] * CH + j);
        int yo = 0;
        for (int q = 0; q < nbits; ++q) yo |= ((y >> q) & 1) << pa.sigma[q];
        tile[(yo >> N) * DP + (yo & (D - 1))] = make_float2(acc[it][j].x * sc, acc[it][j].y * sc);
      }
    }
    __syncthreads();
    float es = 0.f, ns = 0.f;
    for (int e = threadIdx.x; e < nel; e += blockDim.x) {
      const int r = e >> N, c = e & (D - 1);
      const float2 v = tile[r * DP + c];
      const uint64_t x = base + ((uint64_t)r << a) + c;
      psi[x] = v;
      if (pa.x_mask) {
        for (int j = 0; j < N; ++j)
          if ((pa.x_mask >> j) & 1) {
            const int yf = e ^ (1 << pa.sigma[j]);
            es += pa.cx[j] * cdotre(v, tile[(yf >> N) * DP + (yf & (D - 1))]);
          }
      }
      if (pa.diag) {
        const float p = cabs2(v);
        ns += p;
        es += p * dg(to_natural(x, N, pa.diag_lo));
      }
    }
    eacc += (double)es;
    nacc += (double)ns;
    __syncthreads();
  }
  if (pa.partial) block_store_pair(eacc, nacc, pa.partial);
}

template <int N>
cudaError_t prepare_simt_n() {
  return cudaFuncSetAttribute(k_block_simt<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(sizeof(float2) * 128 * ((1 << N) + 1)));
}

template <int N>
cudaError_t launch_simt_n(const PassArgs& pa, void* psi, int grid, cudaStream_t s) {
  const size_t smem = sizeof(float2) * ((size_t)1 << pa.R) * ((1 << N) + 1);
  k_block_simt<N><<<grid, kSimtThreads, smem, s>>>(static_cast<float2*>(psi), pa);
  return cudaGetLastError();
}

// Opt the CUDA-core pass for width n into its shared-memory size (called at
// build time, outside any stream capture).
cudaError_t prepare_simt(int n) {
  switch (n) {
    case 2: return prepare_simt_n<2>();
    case 3: return prepare_simt_n<3>();
    case 4: return prepare_simt_n<4>();
    case 5: return prepare_simt_n<5>();
    case 6: return prepare_simt_n<6>();
    case 7: return prepare_simt_n<7>();
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_block_simt(const PassArgs& pa, void* psi, int grid, cudaStream_t s) {
  switch (pa.n) {
    case 2: return launch_simt_n<2>(pa, psi, grid, s);
    case 3: return launch_simt_n<3>(pa, psi, grid, s);
    case 4: return launch_simt_n<4>(pa, psi, grid, s);
    case 5: return launch_simt_n<5>(pa, psi, grid, s);
    case 6: return launch_simt_n<6>(pa, psi, grid, s);
    case 7: return launch_simt_n<7>(pa, psi, grid, s);
    default: return cudaErrorInvalidValue;
  }
}

// a pass's relabel moves the window by at most its 7 row bits
constexpr int kMaxShiftRows = 7;

std::string block_tile_layout(int L, int n, int R, int lo, int lo_next, int* a_out,
                              int8_t* sigma) {
  const int lo_min = std::min(lo, lo_next);
  const int delta = std::abs(lo_next - lo);
  if (delta > R) return "window moves by more than the tile's row bits";
  const int a = (R == L - n) ? n : std::max(n, std::min(n + lo_min, L - R));
  if (!(a <= n + lo_min && n + lo_min + delta <= a + R)) return "row bits miss moved sites";
  for (int q = 0; q < n + R; ++q) {
    const int p = q < n ? q : a + q - n;
    const int s = site_at(L, n, lo, p);
    const int po = pos_of(L, n, lo_next, s);
    int qo;
    if (po < n) qo = po;
    else if (po >= a && po < a + R) qo = po - a + n;
    else return "site leaves the tile";
    sigma[q] = (int8_t)qo;
  }
  for (int p = 0; p < L; ++p) {
    const bool in_tile = p < n || (p >= a && p < a + R);
    if (!in_tile && site_at(L, n, lo, p) != site_at(L, n, lo_next, p))
      return "layout change outside the tile";
  }
  *a_out = a;
  return std::string();
}

int block_build(int L, const std::vector<Gate2>& gates, const Observable& obs, int n,
                int split, const LaunchCfg& cfg, bool cyclic, cudaStream_t s,
                BlockPlan** out, std::string* msg) {
  *out = nullptr;
  if (split != SV_SPLIT_BF16X3 && split != SV_SPLIT_FP32) {
    *msg = "unknown split";
    return SV_EINVAL;
  }
  BlockPlan* bp = new BlockPlan();
  bp->L = L;
  bp->n = n;
  bp->R = std::min(7, L - n);
  bp->split = split;
  bp->cfg = cfg;
  bp->passes = fusion_plan(L, gates, n, cyclic);
  const int P = (int)bp->passes.size();
  bp->start = bp->passes[0].lo;
  const int R = bp->R;
  bp->tensor_cores = split == SV_SPLIT_BF16X3 && block_tc_supported(L, n);
  const long long ntiles = 1ll << (L - n - R);
  const int per_sm = bp->tensor_cores ? 1 : 2;
  long long grid = std::min<long long>(ntiles, (long long)cfg.num_sms * per_sm);
  if (cfg.min_tiles_per_cta > 0) grid = std::min<long long>(grid, ntiles / cfg.min_tiles_per_cta);
  bp->grid = (int)std::max<long long>(1, grid);
  bp->maxb = bp->grid;
  auto fail = [&](const std::string& m) {
    *msg = m;
    block_free(bp);
    return SV_EINVAL;
  };
  // The launches: the period's P passes, each writing the next pass's layout
  // (the last one the start's); when the start is not site 0, the last
  // period of an evolution ends with a variant of the last pass that writes
  // toward the natural layout (plus relabel steps if it is more than 7 sites
  // away), and an evolution begins with relabel steps from the natural
  // layout to the start.  A relabel step applies the identity.
  struct Op {
    int src;  // pass whose unitary and measurements it applies, -1: identity
    int lo, lo_next;
  };
  std::vector<Op> ops;
  for (int k = 0; k < P; ++k) ops.push_back({k, bp->passes[k].lo, bp->passes[(k + 1) % P].lo});
  auto step = [](int from, int to) {
    return from + std::max(-kMaxShiftRows, std::min(kMaxShiftRows, to - from));
  };
  for (int k = 0; k < P; ++k) bp->seq_cyc.push_back(k);
  if (bp->start == 0) {
    bp->seq_exit = bp->seq_cyc;
  } else {
    for (int k = 0; k + 1 < P; ++k) bp->seq_exit.push_back(k);
    int lo = bp->passes[P - 1].lo, nx = step(lo, 0);
    bp->seq_exit.push_back((int)ops.size());
    ops.push_back({P - 1, lo, nx});
    while (nx != 0) {
      lo = nx;
      nx = step(lo, 0);
      bp->seq_exit.push_back((int)ops.size());
      ops.push_back({-1, lo, nx});
    }
    lo = 0;
    while (lo != bp->start) {
      nx = step(lo, bp->start);
      bp->seq_entry.push_back((int)ops.size());
      ops.push_back({-1, lo, nx});
      lo = nx;
    }
    lo = bp->start;
    while (lo != 0) {  // from the period layout back to the natural one
      nx = step(lo, 0);
      bp->seq_leave.push_back((int)ops.size());
      ops.push_back({-1, lo, nx});
      lo = nx;
    }
  }
  const BlockPass identity_pass = [&]() {
    BlockPass ip;
    ip.n = n;
    ip.U.assign((size_t)1 << (2 * n), cd(0.0, 0.0));
    for (size_t e = 0; e < ((size_t)1 << n); ++e) ip.U[e * ((size_t)1 << n) + e] = 1.0;
    return ip;
  }();
  std::vector<int> slot_of(P, -1);
  int slot = 0;
  for (size_t k = 0; k < ops.size(); ++k) {
    const BlockPass& ps = ops[k].src >= 0 ? bp->passes[ops[k].src] : identity_pass;
    const int lo = ops[k].lo;
    const int lo_next = ops[k].lo_next;
    PassArgs pa;
    pa.L = L;
    pa.n = n;
    pa.R = R;
    pa.lo = lo;
    pa.ntiles = ntiles;
    const std::string why = block_tile_layout(L, n, R, lo, lo_next, &pa.a, pa.sigma);
    if (!why.empty()) return fail(why);
    if (bp->tensor_cores) block_tc_layout(pa);
    for (int s : obs.general ? std::vector<int>() : ps.x_sites) {
      const int j = s - lo;
      if (j < 0 || j >= n) return fail("measured site outside window");
      pa.x_mask |= 1u << j;
      pa.cx[j] = (float)obs.cx[s];
    }
    pa.diag = ps.diag && !obs.general ? 1 : 0;
    if (pa.diag) {
      pa.diag_lo = lo_next;  // the output's layout (natural order: window at 0)
      pa.ep.flags = EPI_DIAG;
      pa.ep.J = obs.J;
      pa.ep.cz_first = obs.cz[0];
      pa.ep.cz_last = obs.cz[L - 1];
      pa.ep.cz_bulk = L >= 3 ? obs.cz[1] : 0.0;
      pa.diag_f[0] = (float)pa.ep.J;
      pa.diag_f[1] = (float)pa.ep.cz_bulk;
      pa.diag_f[2] = (float)pa.ep.cz_first;
      pa.diag_f[3] = (float)pa.ep.cz_last;
      pa.diag_f[4] = (float)(pa.ep.cz_bulk * (L - 2) + pa.ep.cz_first + pa.ep.cz_last);
      // per window bit: its site (window bit j is site lo + j in every
      // layout), its field, and which of its neighbours lie outside the window
      int site[8];
      for (int j = 0; j < n; ++j) site[j] = lo + j;
      for (int j = 0; j < n; ++j) {
        const int g = site[j];
        const double czg = g == 0 ? pa.ep.cz_first : (g == L - 1 ? pa.ep.cz_last : pa.ep.cz_bulk);
        int inside = 0;
        for (int k = 0; k < 2; ++k) {
          const int nb = k == 0 ? g - 1 : g + 1;
          pa.diag_nb[j][k] = -1;
          if (nb < 0 || nb >= L) continue;
          bool in_window = false;
          for (int jj = 0; jj < n; ++jj) in_window = in_window || site[jj] == nb;
          if (in_window) ++inside;
          else pa.diag_nb[j][k] = (int8_t)nb;
        }
        pa.diag_lin0[j] = (float)(-2.0 * (czg + pa.ep.J * inside));
      }
    }
    if (pa.x_mask || pa.diag) {
      // the exit variant of the last pass fills that pass's partials slot
      if (ops[k].src >= 0 && slot_of[ops[k].src] >= 0) pa.slot = slot_of[ops[k].src];
      else pa.slot = slot++;
      if (ops[k].src >= 0) slot_of[ops[k].src] = pa.slot;
    }
    bp->args.push_back(pa);
  }
  const int NA = (int)bp->args.size();
  bp->nslots = slot;
  // device buffers
  const size_t dim = (size_t)1 << n;
  // the operands of the P passes and of the identity (index P), rounded
  // close to unitary (host_round.cpp); every launch takes its source's copy
  const int NU = P + 1;
  std::vector<float2> uu(bp->tensor_cores ? 0 : (size_t)NU * dim * dim);
  std::vector<float4> ul(bp->tensor_cores ? 0 : (size_t)NU * dim);
  std::vector<std::vector<uint32_t>> uw(bp->tensor_cores ? NU : 0);
  round_passes_parallel(NU, [&](int k) {
    const std::vector<cd>& U = k < P ? bp->passes[k].U : identity_pass.U;
    if (bp->tensor_cores) block_tc_pack_w(n, U, uw[k]);
    else round_unitary_fp32((int)dim, U.data(), &uu[k * dim * dim], &ul[k * dim]);
  });
  std::vector<float2> hu(bp->tensor_cores ? 0 : (size_t)NA * dim * dim);
  std::vector<float4> hl(bp->tensor_cores ? 0 : (size_t)NA * dim);
  std::vector<std::vector<uint32_t>> hw(bp->tensor_cores ? NA : 0);
  for (int k = 0; k < NA; ++k) {
    const int from = ops[k].src >= 0 ? ops[k].src : P;
    if (bp->tensor_cores) {
      hw[k] = uw[from];
    } else {
      std::copy(uu.begin() + from * dim * dim, uu.begin() + (from + 1) * dim * dim,
                hu.begin() + k * dim * dim);
      std::copy(ul.begin() + from * dim, ul.begin() + (from + 1) * dim, hl.begin() + k * dim);
    }
  }
  if (!bp->tensor_cores &&
      (cudaMalloc(&bp->d_U, sizeof(float2) * hu.size()) != cudaSuccess ||
       upload(bp->d_U, hu.data(), sizeof(float2) * hu.size(), s) != cudaSuccess ||
       cudaMalloc(&bp->d_Ulead, sizeof(float4) * hl.size()) != cudaSuccess ||
       upload(bp->d_Ulead, hl.data(), sizeof(float4) * hl.size(), s) != cudaSuccess)) {
    cudaGetLastError();
    *msg = "unitary upload failed";
    block_free(bp);
    return SV_ENOMEM;
  }
  if (bp->tensor_cores) {
    bp->w_bytes_per_pass = block_tc_w_bytes(n);
    std::vector<uint32_t> all;
    for (int k = 0; k < NA; ++k) all.insert(all.end(), hw[k].begin(), hw[k].end());
    if (cudaMalloc(&bp->d_W, all.size() * sizeof(uint32_t)) != cudaSuccess ||
        upload(bp->d_W, all.data(), all.size() * sizeof(uint32_t), s) != cudaSuccess) {
      cudaGetLastError();
      *msg = "operand upload failed";
      block_free(bp);
      return SV_ENOMEM;
    }
  }
  const size_t pbytes = sizeof(double) * 2 * std::max(1, bp->nslots) * (size_t)bp->maxb;
  if (cudaMalloc(&bp->d_partials, pbytes) != cudaSuccess ||
      cudaMemsetAsync(bp->d_partials, 0, pbytes, s) != cudaSuccess) {
    cudaGetLastError();
    *msg = "partials allocation failed";
    block_free(bp);
    return SV_ENOMEM;
  }
  for (int k = 0; k < NA; ++k) {
    PassArgs& pa = bp->args[k];
    if (bp->d_U) {
      pa.U = bp->d_U + (size_t)k * dim * dim;
      pa.Ulead = bp->d_Ulead + (size_t)k * dim;
    }
    if (bp->d_W)
      pa.W = static_cast<const char*>(bp->d_W) + (size_t)k * bp->w_bytes_per_pass;
    if (pa.slot >= 0) pa.partial = bp->d_partials + 2 * (size_t)pa.slot * bp->maxb;
  }
  if (bp->tensor_cores) {
    if (block_tc_prepare() != cudaSuccess || cudaMalloc(&bp->d_status, sizeof(int)) != cudaSuccess ||
        cudaMemsetAsync(bp->d_status, 0, sizeof(int), s) != cudaSuccess) {
      cudaGetLastError();
      *msg = "tensor-core pass set-up failed";
      block_free(bp);
      return SV_ECUDA;
    }
  }
  if (prepare_simt(n) != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess) {
    cudaGetLastError();
    *msg = "shared-memory opt-in or upload failed";
    block_free(bp);
    return SV_ECUDA;
  }
  *out = bp;
  return SV_OK;
}

void block_set_renorm(BlockPlan* bp, const Renorm& rn) {
  if (!bp->args.empty()) bp->args[0].ep.rn = rn;
}

void block_info(const BlockPlan* bp, int* passes, int* launches) {
  if (passes) *passes = (int)bp->passes.size();
  if (launches) *launches = (int)bp->passes.size() + 1;
}

size_t block_upload_bytes(const BlockPlan* bp) {
  const size_t P = bp->args.size();
  const size_t dim = (size_t)1 << bp->n;
  const size_t u = bp->tensor_cores ? 0 : sizeof(float2) * dim * dim + sizeof(float4) * dim;
  return P * (u + bp->w_bytes_per_pass);
}

namespace {

// TMA descriptors embed the state address: (re)build them for psi.
cudaError_t ensure_maps(BlockPlan* bp, void* psi) {
  if (!bp->tensor_cores || bp->maps_psi == psi) return cudaSuccess;
  const size_t mb = block_tc_map_bytes();
  bp->maps.assign(mb * bp->args.size(), 0);
  for (size_t k = 0; k < bp->args.size(); ++k)
    if (block_tc_make_map(bp->args[k], psi, bp->maps.data() + k * mb) != SV_OK)
      return cudaErrorInvalidValue;
  bp->maps_psi = psi;
  return cudaSuccess;
}

cudaError_t launch_pass(BlockPlan* bp, size_t k, void* psi, cudaStream_t s) {
  if (bp->tensor_cores)
    return launch_block_tc(bp->args[k], psi, bp->maps.data() + k * block_tc_map_bytes(),
                           bp->d_status, bp->grid, s, bp->cfg.alone());
  return launch_block_simt(bp->args[k], psi, bp->grid, s);
}

}  // namespace

int block_status(BlockPlan* bp, cudaStream_t s) {
  if (!bp || !bp->d_status) return 0;
  int h = 0;
  if (cudaMemcpyAsync(&h, bp->d_status, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return -1;
  return h;
}

cudaError_t block_enqueue_entry(BlockPlan* bp, void* psi, cudaStream_t s) {
  cudaError_t e = ensure_maps(bp, psi);
  if (e != cudaSuccess) return e;
  for (int k : bp->seq_entry) {
    e = launch_pass(bp, k, psi, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t block_enqueue_leave(BlockPlan* bp, void* psi, cudaStream_t s) {
  cudaError_t e = ensure_maps(bp, psi);
  if (e != cudaSuccess) return e;
  for (int k : bp->seq_leave) {
    e = launch_pass(bp, k, psi, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t block_enqueue_period(BlockPlan* bp, void* psi, long long* counter, double* ring,
                                 int ring_len, cudaStream_t s, bool last) {
  cudaError_t e = ensure_maps(bp, psi);
  if (e != cudaSuccess) return e;
  for (int k : last ? bp->seq_exit : bp->seq_cyc) {
    e = launch_pass(bp, k, psi, s);
    if (e != cudaSuccess) return e;
  }
  return launch_period_reduce(bp->d_partials, (long long)bp->nslots * bp->maxb, bp->L, ring,
                              ring_len, counter, 1, s);
}

cudaError_t block_enqueue_period_events(BlockPlan* bp, void* psi, long long* counter,
                                        double* ring, int ring_len, cudaStream_t s,
                                        cudaEvent_t* ev, bool last) {
  cudaError_t e = ensure_maps(bp, psi);
  if (e != cudaSuccess) return e;
  // events around the period's P passes (the exit variant's relabel steps,
  // if any, fall inside the last pass's interval) and the reduce
  const std::vector<int>& seq = last ? bp->seq_exit : bp->seq_cyc;
  const size_t P = bp->seq_cyc.size();
  for (size_t k = 0; k < seq.size(); ++k) {
    if (k < P) {
      e = cudaEventRecord(ev[k], s);
      if (e != cudaSuccess) return e;
    }
    e = launch_pass(bp, (size_t)seq[k], psi, s);
    if (e != cudaSuccess) return e;
  }
  e = cudaEventRecord(ev[P], s);
  if (e != cudaSuccess) return e;
  e = launch_period_reduce(bp->d_partials, (long long)bp->nslots * bp->maxb, bp->L, ring,
                           ring_len, counter, 1, s);
  if (e != cudaSuccess) return e;
  return cudaEventRecord(ev[P + 1], s);
}

// ------------------------------------------------------------ chain groups

namespace {
struct BlockGroup {
  std::vector<GroupMember> m;
  std::vector<PassArgs> ops;        // structure of each pass, ntiles over the group
  GroupChain* d_chains = nullptr;   // [passes][chains]
  double* d_part = nullptr;         // [chains][measuring slots][pairs] (energy, norm) pairs
  int pairs = 0;                    // of a slot: its CTAs, or 1 (tile sums)
  float2* d_sums = nullptr;         // tile sums: [chains][slots][tiles of a chain][rows]
  int nt_log2 = 0;
};
struct TileSumItem {
  const float2* sums = nullptr;
  double* pair = nullptr;
  long long first = 0, tiles = 0;  // the chain's tiles among the group's total
  long long total = 0;
  int ranges = 0;
};
}  // namespace

struct BlockSet {
  std::vector<BlockGroup> groups;
  // CTAs of each group in the k-th passes of a period (0: it has fewer)
  std::vector<std::vector<int>> share;
  ReduceItem* d_reduce = nullptr;   // [chains]
  TileSumItem* d_tile_sums = nullptr;  // [chains][slots] (together; else null)
  int chains = 0, num_sms = 0, ntile_sums = 0;
};

namespace {
template <typename T, size_t N>
bool same_array(const T (&x)[N], const T (&y)[N]) {
  return std::memcmp(x, y, sizeof(x)) == 0;
}
bool same_pass(const PassArgs& x, const PassArgs& y) {
  return x.L == y.L && x.n == y.n && x.R == y.R && x.a == y.a && x.lo == y.lo &&
         x.ntiles == y.ntiles && x.x_mask == y.x_mask && x.diag == y.diag &&
         x.diag_lo == y.diag_lo && same_array(x.diag_nb, y.diag_nb) &&
         same_array(x.sigma, y.sigma) && same_array(x.rowvec, y.rowvec) &&
         same_array(x.spos, y.spos) && same_array(x.ssig, y.ssig) && x.st_ndims == y.st_ndims &&
         x.st_tlo_dim == y.st_tlo_dim && x.st_tlo_shift == y.st_tlo_shift &&
         x.st_thi_dim == y.st_thi_dim && x.st_thi_shift == y.st_thi_shift &&
         x.slot == y.slot && (x.partial == nullptr) == (y.partial == nullptr);
}
bool renorm_active(const PassArgs& pa) { return pa.ep.rn.ring && pa.ep.rn.every > 0; }
}  // namespace

bool block_same_structure(const BlockPlan* a, const BlockPlan* b) {
  if (!a || !b || !a->tensor_cores || !b->tensor_cores) return false;
  if (a->L != b->L || a->n != b->n || a->start != b->start || a->nslots != b->nslots ||
      a->args.size() != b->args.size() || a->seq_cyc != b->seq_cyc ||
      a->seq_exit != b->seq_exit || a->seq_entry != b->seq_entry || a->seq_leave != b->seq_leave)
    return false;
  for (size_t k = 0; k < a->args.size(); ++k)
    if (!same_pass(a->args[k], b->args[k])) return false;
  return true;
}

namespace {

constexpr int kGroupRows = 128;      // rows of a tile
constexpr int kTileSumThreads = 512;

// A chain's (energy, norm) of one slot from its tile sums: the group's tiles in
// `ranges` contiguous ranges, a row's sums over a range in order, compensated, then
// everything in FP64.
__global__ void __launch_bounds__(kTileSumThreads) k_tile_sums(const TileSumItem* __restrict__ items) {
  __shared__ double red[2][kTileSumThreads / 32];
  const TileSumItem it = items[blockIdx.x];
  const int row = threadIdx.x & (kGroupRows - 1);
  const long long end = it.first + it.tiles;
  double e = 0.0, n = 0.0;
  grid_wait();
  grid_trigger();
  // range v holds the tiles from v total / ranges on
  long long v = it.first * it.ranges / it.total;
  while (v > 0 && v * it.total / it.ranges > it.first) --v;
  while ((v + 1) * it.total / it.ranges <= it.first) ++v;
  for (v += threadIdx.x / kGroupRows; v < it.ranges; v += kTileSumThreads / kGroupRows) {
    long long a = v * it.total / it.ranges, b = (v + 1) * it.total / it.ranges;
    if (a >= end) break;
    if (a < it.first) a = it.first;
    if (b > end) b = end;
    float es = 0.f, ec = 0.f, ns = 0.f, nc = 0.f;
    for (long long t = a; t < b; ++t) {
      const float2 s = it.sums[(t - it.first) * kGroupRows + row];
      const float ye = __fsub_rn(s.x, ec), te = __fadd_rn(es, ye);
      ec = __fsub_rn(__fsub_rn(te, es), ye);
      es = te;
      const float yn = __fsub_rn(s.y, nc), tn = __fadd_rn(ns, yn);
      nc = __fsub_rn(__fsub_rn(tn, ns), yn);
      ns = tn;
    }
    e += (double)es - (double)ec;
    n += (double)ns - (double)nc;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    e += __shfl_xor_sync(0xffffffffu, e, o);
    n += __shfl_xor_sync(0xffffffffu, n, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = e;
    red[1][threadIdx.x >> 5] = n;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    e = n = 0.0;
    for (int w = 0; w < kTileSumThreads / 32; ++w) {
      e += red[0][w];
      n += red[1][w];
    }
    it.pair[0] = e;
    it.pair[1] = n;
  }
}

// CTAs (and ranges of tiles) of a group of `tiles` tiles by itself: one an SM, each
// with at least kGroupMinTiles tiles.
constexpr long long kGroupMinTiles = 4;
int group_ranges(long long tiles, int num_sms) {
  return (int)std::max<long long>(1, std::min<long long>(num_sms, tiles / kGroupMinTiles));
}

int group_build(const std::vector<GroupMember>& mem, int num_sms, bool tile_sums, cudaStream_t s,
                BlockGroup* g, std::string* msg) {
  if (mem.empty()) return SV_EINVAL;
  const BlockPlan* ref = mem[0].plan;
  for (const GroupMember& x : mem) {
    if (!block_same_structure(ref, x.plan)) {
      *msg = "the chains' plans differ";
      return SV_EINVAL;
    }
    for (const PassArgs& pa : x.plan->args)
      if (renorm_active(pa)) {
        *msg = "a group does not fold renormalisation";
        return SV_EUNSUPPORTED;
      }
  }
  const long long nt = ref->args[0].ntiles;
  int lg = 0;
  while ((1ll << lg) < nt) ++lg;
  for (const PassArgs& pa : ref->args)
    if (pa.ntiles != nt || (1ll << lg) != nt) {
      *msg = "tile counts differ between passes";
      return SV_EINVAL;
    }
  const size_t C = mem.size(), K = ref->args.size();
  g->m = mem;
  g->nt_log2 = lg;
  g->ops = ref->args;
  for (PassArgs& pa : g->ops) {
    pa.ntiles = nt * (long long)C;
    pa.W = nullptr;        // per chain
    pa.partial = nullptr;  // per chain
  }
  // partial sums: the chains' own buffers hold one pair per CTA of their
  // own launches; a group has its own (zero where a CTA meets no tile of the chain)
  const int S = std::max(1, ref->nslots);
  g->pairs = tile_sums ? 1 : group_ranges(nt * (long long)C, num_sms);
  const size_t part_pairs = C * (size_t)S * g->pairs;
  const size_t chain_sums = (size_t)nt * kGroupRows;
  std::vector<GroupChain> hc(K * C);
  std::vector<uint8_t> maps(block_tc_map_bytes());
  if (cudaMalloc(&g->d_part, sizeof(double) * 2 * part_pairs) != cudaSuccess ||
      (tile_sums && cudaMalloc(&g->d_sums, sizeof(float2) * C * S * chain_sums) != cudaSuccess)) {
    cudaGetLastError();
    *msg = "group partials allocation";
    return SV_ENOMEM;
  }
  for (size_t k = 0; k < K; ++k)
    for (size_t c = 0; c < C; ++c) {
      const PassArgs& pa = mem[c].plan->args[k];
      GroupChain& gc = hc[k * C + c];
      if (block_tc_make_map(pa, mem[c].psi, maps.data()) != SV_OK) {
        *msg = "tensor map";
        return SV_ECUDA;
      }
      std::memcpy(gc.map_in, maps.data(), sizeof(gc.map_in));
      std::memcpy(gc.map_out, maps.data() + sizeof(gc.map_in), sizeof(gc.map_out));
      gc.W = pa.W;
      if (pa.slot >= 0 && tile_sums) gc.partial = g->d_sums + (c * S + pa.slot) * chain_sums;
      else if (pa.slot >= 0) gc.partial = g->d_part + 2 * (c * S + pa.slot) * (size_t)g->pairs;
      std::memcpy(gc.cx, pa.cx, sizeof(gc.cx));
      std::memcpy(gc.diag_f, pa.diag_f, sizeof(gc.diag_f));
      std::memcpy(gc.diag_lin0, pa.diag_lin0, sizeof(gc.diag_lin0));
    }
  cudaError_t e = cudaMalloc(&g->d_chains, sizeof(GroupChain) * hc.size());
  if (e == cudaSuccess) e = cudaMemsetAsync(g->d_part, 0, sizeof(double) * 2 * part_pairs, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(g->d_chains, hc.data(), sizeof(GroupChain) * hc.size(),
                        cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // the host array is freed below
  if (e != cudaSuccess) {
    cudaGetLastError();
    *msg = "group upload";
    return SV_ECUDA;
  }
  return SV_OK;
}

// CTAs of groups of t[g] tiles in one launch (0: not part of it), at most one an SM:
// one each, then one more for the group with most tiles a CTA.
std::vector<int> cta_shares(const std::vector<long long>& t, int num_sms) {
  std::vector<int> n(t.size(), 0);
  int left = num_sms;
  for (size_t g = 0; g < t.size(); ++g)
    if (t[g] > 0) {
      n[g] = 1;
      --left;
    }
  for (; left > 0; --left) {
    size_t most = t.size();
    for (size_t g = 0; g < t.size(); ++g)
      if (t[g] > n[g] && (most == t.size() || t[g] * n[most] > t[most] * n[g])) most = g;
    if (most == t.size()) break;  // one tile a CTA
    ++n[most];
  }
  return n;
}

// One launch (or several, of kGroupsPerLaunch groups each) of op[g] of every group g with
// CTAs in share.
cudaError_t set_pass(BlockSet* set, const std::vector<int>& op, const std::vector<int>& share,
                     bool overlap, cudaStream_t s) {
  GroupPasses p;
  int n = 0, ctas = 0;
  auto launch = [&]() {
    const cudaError_t e =
        n ? launch_block_tc_groups(p, n, set->groups[0].m[0].plan->d_status, overlap, s) : cudaSuccess;
    n = ctas = 0;
    return e;
  };
  for (size_t g = 0; g < set->groups.size(); ++g) {
    if (share[g] == 0) continue;
    const BlockGroup& gr = set->groups[g];
    GroupPass& q = p.g[n++];
    q.pa = gr.ops[op[g]];
    q.chains = gr.d_chains + (size_t)op[g] * gr.m.size();
    q.nt_log2 = gr.nt_log2;
    q.tile_sums = gr.d_sums != nullptr;
    q.cta_end = ctas += share[g];
    if (n == kGroupsPerLaunch) {
      const cudaError_t e = launch();
      if (e != cudaSuccess) return e;
    }
  }
  return launch();
}

// The passes seq(plan) of every group, the k-th of all of them together.
template <typename Seq>
cudaError_t set_sequence(BlockSet* set, const Seq& seq, bool overlap, cudaStream_t s) {
  const size_t G = set->groups.size();
  for (size_t k = 0;; ++k) {
    std::vector<long long> t(G, 0);
    std::vector<int> op(G, 0);
    bool any = false;
    for (size_t g = 0; g < G; ++g) {
      const std::vector<int>& q = seq(set->groups[g].m[0].plan);
      if (k >= q.size()) continue;
      any = true;
      op[g] = q[k];
      t[g] = set->groups[g].ops[0].ntiles;
    }
    if (!any) return cudaSuccess;
    const std::vector<int> share =
        set->d_tile_sums ? cta_shares(t, set->num_sms) : std::vector<int>(1, set->groups[0].pairs);
    const cudaError_t e = set_pass(set, op, share, overlap, s);
    if (e != cudaSuccess) return e;
  }
}

}  // namespace

bool block_groups_together(const std::vector<std::vector<GroupMember>>& groups, const LaunchCfg& cfg) {
  // Below three tiles an SM in all, one launch on one tile or a few a CTA gains: 48
  // chains of 14 sites (96 tiles) take 98 us a period, 24 of 15 to 17 sites (224)
  // 125 us, 48 of them (448) 172 us; in launches of their own, of four tiles a CTA,
  // 153, 165 and 185 us.  From there on these overlap better: 24 chains of 15 to 19
  // sites (595) 190 us, together 213 us.
  constexpr long long kTogether = 3;
  long long tiles = 0;
  for (const auto& g : groups) tiles += g[0].plan->args[0].ntiles * (long long)g.size();
  return tiles < kTogether * cfg.num_sms;
}

int block_set_build(const std::vector<std::vector<GroupMember>>& groups, bool together, int ring_len,
                    const LaunchCfg& cfg, cudaStream_t s, BlockSet** out, std::string* msg) {
  *out = nullptr;
  if (groups.empty() || (!together && groups.size() != 1)) return SV_EINVAL;
  BlockSet* set = new BlockSet();
  set->num_sms = cfg.num_sms;
  set->groups.resize(groups.size());
  int rc = SV_OK;
  size_t longest = 0;
  std::vector<ReduceItem> red;
  std::vector<TileSumItem> sums;
  for (size_t g = 0; g < groups.size() && rc == SV_OK; ++g) {
    BlockGroup& gr = set->groups[g];
    rc = group_build(groups[g], cfg.num_sms, together, s, &gr, msg);
    if (rc) break;
    const size_t S = std::max(1, gr.m[0].plan->nslots);
    longest = std::max(longest, gr.m[0].plan->seq_cyc.size());
    for (size_t c = 0; c < gr.m.size(); ++c) {
      ReduceItem it;
      it.partials = gr.d_part + 2 * (c * S * (size_t)gr.pairs);
      it.n = (long long)S * gr.pairs;
      it.ring = gr.m[c].ring;
      it.counter = gr.m[c].counter;
      it.L = gr.m[c].plan->L;
      it.ring_len = ring_len;
      red.push_back(it);
      for (size_t k = 0; k < S && together; ++k) {
        TileSumItem t;
        t.tiles = 1ll << gr.nt_log2;
        t.sums = gr.d_sums + (c * S + k) * (size_t)t.tiles * kGroupRows;
        t.pair = gr.d_part + 2 * (c * S + k);
        t.first = (long long)c * t.tiles;
        t.total = gr.ops[0].ntiles;
        t.ranges = group_ranges(t.total, cfg.num_sms);
        sums.push_back(t);
      }
    }
  }
  set->chains = (int)red.size();
  set->ntile_sums = (int)sums.size();
  for (size_t k = 0; k < longest && rc == SV_OK; ++k) {
    std::vector<long long> t;
    for (const BlockGroup& gr : set->groups)
      t.push_back(k < gr.m[0].plan->seq_cyc.size() ? gr.ops[0].ntiles : 0);
    set->share.push_back(together ? cta_shares(t, cfg.num_sms) : std::vector<int>(1, set->groups[0].pairs));
  }
  if (rc == SV_OK) {
    cudaError_t e = cudaMalloc(&set->d_reduce, sizeof(ReduceItem) * red.size());
    if (e == cudaSuccess && together) e = cudaMalloc(&set->d_tile_sums, sizeof(TileSumItem) * sums.size());
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(set->d_reduce, red.data(), sizeof(ReduceItem) * red.size(),
                          cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && together)
      e = cudaMemcpyAsync(set->d_tile_sums, sums.data(), sizeof(TileSumItem) * sums.size(),
                          cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // the host arrays are freed below
    if (e != cudaSuccess) {
      cudaGetLastError();
      *msg = "group upload";
      rc = SV_ECUDA;
    }
  }
  if (rc != SV_OK) {
    block_set_free(set);
    return rc;
  }
  *out = set;
  return SV_OK;
}

size_t block_set_size(const BlockSet* set) { return set->chains; }

cudaError_t block_set_enqueue(BlockSet* set, int periods, bool alone, cudaStream_t s) {
  if (periods <= 0) return cudaSuccess;
  cudaError_t e = set_sequence(
      set, [](const BlockPlan* p) -> const std::vector<int>& { return p->seq_entry; }, alone, s);
  for (int k = 0; k < periods && e == cudaSuccess; ++k) {
    const bool last = k + 1 == periods;
    std::vector<int> op(set->groups.size(), 0);
    for (size_t j = 0; j < set->share.size() && e == cudaSuccess; ++j) {
      for (size_t g = 0; g < set->groups.size(); ++g) {
        const BlockPlan* p = set->groups[g].m[0].plan;
        if (j < p->seq_cyc.size()) op[g] = (last ? p->seq_exit : p->seq_cyc)[j];
      }
      e = set_pass(set, op, set->share[j], alone, s);
    }
    if (e == cudaSuccess && set->ntile_sums) {
      void* args[] = {&set->d_tile_sums};
      e = launch_overlapped(reinterpret_cast<const void*>(k_tile_sums), set->ntile_sums, kTileSumThreads,
                            0, s, args, alone);
    }
    if (e == cudaSuccess) e = launch_period_reduce_many(set->d_reduce, set->chains, alone, s);
  }
  // the relabel steps behind the last period's passes
  if (e == cudaSuccess) {
    std::map<const BlockPlan*, std::vector<int>> rest;
    for (const BlockGroup& gr : set->groups) {
      const BlockPlan* p = gr.m[0].plan;
      rest[p].assign(p->seq_exit.begin() + std::min(p->seq_cyc.size(), p->seq_exit.size()),
                     p->seq_exit.end());
    }
    e = set_sequence(
        set, [&](const BlockPlan* p) -> const std::vector<int>& { return rest[p]; }, alone, s);
  }
  return e;
}

void block_set_free(BlockSet* set) {
  if (!set) return;
  for (BlockGroup& g : set->groups) {
    cudaFree(g.d_chains);
    cudaFree(g.d_part);
    cudaFree(g.d_sums);
  }
  cudaFree(set->d_reduce);
  cudaFree(set->d_tile_sums);
  delete set;
}

void block_free(BlockPlan* bp) {
  if (!bp) return;
  cudaFree(bp->d_U);
  cudaFree(bp->d_Ulead);
  cudaFree(bp->d_W);
  cudaFree(bp->d_partials);
  cudaFree(bp->d_status);
  delete bp;
}

}  // namespace fsv
