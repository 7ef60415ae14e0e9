// A chain held in the shared memory of one block, or of a cluster of blocks,
// for a run of periods: every gate of every period (Eq. 2), the energy density
// and norm of each, and one read and one write of the state per run.  Used for
// single short chains in the plain form and for batches of chains.
//
// A block of a cluster of 2^k holds the amplitudes whose k rank bits (k sites of
// the chain) are its rank.  Rounds of two gates on 16 amplitudes a thread as in
// k_tile.cu, in the period's order, with the same arithmetic; a round on one of
// those sites reads and writes the other blocks' shared memory, between cluster
// barriers, the others stay within the block.  The gate tables (up to 96 gates at
// a time) and the rounds are in shared memory.
//
// What bounds it: a chain of 13 sites is 16 warps of work, so the length of one
// warp's round (about 980 instructions, 1 us with a warp a scheduler) and the
// barrier after it, not the FP32 pipe.  Hence the spread over blocks down to four
// warps each, and no further: the rank's bits make more rounds remote, and a
// cluster barrier is most of a remote round's wait.  One gate on four amplitudes a
// thread would shorten the round but loads twice as often and takes twice the
// barriers: 64 batch chains of 9..13 sites 2.02 ms for 32 periods, here 1.48 ms.
//
// Plain form: a period of 44 gates at L = 12 42 us (47 us in one 12-bit tile of
// four warps a scheduler, 128 us in a launch a gate).  Batches: 32 periods of the
// 64 chains 1.48 ms, before (one gate and 512 threads a block, one block a chain)
// 3.72 ms; 160 chains of 12..14 sites, 48 periods, 9.1 ms for 13.4 ms.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "sv_batch.h"
#include "sv_tile.cuh"

namespace fsv {

namespace {

using namespace dev;
namespace cg = cooperative_groups;

constexpr int kMaxThreads = 256;
constexpr int kMaxWarps = kMaxThreads / 32;
static_assert(kShortMaxL == 10, "batch chains here have at least 11 sites");
constexpr int kMaxDynamic = 224 * 1024;  // of 227 KiB a block, beside the static arrays

__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ uint64_t peer_load(uint32_t addr) {
  uint64_t v;
  asm volatile("ld.shared::cluster.b64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void peer_store(uint32_t addr, uint64_t v) {
  asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}

// Which block holds a state index, and where in its part.
struct Spread {
  int pos, kbits;
  __device__ __forceinline__ uint32_t rank(uint32_t e) const { return (e >> pos) & ((1u << kbits) - 1); }
  __device__ __forceinline__ uint32_t part(uint32_t e) const {
    return (e & ((1u << pos) - 1)) | ((e >> (pos + kbits)) << pos);
  }
  __device__ __forceinline__ uint32_t state(uint32_t l, uint32_t r) const {
    return (l & ((1u << pos) - 1)) | (r << pos) | ((l >> pos) << (pos + kbits));
  }
};

// <H0> and the norm of a period's final state (batch chains): the sums over the
// amplitudes that agree in sites 0..8, in ascending order, compensated (Kahan)
// in FP32; each amplitude's diagonal energy in site order, then its <X> terms in
// site order (each pair at the amplitude with the bit clear).
// kNa: sites summed over in registers (the lowest four of them).
template <int kNa>
__device__ __forceinline__ void measure_final(const ChainArgs& ch, const uint8_t* tile, uint32_t sbuf,
                                              const Spread& sp, uint32_t rank, double& e, double& n) {
  constexpr int low = 9;                      // sites that tell sums apart
  const int L = ch.L;
  const int lt = low - sp.kbits;              // of them in the block's part (rank: pos .. 8)
  const int nk = L - low;                     // sites summed over
  constexpr int kM = 1 << kNa;
  const float J = ch.Jf;
  auto at = [&](uint32_t l) { return *reinterpret_cast<const float2*>(tile + tile_byte8(l)); };
  for (uint32_t s = threadIdx.x; s < (1u << lt); s += blockDim.x) {
    const uint32_t x = sp.state(s, rank);  // sites 0..8
    float base = 0.f;
    for (int i = 0; i < low; ++i) {
      const float zi = ((x >> i) & 1) ? -1.f : 1.f;
      base += ch.cz[i] * zi;
      if (i + 1 < low) base += J * zi * (((x >> (i + 1)) & 1) ? -1.f : 1.f);
    }
    const bool last = (x >> (low - 1)) & 1;
    float czr[kNa + 1], cxr[kNa + 1];
#pragma unroll
    for (int j = 0; j < kNa; ++j) {
      czr[j] = ch.cz[low + j];
      cxr[j] = 2.f * ch.cx[low + j];
    }
    float es = 0.f, ec = 0.f, ns = 0.f, nc = 0.f;
    for (uint32_t top = 0; top < (1u << (nk - kNa)); ++top) {
      const uint32_t l0 = s | (top << (lt + kNa));
      float2 v[kM];
      float ex[kM];
#pragma unroll
      for (int m = 0; m < kM; ++m)
        {
          v[m] = at(l0 | ((uint32_t)m << lt));
          ex[m] = 0.f;
        }
      for (int i = 0; i < lt; ++i) {  // (the rank's sites are the highest of the low ones)
        if ((s >> i) & 1) continue;
        const float c = 2.f * ch.cx[i];
#pragma unroll
        for (int m = 0; m < kM; ++m)
          ex[m] = __fmaf_rn(c, cdotre(v[m], at((l0 | (1u << i)) | ((uint32_t)m << lt))), ex[m]);
      }
      for (int i = 0; i < sp.kbits; ++i) {
        if ((rank >> i) & 1) continue;
        const float c = 2.f * ch.cx[sp.pos + i];
        const uint32_t peer = peer_addr(sbuf, rank | (1u << i));
        float2 u[kM];
#pragma unroll
        for (int m = 0; m < kM; ++m)
          u[m] = un2(peer_load(peer + tile_byte8(l0 | ((uint32_t)m << lt))));
#pragma unroll
        for (int m = 0; m < kM; ++m)
          ex[m] = __fmaf_rn(c, cdotre(v[m], u[m]), ex[m]);
      }
#pragma unroll
      for (int j = 0; j < kNa; ++j) {
#pragma unroll
          for (int m = 0; m < kM; ++m)
            if (!(m & (1 << j)))
              ex[m] = __fmaf_rn(cxr[j], cdotre(v[m], v[m | (1 << j)]), ex[m]);
        }
      for (int j = kNa; j < nk; ++j) {
        if ((top >> (j - kNa)) & 1) continue;
        const float c = 2.f * ch.cx[low + j];
#pragma unroll
        for (int m = 0; m < kM; ++m)
          ex[m] = __fmaf_rn(c, cdotre(v[m], at((l0 | (1u << (lt + j))) | ((uint32_t)m << lt))), ex[m]);
      }
#pragma unroll
      for (int m = 0; m < kM; ++m) {
          float d = base;
          bool b = last;  // the site before: its bit
#pragma unroll
          for (int j = 0; j < kNa; ++j) {
              const bool bj = (m >> j) & 1;
              d += b != bj ? -J : J;
              d += bj ? -czr[j] : czr[j];
              b = bj;
            }
          for (int j = kNa; j < nk; ++j) {
            const bool bj = (top >> (j - kNa)) & 1;
            d += b != bj ? -J : J;
            d += bj ? -ch.cz[low + j] : ch.cz[low + j];
            b = bj;
          }
          const float pr = cabs2(v[m]);
          const float ye = __fsub_rn(__fmaf_rn(pr, d, ex[m]), ec), te = __fadd_rn(es, ye);
          ec = __fsub_rn(__fsub_rn(te, es), ye);
          es = te;
          const float yn = __fsub_rn(pr, nc), tn = __fadd_rn(ns, yn);
          nc = __fsub_rn(__fsub_rn(tn, ns), yn);
          ns = tn;
        }
    }
    e += (double)es - (double)ec;
    n += (double)ns - (double)nc;
  }
}

template <bool kPlain, bool kRemote>
__device__ __forceinline__ void run_round(const ResidentRound& rd, const PackedEntry* ga,
                                          const ChainArgs& ch, uint8_t* tile, uint32_t sbuf,
                                          const Spread& sp, uint32_t rank, uint32_t at, bool active,
                                          FloatSum& esum, FloatSum& nsum) {
  // at: the thread's first amplitude, in the block's part or (remote) the state
  const uint32_t base = kRemote ? at : tile_byte8(at);
  const uint32_t e0 = kRemote ? at : sp.state(at, rank);
  const uint32_t o0 = rd.off[0], o1 = rd.off[1], o2 = rd.off[2], o3 = rd.off[3];
  auto place = [&](int m) {
    return base + (((m & 1) ? o0 : 0) + ((m & 2) ? o1 : 0) + ((m & 4) ? o2 : 0) + ((m & 8) ? o3 : 0));
  };
  uint64_t v[16];
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    const uint32_t a = place(m);
    v[m] = kRemote ? peer_load(peer_addr(sbuf + tile_byte8(sp.part(a)), sp.rank(a)))
                   : *reinterpret_cast<const uint64_t*>(tile + a);
  }
  auto from = [&](const PackedEntry* g) {
    return [g](int e) { return *reinterpret_cast<const ulonglong2*>(g + e); };
  };
  if (kPlain && rd.xorder[0]) gate16<0, 1, 2, 3, true>(v, from(ga));
  else gate16<0, 1, 2, 3, false>(v, from(ga));
  // <X> in pairs (of a measured gate most often) has its own, shorter code
  auto pairs = [&](int k) { return rd.egroup[k] == TILE_E_PAIR && !(rd.epi[k] & EPI_DIAG); };
  if (kPlain && rd.epi[0] && rd.sweep != 1) {
    if (pairs(0)) measure16_x<0, 1, 2, 3>(v, ch.cx, rd, 0, active, esum);
    else measure16<0, 1, 2, 3>(v, ch.L, ch.cx, ch.ep, rd, 0, e0, active, esum, nsum);
  }
  if (rd.count == 2) {
    const PackedEntry* gb = ga + kGateEntries;
    if (kPlain && rd.xorder[1]) gate16<2, 3, 0, 1, true>(v, from(gb));
    else gate16<2, 3, 0, 1, false>(v, from(gb));
    if (kPlain && rd.epi[1] && rd.sweep != 2) {
      if (pairs(1)) measure16_x<2, 3, 0, 1>(v, ch.cx, rd, 1, active, esum);
      else measure16<2, 3, 0, 1>(v, ch.L, ch.cx, ch.ep, rd, 1, e0, active, esum, nsum);
    }
  }
  if (active) {
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const uint32_t a = place(m);
      if (kRemote) peer_store(peer_addr(sbuf + tile_byte8(sp.part(a)), sp.rank(a)), v[m]);
      else *reinterpret_cast<uint64_t*>(tile + a) = v[m];
    }
  }
}

// kPlain: one chain, its energy terms measured by the rounds (the per-gate
// kernels' groupings); else a batch, measured on each period's final state.
template <bool kPlain>
__global__ void __launch_bounds__(kMaxThreads, 1)
    k_resident(const __grid_constant__ ChainArgs one, const ChainArgs* __restrict__ chains,
               const long long* __restrict__ counter, int periods, int ring_len, int kbits,
               int pos, uint32_t tab_at) {
  extern __shared__ __align__(16) uint8_t tile[];
  __shared__ __align__(16) uint8_t ch_raw[sizeof(ChainArgs)];
  const ChainArgs& ch = *reinterpret_cast<const ChainArgs*>(ch_raw);
  __shared__ double red[kMaxWarps][2];
  __shared__ double peers[16][2];  // rank 0: every block's sums
  cg::cluster_group cluster = cg::this_cluster();
  const uint32_t rank = kbits ? cluster.block_rank() : 0;
  const uint32_t tid = threadIdx.x, T = blockDim.x, lane = tid & 31;
  {
    const ChainArgs* src = kPlain ? &one : chains + (blockIdx.x >> kbits);
    for (uint32_t k = tid; k < sizeof(ChainArgs) / 4; k += T)
      reinterpret_cast<uint32_t*>(ch_raw)[k] = reinterpret_cast<const uint32_t*>(src)[k];
  }
  const long long c0 = counter[0];
  if (!kPlain && periods == 0) periods = (int)counter[1];
  __syncthreads();
  const int L = ch.L, lb = L - kbits;  // bits of a block's part
  const uint32_t per = 1u << (lb - 4);  // threads' worth of 16 amplitudes
  const uint32_t sbuf = (uint32_t)__cvta_generic_to_shared(tile);
  const int held = ch.ngates < kResidentGates ? ch.ngates : kResidentGates;
  PackedEntry* const tab = reinterpret_cast<PackedEntry*>(tile + tab_at);
  ResidentRound* const rds = reinterpret_cast<ResidentRound*>(tab + (size_t)held * kGateEntries);
  auto barrier = [&](bool wide) {
    if (kbits && wide) cluster.sync();
    else __syncthreads();
  };
  const Spread sp{pos, kbits};
  for (uint32_t q = 2 * tid; q < (1u << lb); q += 2 * T)  // (pos is 0 or at least 1)
    *reinterpret_cast<float4*>(tile + tile_byte8(q)) =
        *reinterpret_cast<const float4*>(ch.psi + sp.state(q, rank));
  // tables of the gates from g0 on, in period c (the period's first gate scaled
  // by a folded renormalisation), and the rounds from r0 on
  const bool scaled = kPlain && ch.ep.rn.ring;
  auto load_tables = [&](int g0, int r0, long long c) {
    const int n = ch.ngates - g0 < held ? ch.ngates - g0 : held;
    const float2* gp = ch.gates + (ch.stride ? c * ch.stride : 0) + (size_t)g0 * kGateEntries;
    const float sc = scaled && g0 == 0 ? (float)period_scale(ch.ep.rn, c) : 1.f;
    for (int k = tid; k < n * kGateEntries; k += T) {
      float2 v = __ldg(gp + k);
      if (k < kGateEntries) {
        v.x *= sc;
        v.y *= sc;
      }
      tab[k] = PackedEntry{{v.x, v.x}, {-v.y, v.y}};
    }
    const uint4* rp = reinterpret_cast<const uint4*>(ch.rounds + r0);
    const int nr = 3 * (ch.nrounds - r0 < held ? ch.nrounds - r0 : held);  // at most one a gate
    for (int k = tid; k < nr; k += T) reinterpret_cast<uint4*>(rds)[k] = __ldg(rp + k);
  };
  const bool reload = ch.ngates > held || ch.stride != 0 || scaled;
  if (!reload) load_tables(0, 0, c0);
  barrier(true);
  FloatSum esum, nsum;
  for (int p = 0; p < periods; ++p) {
    // first gate and round of those held; gates done of them
    int g0 = 0, r0 = 0, g = 0;
    for (int r = 0; r < ch.nrounds; ++r) {
      if (reload && (r == 0 || g == held)) {  // every thread alike, after a barrier
        g0 = r == 0 ? 0 : g0 + held;
        load_tables(g0, r, c0 + p);
        r0 = r;
        g = 0;
        __syncthreads();
      }
      const ResidentRound& rd = rds[r - r0];
      const PackedEntry* const gs = tab + (size_t)g * kGateEntries;
      const bool remote = rd.remote, wide = rd.cluster || r + 1 == ch.nrounds;
      for (uint32_t s0 = tid & ~31u; s0 < per; s0 += T) {  // warps without a share leave
        uint32_t at = (s0 + lane) & (per - 1);
        if (remote) at += rank * per;
#pragma unroll
        for (int k = 0; k < 4; ++k) at += at & rd.ins[k];
        if (!remote)
          run_round<kPlain, false>(rd, gs, ch, tile, sbuf, sp, rank, at, s0 + lane < per, esum, nsum);
        else
          run_round<kPlain, true>(rd, gs, ch, tile, sbuf, sp, rank, at, s0 + lane < per, esum, nsum);
      }
      g += rd.count;
      // read before the barrier: behind it, where the tables held are used up, a
      // faster warp writes the next ones over rd
      const int sweep = kPlain ? rd.sweep : 0;
      barrier(wide);
      if (sweep) {  // (rd stays until every warp has passed the barrier below)
        const int w = sweep - 1;
        measure_sweep(tile, lb, L, ch.cx, ch.ep, rd.bond[w], rd.epi[w],
                      [&](uint32_t l) { return (uint64_t)sp.state(l, rank); }, esum, nsum);
        barrier(wide);
      }
    }
    // the period's sums: over the block, then over the cluster in rank 0
    double e = 0.0, n = 0.0;
    if (!kPlain) {
      switch (L) {  // more than kShortMaxL sites
        case 11: measure_final<2>(ch, tile, sbuf, sp, rank, e, n); break;
        case 12: measure_final<3>(ch, tile, sbuf, sp, rank, e, n); break;
        default: measure_final<4>(ch, tile, sbuf, sp, rank, e, n);
      }
    } else {
      esum.flush(e);
      nsum.flush(n);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      e += __shfl_xor_sync(0xffffffffu, e, o);
      n += __shfl_xor_sync(0xffffffffu, n, o);
    }
    if (lane == 0) {
      red[tid >> 5][0] = e;
      red[tid >> 5][1] = n;
    }
    __syncthreads();
    if (tid == 0) {
      e = n = 0.0;
      for (uint32_t w = 0; w < T / 32; ++w) {
        e += red[w][0];
        n += red[w][1];
      }
      double* to = kbits ? cluster.map_shared_rank(&peers[rank][0], 0) : &peers[0][0];
      to[0] = e;
      to[1] = n;
    }
    barrier(true);
    if (rank == 0 && tid == 0) {
      e = n = 0.0;
      for (uint32_t w = 0; w < (1u << kbits); ++w) {
        e += peers[w][0];
        n += peers[w][1];
      }
      const long long slot = (c0 + p) % ring_len;
      double* const out = ch.ring + 2 * slot * ch.ring_stride;
      // plain: as the period reduce writes it; batch: as the shorter chains' (NaN where
      // the norm is NaN or zero)
      out[0] = !kPlain || n > 0.0 ? e / ((double)L * n) : 0.0;
      out[1] = n;
      if (scaled) __threadfence();
    }
    if (scaled) barrier(true);  // the next period's first table reads the norm
  }
  for (uint32_t q = 2 * tid; q < (1u << lb); q += 2 * T)
    *reinterpret_cast<float4*>(ch.psi + sp.state(q, rank)) =
        *reinterpret_cast<const float4*>(tile + tile_byte8(q));
  if (kPlain && rank == 0 && tid == 0) *ch.counter = c0 + periods;
}

__global__ void k_advance(long long* counter, int periods) {
  counter[0] += periods ? periods : counter[1];
}

// Launch of `nchains` clusters of a shape (at: storage of its attribute).
uint32_t tables_at(const ResidentShape& sh) { return tile_byte8(1u << (sh.L - sh.kbits)); }

cudaLaunchConfig_t launch_config(int nchains, const ResidentShape& sh, int ngates,
                                 cudaLaunchAttribute* at, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)nchains << sh.kbits);
  cfg.blockDim = dim3(sh.threads);
  const size_t held = std::min(ngates, kResidentGates);
  cfg.dynamicSmemBytes = tables_at(sh) + held * (kGateEntries * sizeof(PackedEntry) + sizeof(ResidentRound));
  cfg.stream = s;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = 1u << sh.kbits;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

}  // namespace

// Blocks of a chain: spread until 2^kWarpsKept warps are left in a block, at most
// `most` blocks (a power of two).  With eight warps left 12 sites take 55 us a
// period, with four 42 us, with two 45 us; 13 sites 69, 55 and 55 us.
ResidentShape resident_shape(bool plain, int L, int most) {
  constexpr int kWarpsKept = 2;  // log2
  ResidentShape sh;
  sh.L = L;
  const int warps = std::max(0, L - 9);  // log2, 16 amplitudes a thread
  const int top = plain ? 4 : 3;
  while (sh.kbits < top && (2 << sh.kbits) <= most && warps - (sh.kbits + 1) >= kWarpsKept) ++sh.kbits;
  // (at least four warps: the others load the tables)
  sh.threads = std::min(kMaxThreads, std::max(128, 32 << (warps - sh.kbits)));
  sh.pos = plain ? L - sh.kbits : std::min(L, 9) - sh.kbits;
  return sh;
}

cudaError_t resident_prepare(bool plain, const ResidentShape& sh, int ngates, int* clusters) {
  const void* f = plain ? reinterpret_cast<const void*>(k_resident<true>)
                        : reinterpret_cast<const void*>(k_resident<false>);
  cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kMaxDynamic);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess || !clusters) return e;
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t cfg = launch_config(1, sh, ngates, &at, nullptr);
  return cudaOccupancyMaxActiveClusters(clusters, f, &cfg);
}

cudaError_t launch_resident_chain(const ChainArgs& chain, const ResidentShape& sh, int periods,
                                  int ring_len, cudaStream_t s) {
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t cfg = launch_config(1, sh, chain.ngates, &at, s);
  return cudaLaunchKernelEx(&cfg, k_resident<true>, chain, (const ChainArgs*)nullptr,
                            (const long long*)chain.counter, periods, ring_len, sh.kbits,
                            sh.pos, tables_at(sh));
}

cudaError_t launch_resident_batch(const ChainArgs* chains, int nchains, const ResidentShape& sh,
                                  int ngates, const long long* counter, int periods, int ring_len,
                                  cudaStream_t s) {
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t cfg = launch_config(nchains, sh, ngates, &at, s);
  return cudaLaunchKernelEx(&cfg, k_resident<false>, ChainArgs(), chains, counter, periods, ring_len,
                            sh.kbits, sh.pos, tables_at(sh));
}

cudaError_t launch_advance(long long* counter, int periods, cudaStream_t s) {
  k_advance<<<1, 1, 0, s>>>(counter, periods);
  return cudaGetLastError();
}

}  // namespace fsv
