// Plain form in tiles: consecutive two-qubit gates of the period (Eq. 2 of
// arXiv 2111.08044, one 4x4 complex matvec per group of four amplitudes)
// applied to a tile of the state before it is written back, in the period's
// own order.  Each complex64 or complex128 amplitude sees the operations of one
// pass per gate, in the same order and with the same rounding, so the state is
// the same bit for bit; what changes is how often it travels.
//
// Why: one gate is 32 FP32 FMA an amplitude (table and residual) against 16
// bytes of traffic, so a pass of one gate is bound by HBM, and on a short
// chain by its launch and the latency of its loads (2.85 us a gate at L = 12,
// 0.55 us of it the launch).  With four to six gates a pass the FP32 pipe is
// the bound.  A pass of four gates at L = 27 takes 588 us (467 us of FMAs at
// the pipe's 36.8 TFMA/s), where four passes of one gate take 1350 us; a period
// 17.9 ms (104 gates), before 35.2 ms, at L = 20 0.18 ms for 0.39 ms, at L = 12
// 47 us for 128 us.
//
// complex64 (k_tile_f32): a thread holds 16 amplitudes (four register bits
// of the tile) and applies two gates on disjoint sites before it hands them
// back to the tile in shared memory; the next tile loads (cp.async) while
// this one is computed, and the last round writes the state directly where
// its lanes cover whole line parts.
// complex128 and double-float (k_tile_wide): their arithmetic (16 FP64 FMA
// or about 216 FP32 operations an amplitude and gate) is the bound already at
// one gate a pass; tiles there cut the launches of short chains and spread a
// short chain over the SMs (one output amplitude a thread in FP64, whose
// units take 16 cycles a warp instruction): complex128 at L = 13 0.11 ms a
// period, before 0.53 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <type_traits>

#include "sv_device.cuh"
#include "sv_internal.h"
#include "sv_kernels.h"
#include "sv_tile.cuh"

namespace fsv {

namespace {

using namespace dev;

__device__ __forceinline__ double period_scale(const Renorm& rn, long long c) {
  if (!rn.ring || rn.every <= 0) return 1.0;
  if (c <= 0 || c % rn.every != 0) return 1.0;
  const double n2 = *reinterpret_cast<const volatile double*>(rn.ring + 2 * ((c - 1) % rn.ring_len) + 1);
  return n2 > 0.0 ? 1.0 / sqrt(n2) : 1.0;
}

// Energy terms of one group of four amplitudes w[r] (r = 2 b_i + b_{i+1}), as
// the per-gate kernels form them: fixed products first, then one chain of
// sums per grouping.
template <typename R>
struct GroupTerms {
  R hi, lo, p[4], d[4];
};
template <typename R>
__device__ __forceinline__ void group_terms(const typename CT<R>::C (&w)[4], int epi,
                                            const Diag<R>& dg, uint64_t x,
                                            const uint64_t (&off)[4], GroupTerms<R>& t) {
  if (epi & EPI_X_HI) t.hi = cdotre(w[0], w[2]) + cdotre(w[1], w[3]);
  if (epi & EPI_X_LO) t.lo = cdotre(w[0], w[1]) + cdotre(w[2], w[3]);
  if (epi & EPI_DIAG) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      t.p[r] = cabs2(w[r]);
      t.d[r] = dg(x + off[r]);
    }
  }
}
// es + c t in one rounding (complex64: as the per-gate kernels add it)
template <typename R>
__device__ __forceinline__ R add_term(R es, R c, R t) {
  return es + c * t;
}
template <>
__device__ __forceinline__ float add_term<float>(float es, float c, float t) {
  return __fmaf_rn(c, t, es);
}
template <typename R>
__device__ __forceinline__ void group_chain(const GroupTerms<R>& t, int epi, R cxh, R cxl, R& es,
                                            R& ns) {
  if (epi & EPI_X_HI) es = add_term<R>(es, cxh * (R)2, t.hi);
  if (epi & EPI_X_LO) es = add_term<R>(es, cxl * (R)2, t.lo);
  if (epi & EPI_DIAG) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      ns += t.p[r];
      es += t.p[r] * t.d[r];
    }
  }
}

// ------------------------------------------------------------- complex64
// The gate on register bits (J0: site b, J1: site b + 1) of a thread's 16
// amplitudes; K0, K1 are the other two register bits.  get(e): entry e of the
// table (16, then 16 of its residual).  Residual products first (see
// k_plain.cu).  Packed FMAs on (re, im) pairs, each half the scalar chain: with
// the entries in the constant bank they run at the FP32 pipe's full rate (37.7
// TFMA/s in registers; scalar FMAs with the same operands 35.0, with entries
// loaded from shared memory 33) and leave half the issue slots to the loads,
// stores and addresses.  Each entry serves the four groups in turn.
template <int J0, int J1, int K0, int K1, bool kXor, typename G>
__device__ __forceinline__ void gate16(uint64_t (&v)[16], const G& get) {
  auto idx = [](int r, int k) {
    return ((r >> 1) << J0) | ((r & 1) << J1) | ((k & 1) << K0) | ((k >> 1) << K1);
  };
  uint64_t s[16], w[4][4];
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    const float2 t = un2(v[m]);
    s[m] = pk2(t.y, t.x);
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
#pragma unroll
    for (int k = 0; k < 4; ++k) w[r][k] = 0;
#pragma unroll
    for (int part = 1; part >= 0; --part) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = kXor ? r ^ j : j;
        const ulonglong2 g = get(16 * part + 4 * r + c);
#pragma unroll
        for (int k = 0; k < 4; ++k) w[r][k] = fma2(g.x, v[idx(c, k)], w[r][k]);
#pragma unroll
        for (int k = 0; k < 4; ++k) w[r][k] = fma2(g.y, s[idx(c, k)], w[r][k]);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int k = 0; k < 4; ++k) v[idx(r, k)] = w[r][k];
}

template <int J0, int J1, int K0, int K1>
__device__ __forceinline__ void measure16(const uint64_t (&v)[16], const TileArgs& ta,
                                          const TileRound& rd, int which, uint64_t x0,
                                          bool active, FloatSum& esum, FloatSum& nsum) {
  const int epi = rd.epi[which], bond = rd.bond[which];
  const float cxh = (float)ta.cx[bond], cxl = (float)ta.cx[bond + 1];
  Diag<float> dg;
  if (epi & EPI_DIAG) dg.init(ta.ep, ta.L);
  const uint64_t ro[4] = {1ull << rd.sbit[0], 1ull << rd.sbit[1], 1ull << rd.sbit[2],
                          1ull << rd.sbit[3]};
  const uint64_t off[4] = {0, ro[J1], ro[J0], ro[J0] + ro[J1]};
  const bool odd = threadIdx.x & 1;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float2 w[4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
      w[r] = un2(v[((r >> 1) << J0) | ((r & 1) << J1) | ((k & 1) << K0) | ((k >> 1) << K1)]);
    const uint64_t x = x0 + ((k & 1) ? ro[K0] : 0) + ((k >> 1) ? ro[K1] : 0);
    GroupTerms<float> t;
    group_terms<float>(w, epi, dg, x, off, t);
    float es = 0.f, ns = 0.f;
    group_chain<float>(t, epi, cxh, cxl, es, ns);
    bool take = active;
    if (rd.egroup[which] == TILE_E_PAIR) {
      // the neighbour's sum (bit 0 clear) continues in the lane with bit 0 set
      float e2 = __shfl_xor_sync(0xffffffffu, es, 1), n2 = 0.f;
      if (epi & EPI_DIAG) n2 = __shfl_xor_sync(0xffffffffu, ns, 1);
      group_chain<float>(t, epi, cxh, cxl, e2, n2);
      es = e2;
      ns = n2;
      take = active && odd;
    }
    if (take) {
      esum.add(es);
      if (epi & EPI_DIAG) nsum.add(ns);
    }
  }
}

// A measured gate on bonds 0..5 of a chain of at least 8 sites, from the tile:
// the sums of the per-gate kernel, whose threads hold bits 0, 6 and 7.
__device__ __noinline__ void measure_sweep(const uint8_t* tile, const TileArgs& ta, int bond, int epi,
                                           uint64_t tbase, FloatSum& esum, FloatSum& nsum) {
  const float cxh = (float)ta.cx[bond], cxl = (float)ta.cx[bond + 1];
  Diag<float> dg;
  if (epi & EPI_DIAG) dg.init(ta.ep, ta.L);
  const uint32_t nv = 1u << (ta.tb - 3);
  auto at = [&](uint32_t e) { return *reinterpret_cast<const float2*>(tile + tile_byte8(e)); };
  for (uint32_t vt = threadIdx.x; vt < nv; vt += blockDim.x) {
    const uint32_t e0 = ((vt & 31u) << 1) | ((vt >> 5) << 8);
    float2 w[4][2];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int k = 0; k < 2; ++k) w[c][k] = at(e0 | (c << 6) | k);
    float es = 0.f, ns = 0.f;
    if (epi & EPI_X_HI) {
      float s = 0.f;
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int k = 0; k < 2; ++k)
          s += cdotre(w[c][k], at((e0 | (c << 6) | k) ^ (1u << bond)));
      es += cxh * s;
    }
    if (epi & EPI_X_LO) {
      float s = 0.f;
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int k = 0; k < 2; ++k)
          s += cdotre(w[c][k], at((e0 | (c << 6) | k) ^ (2u << bond)));
      es += cxl * s;
    }
    if (epi & EPI_DIAG) {
      const uint64_t x0 = tbase + elem_state(ta, e0);
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float pr = cabs2(w[c][k]);
          ns += pr;
          es += pr * dg(x0 + ((uint64_t)c << 6) + k);
        }
    }
    esum.add(es);
    if (epi & EPI_DIAG) nsum.add(ns);
  }
}

// sum of (e, n) over the block in thread 0 (fixed order)
__device__ __forceinline__ void block_sum_pair(double& e, double& n, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    e += __shfl_xor_sync(0xffffffffu, e, o);
    n += __shfl_xor_sync(0xffffffffu, n, o);
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (l == 0) {
    sh[2 * w] = e;
    sh[2 * w + 1] = n;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    e = 0.0;
    n = 0.0;
    for (int k = 0; k < nw; ++k) {
      e += sh[2 * k];
      n += sh[2 * k + 1];
    }
  }
}

// a period's energy density and norm into the ring (thread 0), as the period
// reduce writes them
__device__ __forceinline__ void ring_store(const TileArgs& ta, long long c, double e, double n) {
  const long long slot = c % ta.ring_len;
  ta.ring[2 * slot] = n > 0.0 ? e / (ta.L * n) : 0.0;
  ta.ring[2 * slot + 1] = n;
}

// gate tables of the pass into shared memory, the first gate of the period
// scaled by the folded renormalisation
template <typename R>
__device__ __forceinline__ void load_gates(const TileArgs& ta, typename CT<R>::C* gs, long long c,
                                           int entries) {
  using C = typename CT<R>::C;
  const C* gp = static_cast<const C*>(ta.gates) + (ta.stride ? c * ta.stride : 0);
  const R sc = (R)(ta.first ? period_scale(ta.ep.rn, c) : 1.0);
  for (int k = threadIdx.x; k < ta.ngates * entries; k += blockDim.x) {
    const int g = k / entries, j = k - g * entries;
    C v = gp[(size_t)g * kGateEntries + j];
    if (g == 0) {
      v.x *= sc;
      v.y *= sc;
    }
    gs[k] = v;
  }
}

// complex64 tables of per-period gates, as packed operands
__device__ __forceinline__ void load_packed(const TileArgs& ta, PackedEntry* gs, long long c) {
  const float2* gp = static_cast<const float2*>(ta.gates) + (ta.stride ? c * ta.stride : 0);
  const float sc = (float)(ta.first ? period_scale(ta.ep.rn, c) : 1.0);
  for (int k = threadIdx.x; k < ta.ngates * kGateEntries; k += blockDim.x) {
    float2 v = gp[k];
    if (k < kGateEntries) {
      v.x *= sc;
      v.y *= sc;
    }
    gs[k] = PackedEntry{{v.x, v.x}, {-v.y, v.y}};
  }
}

// kSlots > 0: tables and rounds in the parameters; 0: in device memory, copied
// to shared memory (per-period tables, and passes that scale the first gate).
// kXor, kEpi: the pass has gates in the order r ^ j / measured gates; passes
// without them run less code.
template <int kSlots, bool kXor, bool kEpi, int kThreads, int kMinBlocks>
__global__ void __launch_bounds__(kThreads, kMinBlocks)
    k_tile_f32(float2* __restrict__ psi, const __grid_constant__ TileArgs ta,
               const __grid_constant__ TileTab<kSlots ? kSlots : 1> tab) {
  extern __shared__ __align__(16) uint8_t tile_smem[];
  __shared__ double red[2 * 16];
  const uint32_t tile_bytes = tile_byte8(1u << ta.tb);
  PackedEntry* gs = reinterpret_cast<PackedEntry*>(tile_smem + (size_t)ta.buffers * tile_bytes);
  TileRound* rds = reinterpret_cast<TileRound*>(gs + (size_t)ta.ngates * kGateEntries);
  const uint32_t sbuf = (uint32_t)__cvta_generic_to_shared(tile_smem);
  const int tbits = ta.tb - 4;
  const uint32_t tid = threadIdx.x & ((1u << tbits) - 1);
  const bool active = threadIdx.x < (1u << tbits);
  const uint32_t ntiles = 1u << (ta.L - ta.tb);
  const TileIo io = tile_io(ta);
  const TileRound& last = kSlots ? tab.r[ta.nrounds - 1] : ta.rounds[ta.nrounds - 1];
  const uint64_t xout = elem_state(ta, thread_elem<4>(last, tid));
  load_tile(ta, io, sbuf, psi + tile_base(ta, blockIdx.x));
  if (kSlots == 0)
    for (int k = threadIdx.x; k < 2 * ta.nrounds; k += blockDim.x)
      reinterpret_cast<uint4*>(rds)[k] = reinterpret_cast<const uint4*>(ta.rounds)[k];
  const bool reload = kSlots == 0 && (ta.stride != 0 || (ta.first && ta.ep.rn.ring));
  const long long c0 = reload || ta.periods > 0 ? *ta.counter : 0;
  const int periods = ta.periods > 0 ? ta.periods : 1;
  double eacc = 0.0, nacc = 0.0;
  FloatSum esum, nsum;
  for (int p = 0; p < periods; ++p) {
    if (kSlots == 0 && (p == 0 || reload)) load_packed(ta, gs, c0 + p);
    int cur = 0;
    for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
      const uint64_t tbase = tile_base(ta, t);
      uint8_t* tile = tile_smem + (size_t)cur * tile_bytes;
      if (ta.buffers == 2 && t + gridDim.x < ntiles) {
        load_tile(ta, io, sbuf + (cur ^ 1) * tile_bytes, psi + tile_base(ta, t + gridDim.x));
        cp_wait<1>();
      } else {
        cp_wait<0>();
      }
      __syncthreads();
      for (int r = 0; r < ta.nrounds; ++r) {
        const TileRound& rd = kSlots ? tab.r[r] : rds[r];
        const uint32_t e0 = thread_elem<4>(rd, tid);
        uint8_t* const at = tile + tile_byte8(e0);
        uint64_t v[16];
        const uint32_t sl0 = rd.slot[0], sl1 = rd.slot[1], sl2 = rd.slot[2], sl3 = rd.slot[3];
#pragma unroll
        for (int m = 0; m < 16; ++m)
          v[m] = *reinterpret_cast<const uint64_t*>(
              at + (((m & 1) ? sl0 : 0) + ((m & 2) ? sl1 : 0) + ((m & 4) ? sl2 : 0) + ((m & 8) ? sl3 : 0)));
        const int ga = rd.gate[0], gb = rd.gate[1];
        auto from = [&](int g) {
          return [&, g](int e) {
            return *reinterpret_cast<const ulonglong2*>(kSlots ? &tab.g[g][e]
                                                               : &gs[g * kGateEntries + e]);
          };
        };
        if (kXor && rd.xorder[0]) gate16<0, 1, 2, 3, true>(v, from(ga));
        else gate16<0, 1, 2, 3, false>(v, from(ga));
        if (kEpi && rd.epi[0] && rd.egroup[0] != TILE_E_SWEEP)
          measure16<0, 1, 2, 3>(v, ta, rd, 0, tbase + elem_state(ta, e0), active, esum, nsum);
        if (gb >= 0) {
          if (kXor && rd.xorder[1]) gate16<2, 3, 0, 1, true>(v, from(gb));
          else gate16<2, 3, 0, 1, false>(v, from(gb));
          if (kEpi && rd.epi[1] && rd.egroup[1] != TILE_E_SWEEP)
            measure16<2, 3, 0, 1>(v, ta, rd, 1, tbase + elem_state(ta, e0), active, esum, nsum);
        }
        if (active) {
          if (r == ta.nrounds - 1 && ta.direct_out && p == periods - 1) {
            uint64_t* out = reinterpret_cast<uint64_t*>(psi + tbase + xout);
            const uint64_t ro[4] = {1ull << rd.sbit[0], 1ull << rd.sbit[1], 1ull << rd.sbit[2],
                                    1ull << rd.sbit[3]};
#pragma unroll
            for (int m = 0; m < 16; ++m)
              out[((m & 1) ? ro[0] : 0) + ((m & 2) ? ro[1] : 0) + ((m & 4) ? ro[2] : 0) +
                  ((m & 8) ? ro[3] : 0)] = v[m];
          } else {
#pragma unroll
            for (int m = 0; m < 16; ++m)
              *reinterpret_cast<uint64_t*>(at + (((m & 1) ? sl0 : 0) + ((m & 2) ? sl1 : 0) +
                                               ((m & 4) ? sl2 : 0) + ((m & 8) ? sl3 : 0))) = v[m];
          }
        }
        // between rounds, and before the buffer takes another tile
        __syncthreads();
        if (kEpi) {
          const int sw = rd.egroup[1] == TILE_E_SWEEP ? 1 : rd.egroup[0] == TILE_E_SWEEP ? 0 : -1;
          if (sw >= 0) {
            measure_sweep(tile, ta, rd.bond[sw], rd.epi[sw], tbase, esum, nsum);
            __syncthreads();
          }
        }
      }
      if (kEpi && ta.any_epi) {
        esum.flush(eacc);
        nsum.flush(nacc);
      }
      if (!ta.direct_out && p == periods - 1) {
        store_tile(ta, io, tile, psi + tbase);
        __syncthreads();
      }
      if (ta.buffers == 2) cur ^= 1;
      else if (t + gridDim.x < ntiles) {
        load_tile(ta, io, sbuf, psi + tile_base(ta, t + gridDim.x));
      }
    }
    if (ta.periods > 0) {
      block_sum_pair(eacc, nacc, red);
      if (threadIdx.x == 0) ring_store(ta, c0 + p, eacc, nacc);
      eacc = 0.0;
      nacc = 0.0;
      __syncthreads();
    }
  }
  if (ta.periods > 0) {
    if (threadIdx.x == 0) *ta.counter_rw = c0 + periods;
  } else if (kEpi && ta.ep.partial) {
    block_store_pair(eacc, nacc, ta.ep.partial);
  }
}

// --------------------------------------------- complex128 and double-float
// Double-float: a thread takes a group of four amplitudes, in place.
// complex128: a thread takes one output amplitude, between two copies of the
// tile (the FP64 units are busy for 16 cycles a warp instruction, so the
// extra shared-memory reads cost nothing and every lane has work).
template <typename R, int kThreads, int kMinBlocks>
__global__ void __launch_bounds__(kThreads, kMinBlocks)
    k_tile_wide(typename CT<R>::C* __restrict__ psi, const __grid_constant__ TileArgs ta) {
  using C = typename CT<R>::C;
  constexpr bool kRows = std::is_same<R, double>::value;
  constexpr int kEntries = 16;
  extern __shared__ __align__(16) uint8_t tile_smem[];
  __shared__ double red[2 * 16];
  const uint32_t N = 1u << ta.tb;
  C* tile = reinterpret_cast<C*>(tile_smem);
  C* other = tile + N;  // complex128: the other copy; double-float: the next tile
  C* gs = ta.buffers == 2 ? other + N : other;
  TileRound* rds = reinterpret_cast<TileRound*>(gs + (size_t)ta.ngates * kEntries);
  const uint32_t groups = N >> 2;
  const uint32_t tid = threadIdx.x & (groups - 1);
  const bool active = threadIdx.x < groups;
  const uint32_t ntiles = 1u << (ta.L - ta.tb);
  auto load = [&](C* to, uint32_t t) {
    const C* from = psi + tile_base(ta, t);
    for (uint32_t e = threadIdx.x; e < N; e += blockDim.x)
      cp_async16((uint32_t)__cvta_generic_to_shared(to + tile_slot16(e)), from + elem_state(ta, e));
    cp_commit();
  };
  load(tile, blockIdx.x);
  for (int k = threadIdx.x; k < 2 * ta.nrounds; k += blockDim.x)
    reinterpret_cast<uint4*>(rds)[k] = reinterpret_cast<const uint4*>(ta.rounds)[k];
  const bool reload = ta.stride != 0 || (ta.first && ta.ep.rn.ring);
  const long long c0 = reload || ta.periods > 0 ? *ta.counter : 0;
  const int periods = ta.periods > 0 ? ta.periods : 1;
  double eacc = 0.0, nacc = 0.0;
  for (int p = 0; p < periods; ++p) {
    if (p == 0 || reload) load_gates<R>(ta, gs, c0 + p, kEntries);
    for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
      const uint64_t tbase = tile_base(ta, t);
      const bool more = t + gridDim.x < ntiles;
      if (!kRows && ta.buffers == 2 && more) {
        load(other, t + gridDim.x);
        cp_wait<1>();
      } else {
        cp_wait<0>();
      }
      __syncthreads();
      for (int r = 0; r < ta.nrounds; ++r) {
        const TileRound rd = rds[r];
        const C* g = gs + rd.gate[0] * kEntries;
        const uint32_t e0 = thread_elem<2>(rd, tid);
        const uint32_t s0 = tile_slot16(e0);
        const uint32_t sh = rd.slot[0], sl = rd.slot[1];
        const uint64_t xh = 1ull << rd.sbit[0], xl = 1ull << rd.sbit[1];
        C w[4];
        if (kRows) {
          if (threadIdx.x < N) {
            const uint32_t e = threadIdx.x, ml = rd.ins[0] & (0u - rd.ins[0]);
            const uint32_t mh = ml << 1;  // sites b, b + 1: adjacent tile bits
            const int row = ((e & ml) ? 2 : 0) | ((e & mh) ? 1 : 0);
            const uint32_t b = tile_slot16(e & ~(mh | ml));
            C acc = czero<C>();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int c = rd.xorder[0] ? row ^ j : j;
              acc = cmac(acc, g[4 * row + c], tile[b ^ ((c & 2) ? sh : 0) ^ ((c & 1) ? sl : 0)]);
            }
            other[tile_slot16(e)] = acc;
          }
          __syncthreads();
          C* const swap = tile;
          tile = other;
          other = swap;
          if (rd.epi[0]) {
#pragma unroll
            for (int m = 0; m < 4; ++m) w[m] = tile[s0 ^ ((m & 2) ? sh : 0) ^ ((m & 1) ? sl : 0)];
          }
        } else {
          C v[4];
#pragma unroll
          for (int m = 0; m < 4; ++m) v[m] = tile[s0 ^ ((m & 2) ? sh : 0) ^ ((m & 1) ? sl : 0)];
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            C acc = czero<C>();
#pragma unroll
            for (int c = 0; c < 4; ++c) acc = cmac(acc, g[4 * m + c], v[c]);
            w[m] = acc;
          }
          if (active) {
            if (r == ta.nrounds - 1 && ta.direct_out && p == periods - 1) {
              C* out = psi + tbase + elem_state(ta, e0);
#pragma unroll
              for (int m = 0; m < 4; ++m) out[((m & 2) ? xh : 0) + ((m & 1) ? xl : 0)] = w[m];
            } else {
#pragma unroll
              for (int m = 0; m < 4; ++m) tile[s0 ^ ((m & 2) ? sh : 0) ^ ((m & 1) ? sl : 0)] = w[m];
            }
          }
          __syncthreads();
        }
        if (rd.epi[0] && active) {
          const R cxh = (R)ta.cx[rd.bond[0]], cxl = (R)ta.cx[rd.bond[0] + 1];
          Diag<R> dg;
          if (rd.epi[0] & EPI_DIAG) dg.init(ta.ep, ta.L);
          const uint64_t off[4] = {0, xl, xh, xh + xl};
          GroupTerms<R> gt;
          group_terms<R>(w, rd.epi[0], dg, tbase + elem_state(ta, e0), off, gt);
          R es = 0, ns = 0;
          group_chain<R>(gt, rd.epi[0], cxh, cxl, es, ns);
          eacc += (double)es;
          nacc += (double)ns;
        }
      }
      if (!ta.direct_out && p == periods - 1) {
        C* out = psi + tbase;
        for (uint32_t e = threadIdx.x; e < N; e += blockDim.x)
          out[elem_state(ta, e)] = tile[tile_slot16(e)];
        __syncthreads();
      }
      if (!kRows && ta.buffers == 2) {
        C* const swap = tile;
        tile = other;
        other = swap;
      } else if (more) {
        load(tile, t + gridDim.x);
      }
    }
    if (ta.periods > 0) {
      block_sum_pair(eacc, nacc, red);
      if (threadIdx.x == 0) ring_store(ta, c0 + p, eacc, nacc);
      eacc = 0.0;
      nacc = 0.0;
      __syncthreads();
    }
  }
  if (ta.periods > 0) {
    if (threadIdx.x == 0) *ta.counter_rw = c0 + periods;
  } else if (ta.ep.partial) {
    block_store_pair(eacc, nacc, ta.ep.partial);
  }
}

size_t tile_smem_bytes(int precision, const TileArgs& ta) {
  size_t b = (precision == SV_C64 ? (size_t)tile_byte8(1u << ta.tb) : (size_t)16 << ta.tb) * ta.buffers;
  if (!ta.in_params)
    b += (size_t)ta.ngates * (precision == SV_C64 ? 512 : 256) + (size_t)ta.nrounds * sizeof(TileRound);
  return b;
}

template <int kSlots>
const void* f32_kernel(const TileArgs& ta) {
  if (ta.tb > 12) return reinterpret_cast<const void*>(k_tile_f32<kSlots, true, true, 512, 1>);
  // a whole chain in one block, or tables in shared memory: the general form
  if (kSlots != kTileTabSmall)
    return reinterpret_cast<const void*>(k_tile_f32<kSlots, true, true, 256, 2>);
  if (ta.any_epi) return reinterpret_cast<const void*>(k_tile_f32<kTileTabSmall, true, true, 256, 2>);
  return ta.any_xorder ? reinterpret_cast<const void*>(k_tile_f32<kTileTabSmall, true, false, 256, 3>)
                       : reinterpret_cast<const void*>(k_tile_f32<kTileTabSmall, false, false, 256, 3>);
}

bool small_tab(const TileArgs& ta) { return ta.ngates <= kTileTabSmall && ta.nrounds <= kTileTabSmall; }

const void* tile_kernel(int precision, const TileArgs& ta) {
  if (precision == SV_DF64) return reinterpret_cast<const void*>(k_tile_wide<df, 256, 2>);
  if (precision == SV_C128) return reinterpret_cast<const void*>(k_tile_wide<double, 512, 2>);
  if (!ta.in_params) return f32_kernel<0>(ta);
  return small_tab(ta) ? f32_kernel<kTileTabSmall>(ta) : f32_kernel<kTileMaxGates>(ta);
}

}  // namespace

cudaError_t tile_grid(int precision, TileArgs* ta, const LaunchCfg& cfg, int* grid) {
  const uint64_t tiles = 1ull << (ta->L - ta->tb);
  const void* kernel = tile_kernel(precision, *ta);
  // every pass of an instance asks for the same limit (its largest)
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (precision == SV_C64 ? 104 : 64) * 1024);
  // complex128 works between two copies; elsewhere a second buffer takes the
  // next tile while this one is computed
  int per_sm = 1;
  for (int buffers = precision == SV_C128 ? 2 : 1; buffers <= 2 && e == cudaSuccess; ++buffers) {
    ta->buffers = buffers;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, tile_threads(precision, ta->tb),
                                                      tile_smem_bytes(precision, *ta));
    per_sm = std::max(1, std::min(per_sm, 4));  // the partial sums hold four blocks an SM
    if (tiles <= (uint64_t)cfg.num_sms * per_sm) break;  // one tile a block: nothing to prefetch
  }
  *grid = (int)std::min<uint64_t>(tiles, (uint64_t)cfg.num_sms * per_sm);
  return e;
}

cudaError_t launch_tile(int precision, void* psi, const TileArgs& ta,
                        const TileTab<kTileMaxGates>* tab, int grid, cudaStream_t s) {
  const int threads = tile_threads(precision, ta.tb);
  const size_t smem = tile_smem_bytes(precision, ta);
  const void* kernel = tile_kernel(precision, ta);
  TileTab<kTileTabSmall> small;
  TileTab<1> none;
  void* args[] = {&psi, const_cast<TileArgs*>(&ta), nullptr};
  if (precision == SV_C64 && !ta.in_params) {
    args[2] = &none;
  } else if (precision == SV_C64 && small_tab(ta)) {
    std::memcpy(small.g, tab->g, sizeof(small.g));
    std::memcpy(small.r, tab->r, sizeof(small.r));
    args[2] = &small;
  } else if (precision == SV_C64) {
    args[2] = const_cast<TileTab<kTileMaxGates>*>(tab);
  }
  return cudaLaunchKernel(kernel, dim3(grid), dim3(threads), args, smem, s);
}

}  // namespace fsv
