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
// the bound.  A pass of four gates at L = 27 takes 580 us (467 us of FMAs at
// the pipe's 36.8 TFMA/s), where four passes of one gate take 1350 us; a period
// 16.6 ms (104 gates), before 35.2 ms, at L = 20 0.17 ms for 0.39 ms.  Chains of
// up to 15 sites stay in shared memory between periods instead (k_resident.cu).
//
// complex64 (k_tile_f32): a thread holds 16 amplitudes (four register bits
// of the tile) and applies two gates on disjoint sites before it hands them
// back to the tile in shared memory; the next tile loads (cp.async) while
// this one is computed, and the last round writes the state directly where
// its lanes cover whole line parts.
// double-float (k_tile_df) and complex128 (k_tile_c128): their arithmetic (200 FP32
// operations or 16 FP64 FMA an amplitude and gate) is the bound already at one
// gate a pass; tiles there cut the launches of short chains and spread a short
// chain over the SMs.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "sv_device.cuh"
#include "sv_internal.h"
#include "sv_kernels.h"
#include "sv_tile.cuh"

namespace fsv {

namespace {

using namespace dev;

// ------------------------------------------------------------- complex64
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
template <typename R, typename Put>
__device__ __forceinline__ void load_gates(const TileArgs& ta, long long c, int entries,
                                           const Put& put) {
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
    put(k, v);
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
// kXor: the pass has gates in the order r ^ j; kEpi: measured gates (1: <X> terms
// only); passes without them run less code.  <X> alone fits three blocks an SM as
// unmeasured gates do: the last layer's four passes at L = 27 took 5.1 ms with one
// instance for all measured gates (two blocks), 4.1 ms with this one.
template <int kSlots, bool kXor, int kEpi, int kThreads, int kMinBlocks>
__global__ void __launch_bounds__(kThreads, kMinBlocks)
    k_tile_f32(float2* __restrict__ psi, const __grid_constant__ TileArgs ta,
               const __grid_constant__ TileTabOf<kSlots ? kSlots : 1> tab) {
  extern __shared__ __align__(16) uint8_t tile_smem[];
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
  grid_wait();
  grid_trigger();
  load_tile(ta, io, sbuf, psi + tile_base(ta, blockIdx.x));
  if (kSlots == 0)
    for (int k = threadIdx.x; k < 2 * ta.nrounds; k += blockDim.x)
      reinterpret_cast<uint4*>(rds)[k] = reinterpret_cast<const uint4*>(ta.rounds)[k];
  const bool reload = kSlots == 0 && (ta.stride != 0 || (ta.first && ta.ep.rn.ring));
  const long long c0 = reload ? *ta.counter : 0;
  double eacc = 0.0, nacc = 0.0;
  FloatSum esum, nsum;
  if (kSlots == 0) load_packed(ta, gs, c0);
  int cur = 0;
  const int last_r = ta.direct_out ? ta.nrounds - 1 : -1;  // the round that writes the state
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
      if (kEpi == 1 && rd.epi[0] && rd.egroup[0] != TILE_E_SWEEP)
        measure16_x<0, 1, 2, 3>(v, ta.cx, rd, 0, active, esum);
      if (kEpi == 2 && rd.epi[0] && rd.egroup[0] != TILE_E_SWEEP)
        measure16<0, 1, 2, 3>(v, ta.L, ta.cx, ta.ep, rd, 0, tbase + elem_state(ta, e0), active, esum,
                              nsum);
      if (rd.count == 2) {
        if (kXor && rd.xorder[1]) gate16<2, 3, 0, 1, true>(v, from(gb));
        else gate16<2, 3, 0, 1, false>(v, from(gb));
        if (kEpi == 1 && rd.epi[1] && rd.egroup[1] != TILE_E_SWEEP)
          measure16_x<2, 3, 0, 1>(v, ta.cx, rd, 1, active, esum);
        if (kEpi == 2 && rd.epi[1] && rd.egroup[1] != TILE_E_SWEEP)
          measure16<2, 3, 0, 1>(v, ta.L, ta.cx, ta.ep, rd, 1, tbase + elem_state(ta, e0), active, esum,
                                nsum);
      }
      if (active) {
        if (r == last_r) {
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
          measure_sweep<kEpi == 2>(tile, ta.tb, ta.L, ta.cx, ta.ep, rd.bond[sw], rd.epi[sw],
                        [&](uint32_t e) { return tbase + elem_state(ta, e); }, esum, nsum);
          __syncthreads();
        }
      }
    }
    if (kEpi && ta.any_epi) {
      esum.flush(eacc);
      nsum.flush(nacc);
    }
    if (!ta.direct_out) {
      store_tile(ta, io, tile, psi + tbase);
      __syncthreads();
    }
    if (ta.buffers == 2) cur ^= 1;
    else if (t + gridDim.x < ntiles) {
      load_tile(ta, io, sbuf, psi + tile_base(ta, t + gridDim.x));
    }
  }
  if (kEpi && ta.ep.partial) {
    block_store_pair(eacc, nacc, ta.ep.partial);
  }
}

// ---------------------------------------------------- double-float, packed
// A double-float complex number as two packed pairs, the leading and the trailing
// parts of (re, im): one packed operation serves both components.
struct PairDf {
  uint64_t hi, lo;
};
__device__ __forceinline__ PairDf pair_of(dfc v) {
  return PairDf{pk2(v.x.hi, v.y.hi), pk2(v.x.lo, v.y.lo)};
}
__device__ __forceinline__ dfc dfc_of(PairDf p) {
  const float2 h = un2(p.hi), l = un2(p.lo);
  dfc v;
  v.x = df(h.x, l.x);
  v.y = df(h.y, l.y);
  return v;
}
// (swapped: the product with an imaginary part)
__device__ __forceinline__ uint64_t swap2(uint64_t v) {
  const float2 t = un2(v);
  return pk2(t.y, t.x);
}
// acc + g v (s: v swapped): dot2_acc of both components, operation by operation,
// the errors of the products negated.  kFirst: acc is zero.
template <bool kFirst>
__device__ __forceinline__ PairDf cmac2(PairDf acc, const EntryDf& g, PairDf v, PairDf s) {
  const uint64_t p1 = mul2(g.re, v.hi), p2 = mul2(g.im, s.hi);
  uint64_t n1 = fma2(g.nre, v.hi, p1), n2 = fma2(g.nim, s.hi, p2);
  n1 = fma2(g.nre, v.lo, n1);
  n2 = fma2(g.nim, s.lo, n2);
  n1 = fma2(g.nre_lo, v.hi, n1);
  n2 = fma2(g.nim_lo, s.hi, n2);
  uint64_t l1 = 0, l2;
  const uint64_t s1 = kFirst ? p1 : two_sum2(acc.hi, p1, l1);
  const uint64_t s2 = two_sum2(s1, p2, l2);
  uint64_t lo = sub2(l2, n1);
  if (!kFirst) lo = add2(add2(acc.lo, l1), lo);
  lo = sub2(lo, n2);
  const uint64_t hi = add2(s2, lo);
  return PairDf{hi, sub2(lo, sub2(hi, s2))};
}

// kSlots: as in k_tile_f32.  A thread takes a group of four amplitudes, in place;
// after a tile's first round it holds pairs.
//
// The FP32 pipe bounds it: 100 packed operations (of two) an amplitude and gate,
// 0.93 ms a period at L = 21 at the pipe's 37.8 T/s, measured 1.40 ms (before, with
// scalar operations and table entries loaded from shared memory, 1.78 ms).  Packed,
// the operations take half the issue slots; with the entries in the constant bank
// they need no load.  24 warps an SM (80 registers) hide the chain of sums of each
// row better than 16 with more rows in flight: L = 20 0.77 and 0.91 ms.  A chain in
// one block (kMinBlocks 1) keeps all the registers instead (L = 8 37 and 45 us).
template <int kSlots, int kMinBlocks>
__global__ void __launch_bounds__(256, kMinBlocks)
    k_tile_df(dfc* __restrict__ psi, const __grid_constant__ TileArgs ta,
              const __grid_constant__ TileTabDf<kSlots ? kSlots : 1> tab) {
  constexpr int kEntries = 16;
  extern __shared__ __align__(16) uint8_t tile_smem[];
  __shared__ double red[2 * 16];
  const uint32_t N = 1u << ta.tb;
  PairDf* tile = reinterpret_cast<PairDf*>(tile_smem);
  PairDf* other = tile + N;  // the next tile
  EntryDf* gs = reinterpret_cast<EntryDf*>(ta.buffers == 2 ? other + N : other);
  TileRound* rds = reinterpret_cast<TileRound*>(gs + (size_t)ta.ngates * kEntries);
  const uint32_t groups = N >> 2;
  const uint32_t tid = threadIdx.x & (groups - 1);
  const bool active = threadIdx.x < groups;
  const uint32_t ntiles = 1u << (ta.L - ta.tb);
  auto load = [&](PairDf* to, uint32_t t) {
    const dfc* from = psi + tile_base(ta, t);
    for (uint32_t e = threadIdx.x; e < N; e += blockDim.x)
      cp_async16((uint32_t)__cvta_generic_to_shared(to + tile_slot16(e)), from + elem_state(ta, e));
    cp_commit();
  };
  grid_wait();
  grid_trigger();
  load(tile, blockIdx.x);
  if (kSlots == 0)
    for (int k = threadIdx.x; k < 2 * ta.nrounds; k += blockDim.x)
      reinterpret_cast<uint4*>(rds)[k] = reinterpret_cast<const uint4*>(ta.rounds)[k];
  const bool reload = kSlots == 0 && (ta.stride != 0 || (ta.first && ta.ep.rn.ring));
  const long long c0 = reload || ta.periods > 0 ? *ta.counter : 0;
  const int periods = ta.periods > 0 ? ta.periods : 1;
  double eacc = 0.0, nacc = 0.0;
  for (int p = 0; p < periods; ++p) {
    if (kSlots == 0 && (p == 0 || reload))
      load_gates<df>(ta, c0 + p, kEntries, [&](int k, const dfc& v) {
        gs[k] = df_entry(make_float4(v.x.hi, v.x.lo, v.y.hi, v.y.lo));
      });
    for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
      const uint64_t tbase = tile_base(ta, t);
      const bool more = t + gridDim.x < ntiles;
      if (ta.buffers == 2 && more) {
        load(other, t + gridDim.x);
        cp_wait<1>();
      } else {
        cp_wait<0>();
      }
      __syncthreads();
      const bool fresh = p == 0;  // the tile as it was loaded: numbers, not pairs
      for (int r = 0; r < ta.nrounds; ++r) {
        const TileRound& rd = kSlots ? tab.r[r] : rds[r];
        const EntryDf* const g = kSlots ? tab.g[rd.gate[0]] : gs + rd.gate[0] * kEntries;
        const uint32_t e0 = thread_elem<2>(rd, tid);
        const uint32_t s0 = tile_slot16(e0);
        const uint32_t sh = rd.slot[0], sl = rd.slot[1];
        PairDf v[4], s[4], w[4];
        auto at = [&](int m) -> PairDf& { return tile[s0 ^ ((m & 2) ? sh : 0) ^ ((m & 1) ? sl : 0)]; };
        if (r == 0 && fresh) {
#pragma unroll
          for (int m = 0; m < 4; ++m) v[m] = pair_of(*reinterpret_cast<const dfc*>(&at(m)));
        } else {
#pragma unroll
          for (int m = 0; m < 4; ++m) v[m] = at(m);
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) s[m] = PairDf{swap2(v[m].hi), swap2(v[m].lo)};
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          w[m] = cmac2<true>(PairDf{0, 0}, g[4 * m], v[0], s[0]);
#pragma unroll
          for (int c = 1; c < 4; ++c) w[m] = cmac2<false>(w[m], g[4 * m + c], v[c], s[c]);
        }
        if (active) {
          if (r == ta.nrounds - 1 && ta.direct_out && p == periods - 1) {
            dfc* out = psi + tbase + elem_state(ta, e0);
            const uint64_t xh = 1ull << rd.sbit[0], xl = 1ull << rd.sbit[1];
#pragma unroll
            for (int m = 0; m < 4; ++m) out[((m & 2) ? xh : 0) + ((m & 1) ? xl : 0)] = dfc_of(w[m]);
          } else {
#pragma unroll
            for (int m = 0; m < 4; ++m) at(m) = w[m];
          }
        }
        __syncthreads();
        if (rd.epi[0] && active) {
          const df cxh = (df)ta.cx64[rd.bond[0]], cxl = (df)ta.cx64[rd.bond[0] + 1];
          Diag<df> dg;
          if (rd.epi[0] & EPI_DIAG) dg.init(ta.ep, ta.L);
          const uint64_t xh = 1ull << rd.sbit[0], xl = 1ull << rd.sbit[1];
          const uint64_t off[4] = {0, xl, xh, xh + xl};
          const dfc a[4] = {dfc_of(w[0]), dfc_of(w[1]), dfc_of(w[2]), dfc_of(w[3])};
          GroupTerms<df> gt;
          group_terms<df>(a, rd.epi[0], dg, tbase + elem_state(ta, e0), off, gt);
          df es = 0, ns = 0;
          group_chain<df>(gt, rd.epi[0], cxh, cxl, es, ns);
          eacc += (double)es;
          nacc += (double)ns;
        }
      }
      if (!ta.direct_out && p == periods - 1) {
        dfc* out = psi + tbase;
        for (uint32_t e = threadIdx.x; e < N; e += blockDim.x)
          out[elem_state(ta, e)] = dfc_of(tile[tile_slot16(e)]);
        __syncthreads();
      }
      if (ta.buffers == 2) {
        PairDf* const swap = tile;
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

// ---------------------------------------------------------------- complex128
// A thread takes one output amplitude, between two copies of the tile (the FP64
// units are busy for 16 cycles a warp instruction, so the extra shared-memory
// reads cost nothing and every lane has work): L = 13 0.10 ms a period, one gate a
// launch 0.53 ms; at L = 21 the FP64 pipe bounds it (84 gates 3.6 ms at its 0.59
// TFMA/s, measured 5.0 ms).
template <int kThreads, int kMinBlocks>
__global__ void __launch_bounds__(kThreads, kMinBlocks)
    k_tile_c128(double2* __restrict__ psi, const __grid_constant__ TileArgs ta) {
  using R = double;
  using C = double2;
  constexpr int kEntries = 16;
  extern __shared__ __align__(16) uint8_t tile_smem[];
  __shared__ double red[2 * 16];
  const uint32_t N = 1u << ta.tb;
  C* tile = reinterpret_cast<C*>(tile_smem);
  C* other = tile + N;
  C* gs = other + N;
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
  grid_wait();
  grid_trigger();
  load(tile, blockIdx.x);
  for (int k = threadIdx.x; k < 2 * ta.nrounds; k += blockDim.x)
    reinterpret_cast<uint4*>(rds)[k] = reinterpret_cast<const uint4*>(ta.rounds)[k];
  const bool reload = ta.stride != 0 || (ta.first && ta.ep.rn.ring);
  const long long c0 = reload || ta.periods > 0 ? *ta.counter : 0;
  const int periods = ta.periods > 0 ? ta.periods : 1;
  double eacc = 0.0, nacc = 0.0;
  for (int p = 0; p < periods; ++p) {
    if (p == 0 || reload)
      load_gates<R>(ta, c0 + p, kEntries, [&](int k, const C& v) { gs[k] = v; });
    for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
      const uint64_t tbase = tile_base(ta, t);
      cp_wait<0>();
      __syncthreads();
      for (int r = 0; r < ta.nrounds; ++r) {
        const TileRound rd = rds[r];
        const C* g = gs + rd.gate[0] * kEntries;
        const uint32_t e0 = thread_elem<2>(rd, tid);
        const uint32_t s0 = tile_slot16(e0);
        const uint32_t sh = rd.slot[0], sl = rd.slot[1];
        const uint64_t xh = 1ull << rd.sbit[0], xl = 1ull << rd.sbit[1];
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
        if (rd.epi[0] && active) {
          C w[4];
#pragma unroll
          for (int m = 0; m < 4; ++m) w[m] = tile[s0 ^ ((m & 2) ? sh : 0) ^ ((m & 1) ? sl : 0)];
          const R cxh = (R)ta.cx64[rd.bond[0]], cxl = (R)ta.cx64[rd.bond[0] + 1];
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
      if (p == periods - 1) {
        C* out = psi + tbase;
        for (uint32_t e = threadIdx.x; e < N; e += blockDim.x)
          out[elem_state(ta, e)] = tile[tile_slot16(e)];
        __syncthreads();
      }
      if (t + gridDim.x < ntiles) load(tile, t + gridDim.x);
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
    b += (size_t)ta.ngates * 16 * (precision == SV_C64 ? 2 * sizeof(PackedEntry)
                                   : precision == SV_DF64 ? sizeof(EntryDf)
                                                          : sizeof(double2)) +
         (size_t)ta.nrounds * sizeof(TileRound);
  return b;
}

const void* tile_kernel(int precision, const TileArgs& ta) {
  if (precision == SV_C128) return reinterpret_cast<const void*>(k_tile_c128<512, 2>);
  if (precision == SV_DF64)
    return ta.in_params   ? reinterpret_cast<const void*>(k_tile_df<kTileTabSlots, 3>)
           : ta.tb < ta.L ? reinterpret_cast<const void*>(k_tile_df<0, 3>)
                          : reinterpret_cast<const void*>(k_tile_df<0, 1>);
  const int epi = !ta.any_epi ? 0 : (ta.any_epi & EPI_DIAG) ? 2 : 1;
  if (!ta.in_params)
    return epi             ? reinterpret_cast<const void*>(k_tile_f32<0, true, 2, 256, 2>)
           : ta.any_xorder ? reinterpret_cast<const void*>(k_tile_f32<0, true, 0, 256, 2>)
                           : reinterpret_cast<const void*>(k_tile_f32<0, false, 0, 256, 2>);
  if (epi == 2) return reinterpret_cast<const void*>(k_tile_f32<kTileTabSlots, true, 2, 256, 2>);
  if (epi == 1) return reinterpret_cast<const void*>(k_tile_f32<kTileTabSlots, true, 1, 256, 3>);
  return ta.any_xorder ? reinterpret_cast<const void*>(k_tile_f32<kTileTabSlots, true, 0, 256, 3>)
                       : reinterpret_cast<const void*>(k_tile_f32<kTileTabSlots, false, 0, 256, 3>);
}

}  // namespace

cudaError_t tile_grid(int precision, TileArgs* ta, const LaunchCfg& cfg, int* grid) {
  const uint64_t tiles = 1ull << (ta->L - ta->tb);
  const void* kernel = tile_kernel(precision, *ta);
  // every pass of an instance asks for the same limit (its largest)
  cudaError_t e =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kEvenSmemMax);
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
  // Passes of one tile a block start under the one before (20 sites 174 us a period, in
  // turn 176); of several tiles they gain nothing (22 sites 505 and 497 us).
  ta->overlap = cfg.alone() && tiles <= (uint64_t)cfg.num_sms * per_sm;
  ta->smem = (uint32_t)tile_smem_bytes(precision, *ta);
  if (ta->overlap) ta->smem = (uint32_t)even_smem(*grid, cfg.num_sms, ta->smem);
  return e;
}

cudaError_t launch_tile(int precision, void* psi, const TileArgs& ta, const TileTab* tab,
                        const TileTabDf<kTileTabSlots>* tab_df, int grid, cudaStream_t s) {
  if (ta.smem < tile_smem_bytes(precision, ta)) return cudaErrorInvalidValue;
  TileTabOf<1> none;
  TileTabDf<1> none_df;
  void* args[] = {&psi, const_cast<TileArgs*>(&ta), nullptr};
  if (precision == SV_C64) args[2] = ta.in_params ? (void*)const_cast<TileTab*>(tab) : (void*)&none;
  if (precision == SV_DF64)
    args[2] = ta.in_params ? (void*)const_cast<TileTabDf<kTileTabSlots>*>(tab_df) : (void*)&none_df;
  return launch_overlapped(tile_kernel(precision, ta), grid, tile_threads(precision, ta.tb), ta.smem, s,
                           args, ta.overlap);
}

}  // namespace fsv
