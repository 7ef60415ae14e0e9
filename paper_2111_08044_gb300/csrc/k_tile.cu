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
// 17.9 ms (104 gates), before 35.2 ms, at L = 20 0.18 ms for 0.39 ms.  Chains of
// up to 15 sites stay in shared memory between periods instead (k_resident.cu).
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
      if (kEpi && rd.epi[0] && rd.egroup[0] != TILE_E_SWEEP)
        measure16<0, 1, 2, 3>(v, ta.L, ta.cx, ta.ep, rd, 0, tbase + elem_state(ta, e0), active, esum,
                              nsum);
      if (rd.count == 2) {
        if (kXor && rd.xorder[1]) gate16<2, 3, 0, 1, true>(v, from(gb));
        else gate16<2, 3, 0, 1, false>(v, from(gb));
        if (kEpi && rd.epi[1] && rd.egroup[1] != TILE_E_SWEEP)
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
          measure_sweep(tile, ta.tb, ta.L, ta.cx, ta.ep, rd.bond[sw], rd.epi[sw],
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

const void* tile_kernel(int precision, const TileArgs& ta) {
  if (precision == SV_DF64) return reinterpret_cast<const void*>(k_tile_wide<df, 256, 2>);
  if (precision == SV_C128) return reinterpret_cast<const void*>(k_tile_wide<double, 512, 2>);
  if (!ta.in_params) return reinterpret_cast<const void*>(k_tile_f32<0, true, true, 256, 2>);
  if (ta.any_epi) return reinterpret_cast<const void*>(k_tile_f32<kTileTabSlots, true, true, 256, 2>);
  return ta.any_xorder ? reinterpret_cast<const void*>(k_tile_f32<kTileTabSlots, true, false, 256, 3>)
                       : reinterpret_cast<const void*>(k_tile_f32<kTileTabSlots, false, false, 256, 3>);
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
  ta->overlap = cfg.alone();
  ta->smem = (uint32_t)tile_smem_bytes(precision, *ta);
  if (ta->overlap) ta->smem = (uint32_t)even_smem(*grid, cfg.num_sms, ta->smem);
  return e;
}

cudaError_t launch_tile(int precision, void* psi, const TileArgs& ta, const TileTab* tab, int grid,
                        cudaStream_t s) {
  if (ta.smem < tile_smem_bytes(precision, ta)) return cudaErrorInvalidValue;
  TileTabOf<1> none;
  void* args[] = {&psi, const_cast<TileArgs*>(&ta), nullptr};
  if (precision == SV_C64) args[2] = ta.in_params ? (void*)const_cast<TileTab*>(tab) : (void*)&none;
  return launch_overlapped(tile_kernel(precision, ta), grid, tile_threads(precision, ta.tb), ta.smem, s,
                           args, ta.overlap);
}

}  // namespace fsv
