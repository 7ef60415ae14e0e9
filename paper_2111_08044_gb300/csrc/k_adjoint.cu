// Adjoint (reverse-mode) gradient of the final energy density with respect
// to per-period drive parameters: the state psi and the adjoint state
// lambda are walked back through the period's operations, each un-applied
// on both, while 2 Re <lambda| dO O^dagger |psi> is accumulated (the
// derivative of <psi_P|H0|psi_P>/L through operation O, evaluated after it).
// Reverse evolution by U^dagger is the echo construction of Sec. V; the
// energy observable is Eq. 7 divided by L.
//
// Kernels:
//   k_apply_h0      lambda = (H0 / L) psi, and per-block partials of
//                   Re <psi|lambda> (the energy density of a unit-norm psi);
//   k_adjoint_gate  one two-site operation on bond (b, b+1): accumulates
//                   Re <lambda|D|psi> (D = dO O^dagger), then psi <- O^dag psi
//                   and lambda <- O^dag lambda, in place;
//   k_adjoint_tile  the same for several operations, on tiles of both states
//                   (complex64 from five sites);
//   k_grad_reduce   the partials of a range of passes, summed in a fixed
//                   order, times 2, into one gradient entry.
#include <cuda_runtime.h>

#include <cstdint>

#include "sv_device.cuh"
#include "sv_internal.h"
#include "sv_kernels.h"
#include "sv_tile.cuh"

namespace fsv {

namespace {

using namespace dev;

constexpr int kThreads = 256;
constexpr int kBlocksPerSM = 4;

// Deterministic block sum of v, written to out[blockIdx.x].
__device__ inline void block_store(double v, double* out) {
  __shared__ double sv[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) sv[w] = v;
  __syncthreads();
  if (w == 0) {
    const int nw = blockDim.x >> 5;
    v = l < nw ? sv[l] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (l == 0) out[blockIdx.x] = v;
  }
}

template <typename R>
__global__ void __launch_bounds__(kThreads) k_apply_h0(const typename CT<R>::C* __restrict__ psi,
                                                       typename CT<R>::C* __restrict__ lam,
                                                       int L, H0Coef h, double* partial) {
  using C = typename CT<R>::C;
  // the coefficients once in the state's precision (no FP64 work per amplitude
  // for complex64)
  __shared__ R s_cx[34], s_cz[34];
  if (threadIdx.x < (unsigned)L) {
    s_cx[threadIdx.x] = (R)h.cx[threadIdx.x];
    s_cz[threadIdx.x] = (R)h.cz[threadIdx.x];
  }
  const R J = (R)h.J;
  __syncthreads();
  const uint64_t n = 1ull << L;
  const R inv_l = (R)(1.0 / L);
  double acc = 0.0;
  for (uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
       x += (uint64_t)gridDim.x * blockDim.x) {
    const C v = psi[x];
    // diagonal part: J sum_b z_b z_{b+1} + sum_i cz_i z_i, z = 1 - 2 b_i
    R d = 0;
    for (int i = 0; i < L; ++i) {
      const R zi = ((x >> i) & 1) ? (R)-1 : (R)1;
      d += s_cz[i] * zi;
      if (i + 1 < L) d += J * zi * (((x >> (i + 1)) & 1) ? (R)-1 : (R)1);
    }
    C out;
    out.x = d * v.x;
    out.y = d * v.y;
    // transverse part: sum_i cx_i X_i flips bit i
    for (int i = 0; i < L; ++i) {
      const C u = psi[x ^ (1ull << i)];
      out.x += s_cx[i] * u.x;
      out.y += s_cx[i] * u.y;
    }
    out.x *= inv_l;
    out.y *= inv_l;
    lam[x] = out;
    acc += (double)cdotre(v, out);
  }
  block_store(acc, partial);
}

template <typename R>
__global__ void __launch_bounds__(kThreads) k_adjoint_gate(typename CT<R>::C* __restrict__ psi,
                                                           typename CT<R>::C* __restrict__ lam,
                                                           int L, int b,
                                                           const typename CT<R>::C* __restrict__ od,
                                                           const typename CT<R>::C* __restrict__ dd,
                                                           double* partial) {
  using C = typename CT<R>::C;
  // od: O^dagger, dd: D = dO O^dagger; both 4x4 row-major with the local
  // index r = 2 b_b + b_{b+1} (site b is the high bit)
  __shared__ C so[16], sd[16];
  if (threadIdx.x < 16) {
    so[threadIdx.x] = od[threadIdx.x];
    sd[threadIdx.x] = dd[threadIdx.x];
  }
  __syncthreads();
  const uint64_t ng = 1ull << (L - 2);
  const uint64_t lowmask = (1ull << b) - 1;
  const uint64_t off[4] = {0, 2ull << b, 1ull << b, 3ull << b};  // r = 0..3
  double acc = 0.0;
  for (uint64_t g = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; g < ng;
       g += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t x = (g & lowmask) | ((g >> b) << (b + 2));
    C v[4], w[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      v[r] = psi[x + off[r]];
      w[r] = lam[x + off[r]];
    }
    R t = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      C dv = czero<C>();
#pragma unroll
      for (int c = 0; c < 4; ++c) dv = cmac(dv, sd[4 * r + c], v[c]);
      t += cdotre(w[r], dv);
    }
    acc += (double)t;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      C pv = czero<C>(), pw = czero<C>();
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        pv = cmac(pv, so[4 * r + c], v[c]);
        pw = cmac(pw, so[4 * r + c], w[c]);
      }
      psi[x + off[r]] = pv;
      lam[x + off[r]] = pw;
    }
  }
  block_store(acc, partial);
}

// ---------------------------------------------------------- tiles of both states
// 2x2 register bits of a thread's 16 amplitudes: index of member r, group k.
template <int J0, int J1, int K0, int K1>
__device__ __forceinline__ constexpr int member(int r, int k) {
  return ((r >> 1) << J0) | ((r & 1) << J1) | ((k & 1) << K0) | ((k >> 1) << K1);
}
// v <- table v (entries get(0..15)), each output the chain of cmac from zero
template <int J0, int J1, int K0, int K1, typename G>
__device__ __forceinline__ void apply16(uint64_t (&v)[16], const G& get) {
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
    for (int c = 0; c < 4; ++c) {
      const ulonglong2 g = get(4 * r + c);
#pragma unroll
      for (int k = 0; k < 4; ++k) w[r][k] = fma2(g.x, v[member<J0, J1, K0, K1>(c, k)], w[r][k]);
#pragma unroll
      for (int k = 0; k < 4; ++k) w[r][k] = fma2(g.y, s[member<J0, J1, K0, K1>(c, k)], w[r][k]);
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int k = 0; k < 4; ++k) v[member<J0, J1, K0, K1>(r, k)] = w[r][k];
}
// Re <lam|D|psi> of each group (entries get(16..31)), added to the sum
template <int J0, int J1, int K0, int K1, typename G>
__device__ __forceinline__ void derivative16(const uint64_t (&v)[16], const uint64_t (&l)[16],
                                             const G& get, FloatSum& sum) {
  float t[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    uint64_t w[4] = {0, 0, 0, 0};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const ulonglong2 g = get(16 + 4 * r + c);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint64_t x = v[member<J0, J1, K0, K1>(c, k)];
        const float2 f = un2(x);
        w[k] = fma2(g.x, x, w[k]);
        w[k] = fma2(g.y, pk2(f.y, f.x), w[k]);
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) t[k] += cdotre(un2(l[member<J0, J1, K0, K1>(r, k)]), un2(w[k]));
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) sum.add(t[k]);
}

// A pass of the reverse sweep: k_tile.cu's tiles, rounds and layout, on psi and
// lambda at once.  Per operation each group of four amplitudes gives its share
// of Re <lam|D|psi>, then both states take O^dagger: 50 FP32 FMA an amplitude,
// against 32 bytes of traffic a pass over both states.  One pass per operation
// was bound by its launch and by L2 (8.4 us an operation at L = 20, where its
// FMAs take 1.4 us); with four to six a pass the FP32 pipe is the bound.  Each
// group's arithmetic is that of k_adjoint_gate.
__global__ void __launch_bounds__(128, 4)
    k_adjoint_tile(float2* __restrict__ psi, float2* __restrict__ lam,
                   const __grid_constant__ AdjointPass ap, double* __restrict__ part,
                   const __grid_constant__ TileTab tab) {
  extern __shared__ __align__(16) uint8_t tile_smem[];
  const TileArgs& ta = ap.ta;
  const uint32_t tile_bytes = tile_byte8(1u << ta.tb);
  uint8_t* const tp = tile_smem;
  uint8_t* const tl = tile_smem + tile_bytes;
  const uint32_t sbuf = (uint32_t)__cvta_generic_to_shared(tile_smem);
  const int tbits = ta.tb - 4;
  const uint32_t tid = threadIdx.x & ((1u << tbits) - 1);
  const bool active = threadIdx.x < (1u << tbits);
  const uint32_t ntiles = 1u << (ta.L - ta.tb);
  const TileIo io = tile_io(ta);
  const uint64_t xout = elem_state(ta, thread_elem<4>(tab.r[ta.nrounds - 1], tid));
  double acc[2] = {0.0, 0.0};
  grid_wait();
  grid_trigger();
  for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const uint64_t tbase = tile_base(ta, t);
    load_tile(ta, io, sbuf, psi + tbase);
    load_tile(ta, io, sbuf + tile_bytes, lam + tbase);
    cp_wait<0>();
    __syncthreads();
    FloatSum sum[2];
    for (int r = 0; r < ta.nrounds; ++r) {
      const TileRound& rd = tab.r[r];
      const uint32_t at = tile_byte8(thread_elem<4>(rd, tid));
      const uint32_t sl0 = rd.slot[0], sl1 = rd.slot[1], sl2 = rd.slot[2], sl3 = rd.slot[3];
      uint64_t v[16], l[16];
#pragma unroll
      for (int m = 0; m < 16; ++m) {
        const uint32_t o = at + (((m & 1) ? sl0 : 0) + ((m & 2) ? sl1 : 0) + ((m & 4) ? sl2 : 0) +
                                 ((m & 8) ? sl3 : 0));
        v[m] = *reinterpret_cast<const uint64_t*>(tp + o);
        l[m] = *reinterpret_cast<const uint64_t*>(tl + o);
      }
      auto from = [&](int g) {
        return [&, g](int e) { return *reinterpret_cast<const ulonglong2*>(&tab.g[g][e]); };
      };
      const int ga = rd.gate[0], gb = rd.gate[1];
      derivative16<0, 1, 2, 3>(v, l, from(ga), ga < ap.nkick ? sum[0] : sum[1]);
      apply16<0, 1, 2, 3>(v, from(ga));
      apply16<0, 1, 2, 3>(l, from(ga));
      if (rd.count == 2) {
        derivative16<2, 3, 0, 1>(v, l, from(gb), gb < ap.nkick ? sum[0] : sum[1]);
        apply16<2, 3, 0, 1>(v, from(gb));
        apply16<2, 3, 0, 1>(l, from(gb));
      }
      if (active) {
        if (r == ta.nrounds - 1 && ta.direct_out) {
          uint64_t* const po = reinterpret_cast<uint64_t*>(psi + tbase + xout);
          uint64_t* const lo = reinterpret_cast<uint64_t*>(lam + tbase + xout);
          const uint64_t ro[4] = {1ull << rd.sbit[0], 1ull << rd.sbit[1], 1ull << rd.sbit[2],
                                  1ull << rd.sbit[3]};
#pragma unroll
          for (int m = 0; m < 16; ++m) {
            const uint64_t o = ((m & 1) ? ro[0] : 0) + ((m & 2) ? ro[1] : 0) +
                               ((m & 4) ? ro[2] : 0) + ((m & 8) ? ro[3] : 0);
            po[o] = v[m];
            lo[o] = l[m];
          }
        } else {
#pragma unroll
          for (int m = 0; m < 16; ++m) {
            const uint32_t o = at + (((m & 1) ? sl0 : 0) + ((m & 2) ? sl1 : 0) +
                                     ((m & 4) ? sl2 : 0) + ((m & 8) ? sl3 : 0));
            *reinterpret_cast<uint64_t*>(tp + o) = v[m];
            *reinterpret_cast<uint64_t*>(tl + o) = l[m];
          }
        }
      }
      __syncthreads();
    }
    if (active) {
      sum[0].flush(acc[0]);
      sum[1].flush(acc[1]);
    }
    if (!ta.direct_out) {
      store_tile(ta, io, tp, psi + tbase);
      store_tile(ta, io, tl, lam + tbase);
      __syncthreads();
    }
  }
  block_store_pair(acc[0], acc[1], part);
}

// (kick, field) partial pairs of one period a block, summed in a fixed order
__global__ void __launch_bounds__(kThreads) k_grad_reduce_pairs(const double* __restrict__ part,
                                                                int pairs, double* out) {
  const double* p = part + (size_t)blockIdx.x * pairs * 2;
  double a = 0.0, b = 0.0;
  for (int k = threadIdx.x; k < pairs; k += blockDim.x) {
    a += p[2 * k];
    b += p[2 * k + 1];
  }
  __shared__ double sh[2][kThreads];
  sh[0][threadIdx.x] = a;
  sh[1][threadIdx.x] = b;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + w];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x < 2) out[2 * blockIdx.x + threadIdx.x] = 2.0 * sh[threadIdx.x][0];
}

// out[0] = 2 * sum of partials[0 .. n), in a fixed order.
__global__ void __launch_bounds__(kThreads) k_grad_reduce(const double* __restrict__ partials,
                                                          long long n, double* out) {
  double s = 0.0;
  for (long long k = threadIdx.x; k < n; k += blockDim.x) s += partials[k];
  __shared__ double sh[kThreads];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = 2.0 * sh[0];
}

// out[0] = sum of partials (no factor), for the energy density
__global__ void __launch_bounds__(kThreads) k_sum(const double* __restrict__ partials, long long n,
                                                  double* out) {
  double s = 0.0;
  for (long long k = threadIdx.x; k < n; k += blockDim.x) s += partials[k];
  __shared__ double sh[kThreads];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = sh[0];
}

}  // namespace

int adjoint_grid(const LaunchCfg& cfg) { return cfg.num_sms * kBlocksPerSM; }

cudaError_t launch_apply_h0(int precision, const void* psi, void* lam, int L, const H0Coef& h,
                            double* partial, const LaunchCfg& cfg, cudaStream_t s) {
  const int grid = adjoint_grid(cfg);
  if (precision == SV_C128)
    k_apply_h0<double><<<grid, kThreads, 0, s>>>(static_cast<const double2*>(psi),
                                                 static_cast<double2*>(lam), L, h, partial);
  else
    k_apply_h0<float><<<grid, kThreads, 0, s>>>(static_cast<const float2*>(psi),
                                                static_cast<float2*>(lam), L, h, partial);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_gate(int precision, void* psi, void* lam, int L, int bond,
                                const void* odag, const void* dmat, double* partial,
                                const LaunchCfg& cfg, cudaStream_t s) {
  const int grid = adjoint_grid(cfg);
  if (precision == SV_C128)
    k_adjoint_gate<double><<<grid, kThreads, 0, s>>>(
        static_cast<double2*>(psi), static_cast<double2*>(lam), L, bond,
        static_cast<const double2*>(odag), static_cast<const double2*>(dmat), partial);
  else
    k_adjoint_gate<float><<<grid, kThreads, 0, s>>>(
        static_cast<float2*>(psi), static_cast<float2*>(lam), L, bond,
        static_cast<const float2*>(odag), static_cast<const float2*>(dmat), partial);
  return cudaGetLastError();
}

cudaError_t launch_grad_reduce(const double* partials, long long n, double* out, int times_two,
                               cudaStream_t s) {
  if (times_two)
    k_grad_reduce<<<1, kThreads, 0, s>>>(partials, n, out);
  else
    k_sum<<<1, kThreads, 0, s>>>(partials, n, out);
  return cudaGetLastError();
}

cudaError_t adjoint_tile_grid(AdjointPass* ap, const LaunchCfg& cfg, int* grid) {
  const TileArgs& ta = ap->ta;
  const int smem = 2 * (int)tile_byte8(1u << ta.tb);
  int per_sm = 1;
  cudaError_t e =
      cudaFuncSetAttribute(k_adjoint_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, kEvenSmemMax);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_adjoint_tile,
                                                      tile_threads(SV_C64, ta.tb), smem);
  const uint64_t most = (uint64_t)cfg.num_sms * (per_sm > 0 ? per_sm : 1);
  const uint64_t tiles = 1ull << (ta.L - ta.tb);
  *grid = (int)(tiles < most ? tiles : most);
  ap->ta.smem = (uint32_t)even_smem(*grid, cfg.num_sms, smem);
  return e;
}

cudaError_t launch_adjoint_tile(void* psi, void* lam, const AdjointPass& ap, const TileTab& tab,
                                double* part, int grid, cudaStream_t s) {
  void* args[] = {&psi, &lam, const_cast<AdjointPass*>(&ap), &part, const_cast<TileTab*>(&tab)};
  return launch_overlapped(reinterpret_cast<const void*>(k_adjoint_tile), grid,
                           tile_threads(SV_C64, ap.ta.tb), ap.ta.smem, s, args);
}

cudaError_t launch_grad_reduce_pairs(const double* part, int pairs, int periods, double* out,
                                     cudaStream_t s) {
  k_grad_reduce_pairs<<<periods, kThreads, 0, s>>>(part, pairs, out);
  return cudaGetLastError();
}

}  // namespace fsv
