// Measurements of a complex64 state of at least 13 sites, in tiles of 2^12
// amplitudes (on shorter chains a call is its launches and copies either way,
// and the per-gate and per-amplitude kernels stay).  Times at L = 25 (256 MiB;
// one read of it takes 40 us at the measured bandwidth):
//
//   k_energy_tile   <H0> of the driven chain and the norm: sums of <X> over the
//                   bits of a tile, and the diagonal part.  A pass covers the
//                   12 lowest sites or 8 further ones, so the state is read
//                   ceil((L - 12) / 8) + 1 times; one identity gate pass per
//                   pair of sites read it L / 2 times: 1217 -> 236 us a call.
//   k_moments_tile  H0 psi amplitude by amplitude, for E and sigma_E (Eq. 10 and
//   k_bond_moments_tile  11): partners within the tile from registers and shared
//                   memory, the others from the tiles whose number differs in
//                   one bit (or, for a general bond term, two), which mostly
//                   are in L2.  Bound by that traffic: L - 11 tiles read for one
//                   (Ising, 1230 -> 285 us); general bonds by instructions too
//                   (L = 24: 1080 -> 386 us).
//   k_overlap_f32   <phi|psi> of a product state from FP64 factor tables
//   k_factor_f32    and the state itself: the FP64 units (0.59 TFMA/s) bounded
//                   both; products and sums are FP32 triples and pairs here (an
//                   exact product and its error, Dekker and Knuth): 741 -> 142
//                   us; L = 24: 188 -> 57 us.
// Partial sums: FP32 over at most eight terms, FP32 pairs (overlaps: triples) across a
// thread's terms, FP64 across tiles, threads and blocks, in a fixed order.
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

constexpr int kThreads = 256;
constexpr int kBits = 12;  // tile bits: 16 amplitudes a thread
constexpr uint32_t kTileBytes = 8u * (1u << kBits) + 16u * (1u << (kBits - 4));
static_assert(kTileBytes <= 48 * 1024, "no shared-memory opt-in: the calls may be captured");

// Deterministic block sums of K doubles, written to out[K * blockIdx.x + j].
template <int K>
__device__ void block_store_k(double (&v)[K], double* out) {
  __shared__ double sh[K][32];
#pragma unroll
  for (int j = 0; j < K; ++j)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[j] += __shfl_xor_sync(0xffffffffu, v[j], o);
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int j = 0; j < K; ++j) sh[j][w] = v[j];
  __syncthreads();
  if (threadIdx.x < K) {
    double t = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += sh[threadIdx.x][k];
    out[K * blockIdx.x + threadIdx.x] = t;
  }
}

// The diagonal part of H0 over the amplitudes of one contiguous tile as an FP32 pair,
// from tables of its two counts: J (L - 1 - 2 flips), and the fields' sum for nb set
// bits between the ends and the two end bits.  A value of 20 rounded to FP32 is off by
// up to 1e-6, the same for every amplitude of its counts, which does not average out.
struct PairDiag {
  const float2 *zz, *field;  // shared memory: 34, and 4 a count
  int L, nb_hi, flips_hi, last;
  uint32_t top;
  __device__ static void fill(const H0Coef& h, int L, float2* zz, float2* field) {
    auto pair = [](double v) {
      const float hi = (float)v;
      return make_float2(hi, (float)(v - (double)hi));
    };
    const int k = threadIdx.x;
    if (k < L) zz[k] = pair(h.J * (L - 1 - 2 * k));
    if (k < 4 * (L - 1)) {
      const int nb = k >> 2;
      field[k] = pair(h.cz[1] * (L - 2 - 2 * nb) + ((k & 2) ? -h.cz[0] : h.cz[0]) +
                      ((k & 1) ? -h.cz[L - 1] : h.cz[L - 1]));
    }
  }
  __device__ void tile(uint32_t t) {
    const int hi = L - kBits;  // bits of the tile number, at least 1
    flips_hi = __popc((t ^ (t >> 1)) & ((1u << (hi - 1)) - 1));
    last = (t >> (hi - 1)) & 1;
    nb_hi = __popc(t) - last;
    top = (t & 1u) << kBits;
  }
  __device__ __forceinline__ df operator()(uint32_t e) const {
    const uint32_t x = e | top;
    const float2 a = zz[flips_hi + __popc((x ^ (x >> 1)) & ((1u << kBits) - 1))];
    const float2 b = field[4 * (nb_hi + __popc(e & ~1u)) + 2 * (e & 1) + last];
    const df s = two_sum(a.x, b.x);
    return df(s.hi, s.lo + (a.y + b.y));
  }
};

struct EnergyArgs {
  TileArgs ta;          // layout of the pass
  H0Coef h0;            // of the diagonal part
  float cx[kBits] = {};  // coefficient of each tile bit's <X> (0: another pass's)
  int low = 0;          // tile bits 0..3 measured too
  int diag = 0;
};

// 2 Re <v_0|v_1> over the eight pairs of register bit J
template <int J>
__device__ __forceinline__ float pair_sum(const float2 (&v)[16]) {
  float s = 0.f;
#pragma unroll
  for (int m = 0; m < 16; ++m)
    if (!(m & (1 << J))) s += cdotre(v[m], v[m | (1 << J)]);
  return 2.f * s;
}

__global__ void __launch_bounds__(kThreads, 4)
    k_energy_tile(const float2* __restrict__ psi, const __grid_constant__ EnergyArgs ea,
                  double* __restrict__ part) {
  extern __shared__ __align__(16) uint8_t tile[];
  const TileArgs& ta = ea.ta;
  const uint32_t sbuf = (uint32_t)__cvta_generic_to_shared(tile);
  const uint32_t ntiles = 1u << (ta.L - kBits);
  const uint32_t tid = threadIdx.x;
  const TileIo io = tile_io(ta);
  __shared__ float2 zz[34], field[4 * 33];
  if (ea.diag) PairDiag::fill(ea.h0, ta.L, zz, field);
  PairDiag dg{zz, field, ta.L};
  double acc[2] = {0.0, 0.0};
  for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    load_tile(ta, io, sbuf, psi + tile_base(ta, t));
    cp_wait<0>();
    __syncthreads();
    FloatSum es, ns;
    if (ea.diag) dg.tile(t);
    // the tile three times over, each time with other register bits: 8-11,
    // 4-7 and (where measured) 0-3
#pragma unroll
    for (int q = 8; q >= 0; q -= 4) {
      if (q == 0 && !ea.low) break;
      const uint32_t e0 = (tid & ((1u << q) - 1)) | ((tid >> q) << (q + 4));
      float2 v[16];
#pragma unroll
      for (int m = 0; m < 16; ++m)
        v[m] = *reinterpret_cast<const float2*>(tile + tile_byte8(e0 | ((uint32_t)m << q)));
      es.add(ea.cx[q] * pair_sum<0>(v));
      es.add(ea.cx[q + 1] * pair_sum<1>(v));
      es.add(ea.cx[q + 2] * pair_sum<2>(v));
      es.add(ea.cx[q + 3] * pair_sum<3>(v));
      if (q == 8 && ea.diag) {
        // The norm amplitude by amplitude, the diagonal energies four to a sum, their
        // trailing parts apart.  (With sixteen to a sum and the energies in FP32 the
        // norm was off by 4 to 12e-9 at 13..18 sites and the density by 1.6e-8, and L =
        // 25 took 222 us a call; now 0.8 to 3e-9, 2e-9 and 236 us.)
        float dl = 0.f;
#pragma unroll
        for (int g = 0; g < 16; g += 4) {
          float d = 0.f;
#pragma unroll
          for (int m = g; m < g + 4; ++m) {
            const float p = cabs2(v[m]);
            const df c = dg(e0 | ((uint32_t)m << q));
            ns.add(p);
            d = __fmaf_rn(p, c.hi, d);
            dl = __fmaf_rn(p, c.lo, dl);
          }
          es.add(d);
        }
        es.add(dl);
      }
    }
    es.flush(acc[0]);
    ns.flush(acc[1]);
    __syncthreads();
  }
  block_store_k<2>(acc, part);
}

// ------------------------------------------------------------------ moments
struct MomentArgs {
  int L = 0;
  float cx[34] = {};            // Ising: coefficients of X_i
  H0Coef h0;                    // Ising: diagonal coefficients (cz of sites 1..L-2 equal)
  float2 h[33][16] = {};        // general: bond terms
};

// Row r of a bond term as (h[r][r], h[r][r ^ 1], h[r][r ^ 2], h[r][r ^ 3]): the entries
// of the amplitude itself, of its partners with site b + 1, site b and both flipped.
// In shared memory: r is only known at run time.
struct BondRow {
  float4 a, b;
};
__device__ __forceinline__ float2 row_sum(const BondRow& h, float2 out, float2 same, float2 lo,
                                          float2 hi, float2 both) {
  out = cmac(out, make_float2(h.a.x, h.a.y), same);
  out = cmac(out, make_float2(h.a.z, h.a.w), lo);
  out = cmac(out, make_float2(h.b.x, h.b.y), hi);
  return cmac(out, make_float2(h.b.z, h.b.w), both);
}

// A thread's kA amplitudes of a tile of 2^kB: indices 2 tid + (0, 1) + 1024 j (bit 0
// of m: site 0, the bits above: sites 10 and on), so that every read of another tile
// is of whole lines; sites 1..9 are thread bits, their partners in the tile.
constexpr int kMomentThreads = 512;
template <int kA>
struct MomentTile {
  static constexpr int kB = kA == 8 ? 12 : 11;  // tile bits
  uint8_t* tile;
  const float2* psi;
  uint32_t tid;
  __device__ __forceinline__ void set(float2 (&u)[kA], int j, float4 q) const {
    u[2 * j] = make_float2(q.x, q.y);
    u[2 * j + 1] = make_float2(q.z, q.w);
  }
  __device__ __forceinline__ void read(uint32_t from, float2 (&u)[kA]) const {
    const float4* p = reinterpret_cast<const float4*>(psi + ((uint64_t)from << kB));
#pragma unroll
    for (int j = 0; j < kA / 2; ++j) set(u, j, __ldg(p + tid + kMomentThreads * j));
  }
  __device__ __forceinline__ void put(const float2 (&v)[kA]) const {
#pragma unroll
    for (int j = 0; j < kA / 2; ++j)
      *reinterpret_cast<float4*>(tile + tile_byte8(2 * tid + 1024 * j)) =
          make_float4(v[2 * j].x, v[2 * j].y, v[2 * j + 1].x, v[2 * j + 1].y);
  }
  __device__ __forceinline__ void partner(uint32_t flip, float2 (&u)[kA]) const {  // flip: bits 1..9
#pragma unroll
    for (int j = 0; j < kA / 2; ++j)
      set(u, j, *reinterpret_cast<const float4*>(tile + tile_byte8(((2 * tid) ^ flip) + 1024 * j)));
  }
  // <psi|H0|psi>, |H0 psi|^2 and the norm
  __device__ __forceinline__ static void sums(const float2 (&v)[kA], const float2 (&hv)[kA],
                                              double (&acc)[3]) {
    FloatSum s[3];
#pragma unroll
    for (int m = 0; m < kA; ++m) {
      s[0].add(v[m].x * hv[m].x + v[m].y * hv[m].y);
      s[1].add(hv[m].x * hv[m].x + hv[m].y * hv[m].y);
      s[2].add(v[m].x * v[m].x + v[m].y * v[m].y);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) s[k].flush(acc[k]);
  }
};

__global__ void __launch_bounds__(kMomentThreads, 2)
    k_moments_tile(const float2* __restrict__ psi, const __grid_constant__ MomentArgs ma,
                   double* __restrict__ part) {
  extern __shared__ __align__(16) uint8_t tile[];
  constexpr int kA = 8;
  const int L = ma.L;
  const uint32_t ntiles = 1u << (L - kBits);
  const MomentTile<kA> mt{tile, psi, threadIdx.x};
  const uint32_t e0 = 2 * threadIdx.x;
  __shared__ float2 zz[34], field[4 * 33];
  PairDiag::fill(ma.h0, L, zz, field);
  PairDiag dg{zz, field, L};
  __syncthreads();
  double acc[3] = {0.0, 0.0, 0.0};
  for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    float2 v[kA], hv[kA], a[kA];
    mt.read(t, v);
    mt.put(v);
    __syncthreads();
    dg.tile(t);
    auto add = [&](float c, const float2 (&u)[kA]) {
#pragma unroll
      for (int m = 0; m < kA; ++m) {
        hv[m].x += c * u[m].x;
        hv[m].y += c * u[m].y;
      }
    };
#pragma unroll
    for (int m = 0; m < kA; ++m) {
      const df d = dg(e0 + 1024 * (m >> 1) + (m & 1));
      hv[m] = make_float2(__fmaf_rn(d.lo, v[m].x, d.hi * v[m].x), __fmaf_rn(d.lo, v[m].y, d.hi * v[m].y));
#pragma unroll
      for (int k = 0; k < 3; ++k) {  // sites 0, 10, 11: within the thread
        const float c = ma.cx[k == 0 ? 0 : 9 + k];
        hv[m].x += c * v[m ^ (1 << k)].x;
        hv[m].y += c * v[m ^ (1 << k)].y;
      }
    }
#pragma unroll
    for (int i = 1; i < 10; ++i) {
      mt.partner(1u << i, a);
      add(ma.cx[i], a);
    }
#pragma unroll 4
    for (int i = kBits; i < L; ++i) {
      mt.read(t ^ (1u << (i - kBits)), a);
      add(ma.cx[i], a);
    }
    MomentTile<kA>::sums(v, hv, acc);
    __syncthreads();
  }
  block_store_k<3>(acc, part);
}

// General bond terms hold four arrays of partners, so tiles of 2^11: 64 registers a
// thread, two blocks an SM.  Bound by instructions: 16 FMA an amplitude and bond (L =
// 24: 168 us at the pipe's rate) beside the partners' loads; two rows of the term come
// from shared memory (entries selected from the parameters took as many again).
// 393 us at L = 24; 590 us so, and in tiles of 2^12 and one block an SM 750 us.
__global__ void __launch_bounds__(kMomentThreads, 2)
    k_bond_moments_tile(const float2* __restrict__ psi, const __grid_constant__ MomentArgs ma,
                        double* __restrict__ part) {
  extern __shared__ __align__(16) uint8_t tile[];
  __shared__ BondRow rows[33][4];
  constexpr int kA = 4, kB = MomentTile<kA>::kB;
  const int L = ma.L;
  const uint32_t ntiles = 1u << (L - kB);
  const uint32_t tid = threadIdx.x;
  const MomentTile<kA> mt{tile, psi, tid};
  for (uint32_t q = tid; q < 16u * (L - 1); q += kMomentThreads) {
    const uint32_t r = (q >> 2) & 3, c = q & 3;
    reinterpret_cast<float2*>(rows)[q] = ma.h[q >> 4][4 * r + (r ^ c)];
  }
  double acc[3] = {0.0, 0.0, 0.0};
  for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    float2 v[kA], hv[kA], a[kA], b[kA], c[kA];
    mt.read(t, v);
    mt.put(v);
    __syncthreads();
#pragma unroll
    for (int m = 0; m < kA; ++m) hv[m] = make_float2(0.f, 0.f);
    // (0, 1)
    mt.partner(2, a);
    const int s1 = tid & 1;
#pragma unroll
    for (int m = 0; m < kA; ++m)
      hv[m] = row_sum(rows[0][2 * (m & 1) + s1], hv[m], v[m], a[m], v[m ^ 1], a[m ^ 1]);
    // (i, i + 1), i = 1..8: both thread bits; a holds site i's partner
#pragma unroll 1
    for (int i = 1; i < 9; ++i) {
      mt.partner(2u << i, b);
      mt.partner(3u << i, c);
      const BondRow h = rows[i][2 * ((tid >> (i - 1)) & 1) + ((tid >> i) & 1)];
#pragma unroll
      for (int m = 0; m < kA; ++m) {
        hv[m] = row_sum(h, hv[m], v[m], b[m], a[m], c[m]);
        a[m] = b[m];
      }
    }
    // (9, 10)
    const int s9 = (int)(tid >> 8);
#pragma unroll
    for (int m = 0; m < kA; ++m)
      hv[m] = row_sum(rows[9][2 * s9 + (m >> 1)], hv[m], v[m], v[m ^ 2], a[m], a[m ^ 2]);
    // (10, 11): site 11 is the tile number's bit 0
    mt.read(t ^ 1u, a);
    const int s11 = (int)(t & 1u);
#pragma unroll
    for (int m = 0; m < kA; ++m)
      hv[m] = row_sum(rows[10][2 * (m >> 1) + s11], hv[m], v[m], a[m], v[m ^ 2], a[m ^ 2]);
#pragma unroll 2
    for (int i = kB; i + 1 < L; ++i) {  // a holds site i's partner
      const uint32_t at = i - kB;
      mt.read(t ^ (2u << at), b);
      mt.read(t ^ (3u << at), c);
      const BondRow h = rows[i][2 * ((t >> at) & 1) + ((t >> (at + 1)) & 1)];
#pragma unroll
      for (int m = 0; m < kA; ++m) {
        hv[m] = row_sum(h, hv[m], v[m], b[m], a[m], c[m]);
        a[m] = b[m];
      }
    }
    MomentTile<kA>::sums(v, hv, acc);
    __syncthreads();
  }
  block_store_k<3>(acc, part);
}

// --------------------------------------------------- products of FP64 factors
// Double-precision table entry as FP32 pairs (48 bits).
__device__ __forceinline__ float4 split_pair(double2 v) {
  const float xr = (float)v.x, xi = (float)v.y;
  return make_float4(xr, (float)(v.x - (double)xr), xi, (float)(v.y - (double)xi));
}
// A packed sum of products (re, im) in three FP32 parts s + c + d, each addition exact
// in the leading two.  A factor x as packed operands: leading part and its negative, the
// middle one's, the trailing one's negative (24 + 24 + 5 bits: all of an FP64 value).
struct TripleFactor {
  uint64_t x, nx, m, nm, nt;
};
struct TripleSum {
  uint64_t s = 0, c = 0, d = 0;
  __device__ __forceinline__ void add(const TripleFactor& g, uint64_t v) {
    const uint64_t p = mul2(g.x, v), pe = fma2(g.nx, v, p);  // pe, qe: errors, negated
    const uint64_t q = mul2(g.m, v), qe = fma2(g.nt, v, fma2(g.nm, v, q));
    uint64_t t, e1, e2, e3;
    s = two_sum2(s, p, t);
    c = two_sum2(c, t, e1);
    const uint64_t r = sub2(c, pe), b = sub2(r, c);  // c - pe and its error
    e2 = sub2(sub2(c, sub2(r, b)), add2(pe, b));
    c = two_sum2(r, q, e3);
    d = add2(d, sub2(add2(add2(e1, e2), e3), qe));
  }
  __device__ __forceinline__ void add(const TripleSum& o) {
    uint64_t t, e1, e2;
    s = two_sum2(s, o.s, t);
    c = two_sum2(c, o.c, e1);
    c = two_sum2(c, t, e2);
    d = add2(add2(d, o.d), add2(e1, e2));
  }
};

// <phi|psi> = sum_m conj(lo[m]) sum_k conj(hi[k]) psi[k, m]: a block keeps the inner
// sums of a quarter of the low indices m, a thread two of them in four parts, over its
// chunks k.  So FP64 is left for two products a thread (with eight low indices a
// thread a call at 13 to 18 sites took 60 us, now 50).
//
// Bound by the FP32 pipe: 66 packed operations an amplitude, 117 us at L = 25 at the
// pipe's rate, measured 142 us; 76 us at L = 24, 13 us at L = 20.  In two FP32 parts (44
// scalar operations) 92, 57 and 24 us, but an overlap was off by 6 to 9e-14 of its
// value (rms, 13 to 20 sites) where it is by 1 to 2e-15 now and was by 1 to 4e-15 in FP64 (741
// us), and what lies below FP32's range was lost.  (A fourth of the sums in FP64 beside
// them: 130 us, but sparse states then take the sums again.)
//
// Where an inner sum is so small that FP32 parts of its terms may have been lost
// (below 2^-126 each, against 2^-70), or not finite, the thread takes it again in FP64.
constexpr int kOverlapThreads = 512;
// (double)f of a normal number or zero, without the FP64 unit; subnormal: zero
__device__ __forceinline__ double widen(float f) {
  const uint32_t u = __float_as_uint(f);
  const bool z = (u & 0x7f800000u) == 0;
  const uint32_t hi = (u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u);
  return __hiloint2double(z ? 0 : (int)hi, z ? 0 : (int)(u << 29));
}
__global__ void __launch_bounds__(kOverlapThreads, 1)
    k_overlap_f32(const float2* __restrict__ psi, int L, const double2* __restrict__ lo,
                  const double2* __restrict__ hi, double* __restrict__ part) {
  const uint32_t chunks = 1u << (L - kBits), tid = threadIdx.x, lane = tid & 31;
  const uint32_t slice = blockIdx.x & 3, first = blockIdx.x >> 2, step = gridDim.x >> 2;
  const uint32_t n = first < chunks ? (chunks - first + step - 1) / step : 0;  // chunks of the block
  const uint32_t at0 = 2 * kOverlapThreads * slice + 2 * tid;  // the thread's first m
  auto read = [&](uint32_t i, float4 (&u)[4]) {  // of chunks i .. i + 3 of the block's
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (i + j < n)
        u[j] = __ldg(reinterpret_cast<const float4*>(psi + ((uint64_t)(first + (i + j) * step) << kBits) + at0));
  };
  TripleSum sum[4][2];
  float vmax = 0.f, hmax = 0.f;
  uint32_t any = 0;  // bit m: an amplitude other than zero
  float4 next[4];
  read(0, next);
  for (uint32_t i0 = 0; i0 < n; i0 += 32) {
    // a lane splits the factor of one of the next 32 chunks
    float part3[2][3] = {};
    if (i0 + lane < n) {
      const double2 h = hi[first + (i0 + lane) * step];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        double r = i ? h.y : h.x;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          part3[i][j] = (float)r;
          r -= (double)part3[i][j];
        }
      }
      hmax = fmaxf(hmax, (h.x != 0.0 || h.y != 0.0) ? 1.f : 0.f);
    }
#pragma unroll 1
    for (uint32_t i = i0; i < n && i < i0 + 32; i += 4) {
      float4 u[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) u[j] = next[j];
      read(i + 4, next);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (i + j >= n) break;
        TripleFactor g[2];  // (re, re) and (im, -im)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          float f[3];
#pragma unroll
          for (int q = 0; q < 3; ++q) f[q] = __shfl_sync(0xffffffffu, part3[k][q], i - i0 + j);
          const float sg = k ? -1.f : 1.f;
          g[k] = TripleFactor{pk2(f[0], sg * f[0]), pk2(-f[0], -sg * f[0]), pk2(f[1], sg * f[1]),
                              pk2(-f[1], -sg * f[1]), pk2(-f[2], -sg * f[2])};
        }
        vmax = fmaxf(vmax, fmaxf(fmaxf(fabsf(u[j].x), fabsf(u[j].y)), fmaxf(fabsf(u[j].z), fabsf(u[j].w))));
        any |= (u[j].x != 0.f || u[j].y != 0.f) ? 1u : 0u;
        any |= (u[j].z != 0.f || u[j].w != 0.f) ? 2u : 0u;
        sum[j][0].add(g[0], pk2(u[j].x, u[j].y));
        sum[j][0].add(g[1], pk2(u[j].y, u[j].x));
        sum[j][1].add(g[0], pk2(u[j].z, u[j].w));
        sum[j][1].add(g[1], pk2(u[j].w, u[j].z));
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) hmax = fmaxf(hmax, __shfl_xor_sync(0xffffffffu, hmax, o));
  double acc[2] = {0.0, 0.0};
  const float least = 0x1p-70f * fmaxf(vmax, 1.f);
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    const uint32_t at = at0 + m;
    const double2 g = lo[at];
    sum[0][m].add(sum[1][m]);
    sum[2][m].add(sum[3][m]);
    sum[0][m].add(sum[2][m]);
    const float2 s = un2(sum[0][m].s), c = un2(sum[0][m].c), d = un2(sum[0][m].d);
    double re = widen(s.x) + (widen(c.x) + widen(d.x));
    double im = widen(s.y) + (widen(c.y) + widen(d.y));
    const float size = fabsf(s.x) + fabsf(s.y);
    // (not where every term is zero; vmax passes over NaN, size does not)
    if (!(size >= least && size <= 3e38f) && hmax != 0.f && (g.x != 0.0 || g.y != 0.0) &&
        ((any >> m) & 1)) {
      re = im = 0.0;
#pragma unroll 1
      for (uint32_t k = first; k < chunks; k += step) {
        const float2 v = __ldg(psi + ((uint64_t)k << kBits) + at);
        const double2 h = hi[k];
        re += h.x * (double)v.x + h.y * (double)v.y;
        im += h.x * (double)v.y - h.y * (double)v.x;
      }
    }
    acc[0] += g.x * re + g.y * im;
    acc[1] += g.x * im - g.y * re;
  }
  block_store_k<2>(acc, part);
}

// a b - c d with FP32 pairs, rounded once
__device__ __forceinline__ float mul_sub(float ah, float al, float bh, float bl, float ch, float cl,
                                         float dh, float dl) {
  return dot2_acc(df(0.f, 0.f), df(ah, al), df(bh, bl), df(-ch, -cl), df(dh, dl)).hi;
}

// The thread's amplitudes in `small` again, in FP64 (a call: kept out of the others' way).
__device__ __noinline__ void factor_small(float2* chunk, const double2* lo, double2 h, uint32_t small) {
  for (; small; small &= small - 1) {
    const uint32_t m = __ffs(small) - 1, at = 2 * threadIdx.x + 512 * (m >> 1) + (m & 1);
    const double2 g = lo[at];
    chunk[at] = make_float2((float)(g.x * h.x - g.y * h.y), (float)(g.x * h.y + g.y * h.x));
  }
}

__global__ void __launch_bounds__(kThreads, 2)
    k_factor_f32(float2* __restrict__ psi, int L, const double2* __restrict__ lo,
                 const double2* __restrict__ hi) {
  float4 g[16];
#pragma unroll
  for (int m = 0; m < 16; ++m) g[m] = split_pair(lo[2 * threadIdx.x + 512 * (m >> 1) + (m & 1)]);
  const uint32_t chunks = 1u << (L - kBits);
  for (uint32_t k = blockIdx.x; k < chunks; k += gridDim.x) {
    const float4 h = split_pair(hi[k]);
    uint32_t small = 0;  // bit 2 j + q
    float4* p = reinterpret_cast<float4*>(psi + ((uint64_t)k << kBits));
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float o[4];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float4 f = g[2 * j + q];
        o[2 * q] = mul_sub(f.x, f.y, h.x, h.y, f.z, f.w, h.z, h.w);
        o[2 * q + 1] = mul_sub(f.x, f.y, h.z, h.w, -f.z, -f.w, h.x, h.y);
        // trailing parts or errors of the products below FP32's range
        small |= (fmaxf(fabsf(o[2 * q]), fabsf(o[2 * q + 1])) < 0x1p-98f && (f.x != 0.f || f.z != 0.f))
                     ? 1u << (2 * j + q)
                     : 0u;
      }
      p[threadIdx.x + kThreads * j] = make_float4(o[0], o[1], o[2], o[3]);
    }
    if (small && (h.x != 0.f || h.z != 0.f)) factor_small(psi + ((uint64_t)k << kBits), lo, hi[k], small);
  }
}

int grid_of(int L, const LaunchCfg& cfg, int per_sm) {
  return (int)std::min<uint64_t>(1ull << (L - kBits), (uint64_t)cfg.num_sms * per_sm);
}

}  // namespace

bool observe_supported(int precision, int L) { return precision == SV_C64 && L > kBits; }

int observe_energy_pairs(int L, const LaunchCfg& cfg) {
  return ((L - kBits + 7) / 8 + 1) * grid_of(L, cfg, 4);
}

cudaError_t launch_energy_tile(const void* psi, int L, const H0Coef& h, double* part,
                               const LaunchCfg& cfg, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  const int grid = grid_of(L, cfg, 4);
  // the 12 lowest sites; then 8 at a time beside the lowest 4 state bits
  for (int first = 0; first < L && e == cudaSuccess; first += first == 0 ? kBits : 8) {
    EnergyArgs ea;
    TileArgs& ta = ea.ta;
    ta.L = L;
    ta.tb = kBits;
    ea.h0 = h;
    ea.low = ea.diag = first == 0;
    const int win = first == 0 ? 0 : std::min(first, L - 8);  // first window site
    if (first == 0) {
      ta.erun_m[0] = (1u << kBits) - 1;
      ta.run_m[0] = ~0u;
      ta.run_d[0] = kBits;
      for (int q = 0; q < kBits; ++q) ea.cx[q] = (float)h.cx[q];
    } else {
      ta.erun_m[0] = 15;
      ta.erun_m[1] = 0xff0;
      ta.erun_s[1] = (uint8_t)(win - 4);
      ta.run_m[0] = (uint32_t)((1ull << (win - 4)) - 1);
      ta.run_d[0] = 4;
      ta.run_s[1] = (uint8_t)(win - 4);
      ta.run_m[1] = (uint32_t)((1ull << (L - win - 8)) - 1);
      ta.run_d[1] = (uint8_t)(win + 8);
      for (int q = 0; q < 8; ++q)
        if (win + q >= first) ea.cx[4 + q] = (float)h.cx[win + q];
    }
    k_energy_tile<<<grid, kThreads, kTileBytes, s>>>(static_cast<const float2*>(psi), ea, part);
    e = cudaGetLastError();
    part += 2 * grid;
  }
  return e;
}

int observe_moments_grid(int L, const LaunchCfg& cfg) { return grid_of(L, cfg, 2); }

cudaError_t launch_moments_tile(const void* psi, int L, const H0Coef& h, const cd* bonds, double* part, const LaunchCfg& cfg,
                                cudaStream_t s) {
  MomentArgs ma;
  ma.L = L;
  ma.h0 = h;
  for (int i = 0; i < L; ++i) ma.cx[i] = (float)h.cx[i];
  for (int b = 0; bonds && b + 1 < L; ++b)
    for (int k = 0; k < 16; ++k)
      ma.h[b][k] = make_float2((float)bonds[16 * b + k].real(), (float)bonds[16 * b + k].imag());
  const int grid = observe_moments_grid(L, cfg);
  const float2* p = static_cast<const float2*>(psi);
  if (bonds) k_bond_moments_tile<<<grid, kMomentThreads, kTileBytes / 2, s>>>(p, ma, part);
  else k_moments_tile<<<grid, kMomentThreads, kTileBytes, s>>>(p, ma, part);
  return cudaGetLastError();
}

int observe_overlap_grid(int L, const LaunchCfg& cfg) {
  // four quarters of the low indices
  return 4 * (int)std::min<uint64_t>(1ull << (L - kBits), (uint64_t)std::max(1, cfg.num_sms / 4));
}

cudaError_t launch_overlap_f32(const void* psi, int L, const void* lo, const void* hi, double* part,
                               const LaunchCfg& cfg, cudaStream_t s) {
  k_overlap_f32<<<observe_overlap_grid(L, cfg), kOverlapThreads, 0, s>>>(
      static_cast<const float2*>(psi), L, static_cast<const double2*>(lo),
      static_cast<const double2*>(hi), part);
  return cudaGetLastError();
}

cudaError_t launch_factor_f32(void* psi, int L, const void* lo, const void* hi, const LaunchCfg& cfg,
                              cudaStream_t s) {
  k_factor_f32<<<grid_of(L, cfg, 2), kThreads, 0, s>>>(static_cast<float2*>(psi), L,
                                                      static_cast<const double2*>(lo),
                                                      static_cast<const double2*>(hi));
  return cudaGetLastError();
}

}  // namespace fsv
