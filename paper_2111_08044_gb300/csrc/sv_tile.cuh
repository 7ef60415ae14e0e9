// Device helpers of the tile kernels: the state's layout of a tile, its copies
// to and from shared memory, packed FP32 arithmetic, partial sums.
#pragma once

#include "sv_device.cuh"
#include "sv_tile.h"

namespace fsv {
namespace dev {

__device__ __forceinline__ uint64_t tile_base(const TileArgs& ta, uint32_t t) {
  uint64_t x = 0;
#pragma unroll
  for (int k = 0; k < kTileRuns; ++k)
    x |= (uint64_t)((t >> ta.run_s[k]) & ta.run_m[k]) << ta.run_d[k];
  return x;
}
// state offset of tile index e
__device__ __forceinline__ uint64_t elem_state(const TileArgs& ta, uint32_t e) {
  uint64_t x = 0;
#pragma unroll
  for (int k = 0; k < kTileRuns; ++k) x |= (uint64_t)(e & ta.erun_m[k]) << ta.erun_s[k];
  return x;
}
// tile index of a thread: zeros inserted at the round's N register bits
template <int N>
__device__ __forceinline__ uint32_t thread_elem(const TileRound& rd, uint32_t tid) {
  uint32_t e = tid;
#pragma unroll
  for (int k = 0; k < N; ++k) e += e & rd.ins[k];
  return e;
}

// packed pairs of FP32 values: each half is the scalar operation
__device__ __forceinline__ uint64_t pk2(float x, float y) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 un2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// leading part of a + b and its error
__device__ __forceinline__ uint64_t two_sum2(uint64_t a, uint64_t b, uint64_t& err) {
  const uint64_t s = add2(a, b), bb = sub2(s, a);
  err = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
  return s;
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// A tile's partial sums as an unevaluated sum hi + lo of FP32 values (each
// addition exact in hi plus its rounding error), moved to FP64 once a tile: an
// FP64 addition and conversion per sum instead held the measuring passes at
// twice their arithmetic (the FP64 units take 16 cycles a warp instruction).
struct FloatSum {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float v) {
    const df s = two_sum(hi, v);
    hi = s.hi;
    lo = __fadd_rn(lo, s.lo);
  }
  // (an infinite hi is the sum, its rounding errors are NaN)
  __device__ __forceinline__ void flush(double& acc) {
    acc += (double)hi + (double)(lo == lo ? lo : 0.f);
    hi = lo = 0.f;
  }
};

// The tile between the state and shared memory in 16-byte pieces (two
// amplitudes), consecutive threads on consecutive pieces of a line.  Tiles of
// at least 2^9 amplitudes are eight pieces a thread: their offsets from the
// thread's first are the pass's.
struct TileIo {
  uint32_t s0;   // shared-memory byte offset of the thread's first piece
  uint64_t x0;   // its state offset within the tile
  uint32_t s[3]; // of the piece-index bits above the thread's
  uint64_t x[3];
};
__device__ __forceinline__ TileIo tile_io(const TileArgs& ta) {
  TileIo io;
  const uint32_t e = 2 * threadIdx.x;
  io.s0 = tile_byte8(e);
  io.x0 = elem_state(ta, e);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const uint32_t b = 1u << (ta.tb - 3 + j);
    io.s[j] = tile_byte8(b);
    io.x[j] = elem_state(ta, b);
  }
  return io;
}
__device__ __forceinline__ void load_tile(const TileArgs& ta, const TileIo& io, uint32_t tile,
                                          const float2* psi) {
  if (ta.tb >= 9) {
#pragma unroll
    for (int m = 0; m < 8; ++m)
      cp_async16(tile + io.s0 + ((m & 1) ? io.s[0] : 0) + ((m & 2) ? io.s[1] : 0) + ((m & 4) ? io.s[2] : 0),
                 psi + io.x0 + ((m & 1) ? io.x[0] : 0) + ((m & 2) ? io.x[1] : 0) + ((m & 4) ? io.x[2] : 0));
  } else {
    for (uint32_t e = 2 * threadIdx.x; e < (1u << ta.tb); e += 2 * blockDim.x)
      cp_async16(tile + tile_byte8(e), psi + elem_state(ta, e));
  }
  cp_commit();
}
__device__ __forceinline__ void store_tile(const TileArgs& ta, const TileIo& io, const uint8_t* tile,
                                           float2* psi) {
  if (ta.tb >= 9) {
#pragma unroll
    for (int m = 0; m < 8; ++m)
      *reinterpret_cast<float4*>(psi + io.x0 + ((m & 1) ? io.x[0] : 0) + ((m & 2) ? io.x[1] : 0) +
                                 ((m & 4) ? io.x[2] : 0)) =
          *reinterpret_cast<const float4*>(tile + io.s0 + ((m & 1) ? io.s[0] : 0) +
                                           ((m & 2) ? io.s[1] : 0) + ((m & 4) ? io.s[2] : 0));
  } else {
    for (uint32_t e = 2 * threadIdx.x; e < (1u << ta.tb); e += 2 * blockDim.x)
      *reinterpret_cast<float4*>(psi + elem_state(ta, e)) =
          *reinterpret_cast<const float4*>(tile + tile_byte8(e));
  }
}

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

template <int J0, int J1, int K0, int K1, typename Round>
__device__ __forceinline__ void measure16(const uint64_t (&v)[16], int L, const float* cx,
                                          const EpiParams& ep, const Round& rd, int which,
                                          uint64_t x0, bool active, FloatSum& esum,
                                          FloatSum& nsum) {
  const int epi = rd.epi[which], bond = rd.bond[which];
  const float cxh = cx[bond], cxl = cx[bond + 1];
  Diag<float> dg;
  if (epi & EPI_DIAG) dg.init(ep, L);
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

// The same of a gate that measures <X> only, in neighbouring pairs (TILE_E_PAIR): a
// term that is not measured has the coefficient 0.
template <int J0, int J1, int K0, int K1, typename Round>
__device__ __forceinline__ void measure16_x(const uint64_t (&v)[16], const float* cx, const Round& rd,
                                            int which, bool active, FloatSum& esum) {
  const int epi = rd.epi[which], bond = rd.bond[which];
  const float ch = (epi & EPI_X_HI) ? cx[bond] * 2.f : 0.f;
  const float cl = (epi & EPI_X_LO) ? cx[bond + 1] * 2.f : 0.f;
  const bool take = active && (threadIdx.x & 1);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float2 w[4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
      w[r] = un2(v[((r >> 1) << J0) | ((r & 1) << J1) | ((k & 1) << K0) | ((k >> 1) << K1)]);
    const float hi = cdotre(w[0], w[2]) + cdotre(w[1], w[3]);
    const float lo = cdotre(w[0], w[1]) + cdotre(w[2], w[3]);
    const float es = __fmaf_rn(cl, lo, __fmaf_rn(ch, hi, 0.f));
    const float e2 = __shfl_xor_sync(0xffffffffu, es, 1);
    const float s = __fmaf_rn(cl, lo, __fmaf_rn(ch, hi, e2));
    if (take) esum.add(s);
  }
}

// A measured gate on bonds 0..5 of a chain of at least 8 sites, from the tile:
// the sums of the per-gate kernel, whose threads hold bits 0, 6 and 7.
// state(e): state index of tile index e; 2^tb amplitudes in the tile.
template <bool kDiag = true, typename S>
__device__ __forceinline__ void measure_sweep(const uint8_t* tile, int tb, int L, const float* cx,
                                              const EpiParams& ep, int bond, int epi, const S& state,
                                              FloatSum& esum, FloatSum& nsum) {
  const float cxh = cx[bond], cxl = cx[bond + 1];
  Diag<float> dg;
  if (kDiag && (epi & EPI_DIAG)) dg.init(ep, L);
  const uint32_t nv = 1u << (tb - 3);
  // amplitudes e and e + 1 (e even)
  auto at = [&](uint32_t e) { return *reinterpret_cast<const float4*>(tile + tile_byte8(e)); };
  for (uint32_t vt = threadIdx.x; vt < nv; vt += blockDim.x) {
    const uint32_t e0 = ((vt & 31u) << 1) | ((vt >> 5) << 8);
    float2 w[4][2];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float4 q = at(e0 | (c << 6));
      w[c][0] = make_float2(q.x, q.y);
      w[c][1] = make_float2(q.z, q.w);
    }
    float es = 0.f, ns = 0.f;
    // sum over the thread's amplitudes of the products with site bit `flip` flipped
    auto pairs = [&](uint32_t flip) {
      float s = 0.f;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float2 u[2] = {w[c][1], w[c][0]};
        if (flip > 1) {
          const float4 q = at((e0 | (c << 6)) ^ flip);
          u[0] = make_float2(q.x, q.y);
          u[1] = make_float2(q.z, q.w);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) s += cdotre(w[c][k], u[k]);
      }
      return s;
    };
    if (epi & EPI_X_HI) es += cxh * pairs(1u << bond);
    if (epi & EPI_X_LO) es += cxl * pairs(2u << bond);
    if (kDiag && (epi & EPI_DIAG)) {
      const uint64_t x0 = state(e0);
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
    if (kDiag && (epi & EPI_DIAG)) nsum.add(ns);
  }
}

}  // namespace dev
}  // namespace fsv
