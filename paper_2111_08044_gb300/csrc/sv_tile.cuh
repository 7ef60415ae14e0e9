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
  __device__ __forceinline__ void flush(double& acc) {
    acc += (double)hi + (double)lo;
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

}  // namespace dev
}  // namespace fsv
