// Batch chains of two to kShortMaxL sites: one block a chain, its state in shared
// memory for a run of periods, one group of four amplitudes a thread and gate.
//
// A chain that short is a few warps (eight of ten sites), so that the length of a warp's
// chain of instructions per gate bounds it, not the device's rates; the resident
// form of longer chains (two gates on 16 amplitudes a thread) takes fewer
// instructions in all but more in a row.  Tables and coefficients in shared
// memory, the diagonal energies of a thread's amplitudes in registers for the
// run.  16 chains of eight sites: 11.2 us a period of 28 gates, with the tables
// read from L2 and the diagonal energies built every period 12.4 us.
#include <cuda_runtime.h>

#include <cstdint>

#include "sv_batch.h"
#include "sv_device.cuh"

namespace fsv {

namespace {

using namespace dev;

constexpr int kThreads = 128;      // a group of four amplitudes each, up to nine sites
constexpr int kThreadsMost = 256;  // ten sites

template <int T>
__global__ void __launch_bounds__(T)
    k_chain_short(const ChainArgs* __restrict__ chains, const long long* __restrict__ counter,
                  int periods, int ring_len) {
  constexpr int kMaxL = T == kThreads ? kShortMaxL - 1 : kShortMaxL;
  __shared__ float2 sp[1 << kMaxL];
  __shared__ __align__(16) float2 tables[kShortGates * kGateEntries];
  __shared__ int bonds[kShortGates];
  __shared__ ChainArgs ch;
  __shared__ double se[T / 32], sn[T / 32];
  for (uint32_t k = threadIdx.x; k < sizeof(ChainArgs) / 4; k += T)
    reinterpret_cast<uint32_t*>(&ch)[k] = reinterpret_cast<const uint32_t*>(chains + blockIdx.x)[k];
  const long long p0 = counter[0];
  if (periods == 0) periods = (int)counter[1];
  __syncthreads();
  const int L = ch.L;
  const uint32_t n = 1u << L;
  // a period of more gates is read from global memory
  const bool held = ch.ngates <= kShortGates;
  if (held) {
    for (int k = threadIdx.x; k < ch.ngates * (kGateEntries / 2); k += T)
      reinterpret_cast<float4*>(tables)[k] = __ldg(reinterpret_cast<const float4*>(ch.gates) + k);
    for (int k = threadIdx.x; k < ch.ngates; k += T) bonds[k] = __ldg(ch.bonds + k);
  }
  for (uint32_t i = threadIdx.x; i < n; i += T) sp[i] = ch.psi[i];
  __syncthreads();
  // diagonal energy of the thread's amplitudes, site by site
  constexpr int kAmps = (1 << kMaxL) / T;
  float diag[kAmps];
#pragma unroll
  for (int k = 0; k < kAmps; ++k) {
    const uint32_t x = threadIdx.x + k * T;
    float d = 0.f;
    for (int i = 0; i < L; ++i) {
      const float zi = ((x >> i) & 1) ? -1.f : 1.f;
      d += ch.cz[i] * zi;
      if (i + 1 < L) d += ch.Jf * zi * (((x >> (i + 1)) & 1) ? -1.f : 1.f);
    }
    diag[k] = d;
  }
  const uint32_t q = threadIdx.x;
  auto gate = [&](int b, const float4* gs) {
    const uint32_t lowmask = (1u << b) - 1;
    // local index r = 2 b_b + b_{b+1}: offsets of r = 0..3
    const uint32_t o1 = 2u << b, o2 = 1u << b, o3 = 3u << b;
    const uint32_t x = (q & lowmask) | ((q >> b) << (b + 2));
    const float2 v0 = sp[x], v1 = sp[x + o1], v2 = sp[x + o2], v3 = sp[x + o3];
    float2 w[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) w[r] = czero<float2>();
    // residual products first, then the table's on top: a bare first
    // product with a fixed table entry would bias the norm downwards
#pragma unroll
    for (int part = 1; part >= 0; --part) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float4 s = gs[8 * part + 2 * r], t = gs[8 * part + 2 * r + 1];
        w[r] = cmac(w[r], make_float2(s.x, s.y), v0);
        w[r] = cmac(w[r], make_float2(s.z, s.w), v1);
        w[r] = cmac(w[r], make_float2(t.x, t.y), v2);
        w[r] = cmac(w[r], make_float2(t.z, t.w), v3);
      }
    }
    sp[x] = w[0];
    sp[x + o1] = w[1];
    sp[x + o2] = w[2];
    sp[x + o3] = w[3];
  };
  for (int p = 0; p < periods; ++p) {
    for (int g = 0; g < ch.ngates; ++g) {
      if (q < (n >> 2)) {
        if (held) gate(bonds[g], reinterpret_cast<const float4*>(tables + kGateEntries * g));
        else gate(__ldg(ch.bonds + g), reinterpret_cast<const float4*>(ch.gates + kGateEntries * g));
      }
      __syncthreads();
    }
    // <H0> and the norm of the period's final state.  Of ten sites, as in the
    // resident form (k_resident.cu): amplitudes that agree in sites 0..8 are added
    // in ascending order, compensated in FP32
    double e = 0.0, nn = 0.0;
    constexpr int kSums = 512 / T;
#pragma unroll
    for (int k = 0; k < kSums; ++k) {
      float es = 0.f, ec = 0.f, ns = 0.f, nc = 0.f;
#pragma unroll
      for (int m = k; m < kAmps; m += kSums) {
        const uint32_t x = threadIdx.x + m * T;
        if (x >= n) break;
        const float2 v = sp[x];
        const float pr = cabs2(v);
        float ex = 0.f;
#pragma unroll
        for (int i = 0; i < kMaxL; ++i)
          if (i < L && !((x >> i) & 1)) ex += 2.f * ch.cx[i] * cdotre(v, sp[x | (1u << i)]);
        if constexpr (kSums == kAmps) {
          e += (double)(pr * diag[m] + ex);
          nn += (double)pr;
        } else {
          const float ye = __fsub_rn(__fmaf_rn(pr, diag[m], ex), ec), te = __fadd_rn(es, ye);
          ec = __fsub_rn(__fsub_rn(te, es), ye);
          es = te;
          const float yn = __fsub_rn(pr, nc), tn = __fadd_rn(ns, yn);
          nc = __fsub_rn(__fsub_rn(tn, ns), yn);
          ns = tn;
        }
      }
      if constexpr (kSums != kAmps) {
        e += (double)es - (double)ec;
        nn += (double)ns - (double)nc;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      e += __shfl_xor_sync(0xffffffffu, e, o);
      nn += __shfl_xor_sync(0xffffffffu, nn, o);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) {
      se[w] = e;
      sn[w] = nn;
    }
    __syncthreads();
    if (threadIdx.x == T - 32) {  // its warp has no gates in chains below nine sites
      double te = 0.0, tn = 0.0;
      for (int k = 0; k < T / 32; ++k) {
        te += se[k];
        tn += sn[k];
      }
      const long long slot = (p0 + p) % ring_len;
      double* const out = ch.ring + 2 * slot * ch.ring_stride;
      out[0] = te / ((double)L * tn);
      out[1] = tn;
    }
  }
  for (uint32_t i = threadIdx.x; i < n; i += T) ch.psi[i] = sp[i];
}

// Ring slots of periods c0 .. c0 + count - 1 of each chain, and its flag: one block
// a chain.
__global__ void k_gather_rings(const RingSource* __restrict__ from, long long c0, int count,
                               int ring_len, double2* __restrict__ out, int* __restrict__ status) {
  const RingSource src = from[blockIdx.x];
  const double2* ring = reinterpret_cast<const double2*>(src.ring);
  for (int q = threadIdx.x; q < count; q += blockDim.x)
    out[(size_t)blockIdx.x * count + q] = ring[(c0 + q) % ring_len];
  if (threadIdx.x == 0) status[blockIdx.x] = src.status ? *src.status : 0;
}

}  // namespace

cudaError_t launch_gather_rings(const RingSource* from, int chains, long long c0, int count,
                                int ring_len, double* out, int* status, cudaStream_t s) {
  k_gather_rings<<<chains, 128, 0, s>>>(from, c0, count, ring_len, reinterpret_cast<double2*>(out), status);
  return cudaGetLastError();
}

cudaError_t short_prepare() {
  // the carve-out of the resident form's blocks, so that both share an SM
  cudaError_t e = cudaFuncSetAttribute(k_chain_short<kThreads>,
                                       cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_chain_short<kThreadsMost>,
                             cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  return e;
}

int short_threads(int L) { return L < kShortMaxL ? kThreads : kThreadsMost; }

cudaError_t launch_chain_short(const ChainArgs* chains, int nchains, int threads,
                               const long long* counter, int periods, int ring_len, cudaStream_t s) {
  if (nchains <= 0) return cudaSuccess;
  if (threads == kThreads)
    k_chain_short<kThreads><<<nchains, kThreads, 0, s>>>(chains, counter, periods, ring_len);
  else
    k_chain_short<kThreadsMost>
        <<<nchains, kThreadsMost, 0, s>>>(chains, counter, periods, ring_len);
  return cudaGetLastError();
}

}  // namespace fsv
