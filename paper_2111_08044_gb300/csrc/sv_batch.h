// Batched evolution of many independent chains (internal).  Not public.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

#include "sv_internal.h"
#include "sv_kernels.h"
#include "sv_tile.h"

namespace fsv {

constexpr int kResidentMaxL = 14;       // of a batch chain
// Batch chains of k_batch.cu.  While a thread has one group of four amplitudes (up to
// nine sites of 128 threads, ten of 256) they are the faster ones: 16 chains of nine
// sites take 14.7 us a period there and 23.6 us in the resident form, of ten sites
// 20.9 and 25.7, 600 of ten sites 50 and 73 (with two groups a thread 26 against
// 25.5); 256 threads for the shorter ones gain nothing.
constexpr int kShortMaxL = 10;
constexpr int kShortGates = 64;         // its gate tables held in shared memory (16 KiB)
// Of a single chain in the plain form: with 16 blocks one of 15 sites takes 80 us a
// period; tile passes (k_tile.cu) take 106 us at 16 sites and 98 us at 17, over all SMs.
constexpr int kResidentPlainMaxL = 15;
// One round of the resident form: a gate, or two on disjoint sites, on the 16
// amplitudes a thread holds.  off: places of the four register bits (sites b and
// b + 1 of the first gate, then of the second): byte offsets in the block's part
// of the chain, in remote rounds state indices.
struct __align__(16) ResidentRound {
  uint32_t ins[4];   // index bits that move up at each register bit, lowest first (of
                     // the block's part; in remote rounds of the state)
  uint32_t off[4];
  uint8_t count;     // gates
  uint8_t remote;    // a register bit lies beyond the block's part
  uint8_t cluster;   // the round ends at a cluster barrier
  uint8_t sweep;     // 1 + the gate whose sums are taken from the finished round (0: none)
  uint8_t bond[2], epi[2], egroup[2], xorder[2], sbit[4];  // as in TileRound
};
static_assert(sizeof(ResidentRound) == 48, "three 16-byte loads a round");
constexpr int kResidentGates = 96;  // gate tables held at a time (48 KiB)
// One chain of the resident form: state, its period's gate tables (kGateEntries
// complex64 a gate) and rounds, the observable's coefficients, its energy ring
// of (E / (L n), n) pairs.
struct ChainArgs {
  float2* psi = nullptr;
  const float2* gates = nullptr;
  const ResidentRound* rounds = nullptr;
  const int* bonds = nullptr;     // chains of up to kShortMaxL sites
  double* ring = nullptr;
  long long ring_stride = 1;      // pairs from one slot to the next
  long long* counter = nullptr;   // single chain: its period counter
  long long stride = 0;           // per-period table stride (entries; 0: one table)
  int L = 0, ngates = 0, nrounds = 0;
  float Jf = 0.f;
  float cx[kResidentPlainMaxL + 1] = {}, cz[kResidentPlainMaxL + 1] = {};
  EpiParams ep;                   // single chain: diagonal coefficients, renormalisation
};
static_assert(sizeof(ChainArgs) % 4 == 0, "copied in words");

// Blocks (2^kbits, one cluster) and threads a block that hold a chain of L sites;
// a block's rank is state bits pos .. pos + kbits - 1 of its amplitudes.
struct ResidentShape {
  int L = 0, kbits = 0, threads = 32, pos = 0;
  bool local(int q) const { return q < pos || q >= pos + kbits; }
  int place(int q) const { return q < pos ? q : q - kbits; }  // bit of the block's part
};
// plain: the highest sites are spread (its measured sums take sites 0..7 together);
// batch: sites below 9 (its sums take the amplitudes that agree in sites 0..8).
ResidentShape resident_shape(bool plain, int L, int most_blocks);
// The rounds of a period for that shape (one list, any number of gates).
std::vector<ResidentRound> resident_rounds(const std::vector<Gate2>& gates, const ResidentShape& sh);
// Shared memory and cluster size opt-in, at build time; clusters (nullable): how
// many clusters of the shape the device can hold.
cudaError_t resident_prepare(bool plain, const ResidentShape& sh, int ngates, int* clusters);
// `periods` periods of one chain in the plain form; its counter advances.
cudaError_t launch_resident_chain(const ChainArgs& chain, const ResidentShape& sh, int periods,
                                  int ring_len, cudaStream_t s);
// `periods` periods of every chain in chains[0 .. nchains) (device array, all of
// sh.L sites, at most ngates gates a period): energies go to ring slot
// (counter[0] + p) mod ring_len.  periods 0: counter[1] periods.
cudaError_t launch_resident_batch(const ChainArgs* chains, int nchains, const ResidentShape& sh,
                                  int ngates, const long long* counter, int periods, int ring_len,
                                  cudaStream_t s);
// The same for chains of up to kShortMaxL sites (any mix), one block each.
// threads: short_threads of their lengths (one value a launch).
int short_threads(int L);
cudaError_t launch_chain_short(const ChainArgs* chains, int nchains, int threads,
                               const long long* counter, int periods, int ring_len, cudaStream_t s);
cudaError_t short_prepare();
// (energy, norm) of `count` periods from c0 on of each chain into out[chain][count],
// its flag into status[chain].
cudaError_t launch_gather_rings(const RingSource* from, int chains, long long c0, int count,
                                int ring_len, double* out, int* status, cudaStream_t s);
cudaError_t launch_advance(long long* counter, int periods, cudaStream_t s);

// The complex64 tables of a period's gates (kGateEntries each: the rounded gate
// and its residual) into out (sv_api.cu).
void gate_tables(const std::vector<Gate2>& gates, float2* out);
// FP32 copy of a 4x4 unitary, rounded with a one-ulp search that keeps it
// unitary to FP32 resolution (sv_api.cu).
void round_unitary4(const cd* m, float2* out);

}  // namespace fsv
