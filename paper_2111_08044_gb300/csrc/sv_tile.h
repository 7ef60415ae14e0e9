// Tile passes of the plain form: consecutive gates of the period applied to
// tiles of the state, in the period's own order (host plan and launch).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "sv_internal.h"
#include "sv_kernels.h"

namespace fsv {

constexpr int kTileMaxBits = 12;   // largest tile: 2^12 complex64 amplitudes (32 KiB)
constexpr int kTileTabSlots = 8;   // gates and rounds of a complex64 pass
constexpr int kTileMaxGates = 96;  // gates of a pass of the wider types
constexpr int kTileRuns = 4;  // runs of consecutive state bits inside, and outside, a tile

// How a round's measured gate sums its energy terms (the FP32 grouping of
// the per-gate kernels, which fixes the rounding of the partial sums).
enum : int {
  TILE_E_GROUP = 1,  // one sum per four amplitudes
  TILE_E_PAIR = 2,   // complex64: two neighbouring amplitudes (bit 0) share a sum
  TILE_E_SWEEP = 3,  // complex64, bonds 0..5: sums over bits 0, 6 and 7, after the round
};

// One round: a gate, or two gates on disjoint sites one after the other, on
// the amplitudes that a thread holds.  The thread's tile index is its number
// with a zero inserted at each register bit, lowest first.
struct __align__(16) TileRound {
  uint8_t gate[2];    // slots of the gates in the pass's table
  uint8_t bond[2];
  uint8_t epi[2];     // EPI_* of each gate
  uint8_t egroup[2];  // TILE_E_* of each measured gate
  uint16_t ins[4];    // index bits that move up at each insertion
  uint16_t slot[4];   // place of each register bit (tile_byte8 or tile_slot16): sites
                      // b and b + 1 of the first gate, then of the second
  uint8_t sbit[4];    // their state bits
  uint8_t xorder[2];  // each gate's products in the order r ^ j (see tile_plan)
  uint8_t count;      // gates of the round
  uint8_t pad;
};
static_assert(sizeof(TileRound) == 32, "two 16-byte loads a round");

// Place of tile index e in shared memory.  complex64: byte offset, rows of 16
// amplitudes (a 128-byte line) 144 bytes apart, so that lanes on different rows
// meet different banks; additive over the bits of e.  16-byte amplitudes: slot
// number, low index bits XORed with bits above them; linear over XOR.
__host__ __device__ inline uint32_t tile_byte8(uint32_t e) { return 8 * e + 16 * (e >> 4); }
__host__ __device__ inline uint32_t tile_slot16(uint32_t e) {
  return e ^ ((e >> 2) & 2u) ^ (((e >> 4) & 1u) * 5u) ^ ((e >> 3) & 4u);
}

struct TilePassPlan {
  std::vector<int> bits;   // state bits of the tile, ascending; bit q of a tile index
  std::vector<int> gates;  // indices into the period's gate list, consecutive
  std::vector<TileRound> rounds;
  bool measures = false;
  bool direct_out = false;  // the last round writes the state
};

// The passes of a period in tiles of 2^tb amplitudes (tb >= 4, tb <= L).
// Gates are taken in the order given; a pass ends where the next gate's
// sites no longer fit beside the pass's.  complex64: up to two gates a round.
// max_gates: gates of a pass (0: the type's).
std::vector<TilePassPlan> tile_plan(int L, const std::vector<Gate2>& gates, int precision, int tb,
                                    int max_gates = 0);
// Tile size for a chain (0: the chain is too short for tiles).
int tile_bits(int L, int precision, const LaunchCfg& cfg);
int tile_threads(int precision, int tb);

// A complex64 table entry g as the operands of packed FMAs: (gx, gx) and
// (-gy, gy).
struct __align__(16) PackedEntry {
  float re[2], im[2];
};
// Gate tables and rounds as kernel parameters (complex64): read through the
// constant bank, a table entry is a uniform FMA operand that costs no load and
// no register.
template <int kSlots>
struct TileTabOf {
  PackedEntry g[kSlots][kGateEntries];
  TileRound r[kSlots];
};
using TileTab = TileTabOf<kTileTabSlots>;

// A double-float table entry as packed operands (df_entry): (re, re) and
// (-im, im) leading parts, their negatives, the trailing parts negated.
struct EntryDf {
  uint64_t re, nre, nre_lo, im, nim, nim_lo;
};
// entry (re hi, re lo, im hi, im lo)
__host__ __device__ inline EntryDf df_entry(float4 g) {
  auto pair = [](float x, float y) {
    union {
      float f[2];
      uint64_t u;
    } p = {{x, y}};
    return p.u;
  };
  return EntryDf{pair(g.x, g.x),  pair(-g.x, -g.x), pair(-g.y, -g.y),
                 pair(-g.z, g.z), pair(g.z, -g.z),  pair(g.w, -g.w)};
}
template <int kSlots>
struct TileTabDf {
  EntryDf g[kSlots][16];
  TileRound r[kSlots];
};

struct TileArgs {
  int L = 0, tb = 0;
  int ngates = 0, nrounds = 0;
  int direct_out = 0;
  int first = 0;                   // the period's first pass (folded renormalisation)
  int buffers = 1;                 // tile buffers (2: the next tile loads during this one)
  int overlap = 0;                 // launched while the pass before still runs
  uint32_t smem = 0;               // dynamic shared memory
  // state bits of the tile index, in runs: (e & m) << s
  uint8_t erun_s[kTileRuns] = {};
  uint16_t erun_m[kTileRuns] = {};
  // the state bits outside the tile, from the tile number: ((t >> s) & m) << d
  uint8_t run_s[kTileRuns] = {}, run_d[kTileRuns] = {};
  uint32_t run_m[kTileRuns] = {};
  const TileRound* rounds = nullptr;  // device
  const void* gates = nullptr;        // device: the pass's first gate table
  int in_params = 0;                  // tables and rounds in the parameters
  int any_xorder = 0, any_epi = 0;    // over the pass's gates
  long long stride = 0;               // per-period table stride (entries; 0: one table)
  const long long* counter = nullptr;
  float cx[34] = {};                  // complex64: <X> coefficients (measured gates)
  double cx64[34] = {};               // the wider types'
  EpiParams ep;                       // diagonal coefficients, renormalisation, partials
  // a whole period in one pass on one tile: `periods` periods in one launch,
  // each period's energy and norm written to the ring, the counter advanced
  int periods = 0;
  double* ring = nullptr;
  int ring_len = 0;
  long long* counter_rw = nullptr;
};

// grid of a pass (also its number of partial pairs), its tile buffers and shared
// memory; opts
// its kernel into the shared memory it needs (at build time, outside a capture)
cudaError_t tile_grid(int precision, TileArgs* ta, const LaunchCfg& cfg, int* grid);
// tab, tab_df: the pass's tables and rounds on the host (in_params; else unused)
cudaError_t launch_tile(int precision, void* psi, const TileArgs& ta, const TileTab* tab,
                        const TileTabDf<kTileTabSlots>* tab_df, int grid, cudaStream_t s);

// ------------------------------------------------------------ adjoint sweep
// A pass of the reverse sweep on tiles of psi and lambda (complex64): operations
// [0, nkick) of the pass differentiate the kick angle, the others the field.
constexpr int kAdjointTileBits = 11;  // both states of a tile: 36 KiB
struct AdjointPass {
  TileArgs ta;
  int nkick = 0;
  int pair_at = 0;  // its partial pairs (kick, field) within the period's
};
cudaError_t adjoint_tile_grid(AdjointPass* ap, const LaunchCfg& cfg, int* grid);
// tab: odag (16 entries) and d (16) per operation, and the rounds
cudaError_t launch_adjoint_tile(void* psi, void* lam, const AdjointPass& ap,
                                const TileTab& tab, double* part, int grid, cudaStream_t s);
// out[2 k], out[2 k + 1] = 2 x the sums of period k's (kick, field) partial
// pairs, periods `pairs` pairs apart, fixed order
cudaError_t launch_grad_reduce_pairs(const double* part, int pairs, int periods, double* out,
                                     cudaStream_t s);

}  // namespace fsv
