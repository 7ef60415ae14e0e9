// Plan of the plain form's tile passes (host).
//
// The gates of a period are applied in the order given, so every amplitude
// sees the same operations, in the same order, as one pass per gate would
// apply: only the number of passes over the state changes.  A pass takes
// consecutive gates while their sites fit in a tile of 2^tb amplitudes
// beside the lowest state bits (whole memory lines).
#include <algorithm>
#include <cstring>

#include "sv_batch.h"
#include "sv_tile.h"

namespace fsv {

namespace {

// lowest state bits in every tile: 128-byte (complex64) or 64-byte lines
int line_bits(int precision) { return precision == SV_C64 ? 4 : 2; }

// the per-gate kernels' grouping of a measured gate's partial sums
int energy_group(int L, int precision, int bond, int epi) {
  if (!epi) return 0;
  if (precision != SV_C64 || L < 8) return TILE_E_GROUP;
  return bond < 6 ? TILE_E_SWEEP : TILE_E_PAIR;
}

// The per-gate kernels sum a row's products in the order of its columns,
// except on bonds that pair amplitudes inside a warp's span, where row r takes
// column r ^ j at step j.
bool xor_order(int L, int precision, int bond) {
  const int lv = precision == SV_C64 ? 1 : 0;
  return L >= lv + 7 && bond < lv + 5;
}

// runs of consecutive set bits
int bit_runs(uint64_t m) { return __builtin_popcountll(m & ~(m << 1)); }

}  // namespace

int tile_threads(int precision, int tb) {
  const int t = precision == SV_C64 ? 1 << (tb - 4) : precision == SV_DF64 ? 1 << (tb - 2) : 1 << tb;
  return std::max(32, t);
}

// Gates [at, end) of one pass in a tile of 2^tb amplitudes and its state bits
// before filling up (end = at: the tile is too small for the gate).
static int pass_end(int L, const std::vector<Gate2>& gates, int precision, int tb, int at,
                    int max_gates, uint64_t* bits) {
  const int ng = (int)gates.size(), first = at;
  uint64_t set = (1ull << std::min(line_bits(precision), L)) - 1;
  while (at < ng && at - first < max_gates) {
    const Gate2& g = gates[at];
    uint64_t need = set | (3ull << g.bond);
    if (energy_group(L, precision, g.bond, g.epi) == TILE_E_SWEEP) need |= 0xff;
    if (__builtin_popcountll(need) > tb || bit_runs(need) > kTileRuns - 1) break;
    set = need;
    ++at;
  }
  *bits = set;
  return at;
}

static int most_gates(int precision) { return precision == SV_C64 ? kTileTabSlots : kTileMaxGates; }

std::vector<TilePassPlan> tile_plan(int L, const std::vector<Gate2>& gates, int precision, int tb,
                                    int max_gates) {
  if (max_gates == 0) max_gates = most_gates(precision);
  std::vector<TilePassPlan> out;
  const int ng = (int)gates.size();
  int at = 0;
  while (at < ng) {
    TilePassPlan p;
    uint64_t set = 0;
    const int end = pass_end(L, gates, precision, tb, at, max_gates, &set);
    while (at < end) p.gates.push_back(at++);
    if (p.gates.empty()) return {};  // a tile too small for one gate
    for (int q = 0; __builtin_popcountll(set) < tb; ++q) set |= 1ull << q;  // lowest free bits
    std::vector<int> where(L, -1);
    for (int q = 0; q < L; ++q)
      if ((set >> q) & 1) {
        where[q] = (int)p.bits.size();
        p.bits.push_back(q);
      }
    for (size_t i = 0; i < p.gates.size();) {
      TileRound r;
      std::memset(&r, 0, sizeof(r));
      const Gate2& a = gates[p.gates[i]];
      std::vector<int> reg = {where[a.bond], where[a.bond + 1]};
      const int ea = energy_group(L, precision, a.bond, a.epi);
      r.gate[0] = (uint8_t)i;
      r.count = 1;
      r.bond[0] = (uint8_t)a.bond;
      r.epi[0] = (uint8_t)a.epi;
      r.egroup[0] = (uint8_t)ea;
      size_t next = i + 1;
      if (precision == SV_C64) {
        // a second gate: on other sites, the first gate's sums not taken from
        // the finished round, and bit 0 left to the lanes where a sum pairs it
        if (next < p.gates.size()) {
          const Gate2& b = gates[p.gates[next]];
          const int eb = energy_group(L, precision, b.bond, b.epi);
          const bool apart = b.bond > a.bond + 1 || a.bond > b.bond + 1;
          const bool bit0 = (ea == TILE_E_PAIR && b.bond == 0) || (eb == TILE_E_PAIR && a.bond == 0);
          if (apart && ea != TILE_E_SWEEP && !bit0) {
            reg.push_back(where[b.bond]);
            reg.push_back(where[b.bond + 1]);
            r.gate[1] = (uint8_t)next;
            r.count = 2;
            r.bond[1] = (uint8_t)b.bond;
            r.epi[1] = (uint8_t)b.epi;
            r.egroup[1] = (uint8_t)eb;
            ++next;
          }
        }
        // a lone gate: the tile bits above it (or the highest below it), not
        // bit 0 where a sum pairs it
        for (int q = where[a.bond + 1] + 1; reg.size() < 4 && q < tb; ++q) reg.push_back(q);
        for (int q = where[a.bond] - 1; reg.size() < 4; --q) reg.push_back(q);
      }
      std::vector<int> sorted = reg;
      std::sort(sorted.begin(), sorted.end());
      for (size_t k = 0; k < reg.size(); ++k) {
        const uint32_t one = 1u << reg[k];
        r.slot[k] = (uint16_t)(precision == SV_C64 ? tile_byte8(one) : tile_slot16(one));
        r.sbit[k] = (uint8_t)p.bits[reg[k]];
        r.ins[k] = (uint16_t)(0xffffu << sorted[k]);
      }
      for (int k = 0; k < r.count; ++k)
        r.xorder[k] = xor_order(L, precision, r.bond[k]) ? 1 : 0;
      p.measures = p.measures || r.epi[0] || r.epi[1];
      p.rounds.push_back(r);
      i = next;
    }
    // the state is written from the last round itself where its lanes cover at
    // least 64 bytes of each line
    const TileRound& last = p.rounds.back();
    p.direct_out = precision != SV_C128;
    for (int k = 0; k < (precision == SV_C64 ? 4 : 2); ++k)
      if (last.sbit[k] < (precision == SV_C64 ? 3 : 2)) p.direct_out = false;
    for (int k = 0; k < 2; ++k)
      if (last.egroup[k] == TILE_E_SWEEP) p.direct_out = false;
    out.push_back(std::move(p));
  }
  return out;
}

int tile_bits(int L, int precision, const LaunchCfg& cfg) {
  const int num_sms = cfg.num_sms;
  if (L < 5) return 0;
  // Double-float: a chain that one tile holds stays in one block (10 sites 67 us a
  // period, 98 in tiles of 2^9); else tiles of 2^10, eight warps each, where they
  // leave most SMs one (21 sites 1.40 ms a period, 1.44 in tiles of 2^9, 1.58 of
  // 2^8), and of 2^9 below (13 sites 119 us; 137 in tiles of 2^10, 123 of 2^8).
  if (precision == SV_DF64) return std::min(L, L <= 10 || (4ll << (L - 10)) >= 3ll * num_sms ? 10 : 9);
  // complex128: one block up to 8 sites (42 us a period, 52 in tiles of 2^7; 9 sites
  // 70 and 61); then FP64 work against launches: 13 sites 100 us in tiles of 2^7, 105
  // of 2^6, 115 of 2^8; 21 sites 5.03 ms of 2^8, 5.07 of 2^7, 5.21 of 2^9.
  if (precision == SV_C128) return L <= 8 ? L : L < 15 ? 7 : 8;
  // complex64 (chains too long for the resident form): tiles of 2^12 where they leave
  // most SMs one (21 sites 307 us a period, 330 in tiles of 2^11; 24 sites 2.12 and
  // 2.17 ms), of 2^11 below (16 sites 86 us, 104 in tiles of 2^12, 88 of 2^10) unless
  // other chains' passes fill the rest (12 chains of 16 to 18 sites, 32 periods: 7.5 ms
  // and 9.4 ms in tiles of 2^11).
  // A chain that the tile would hold (where the resident form finds no room on the
  // device) takes one launch a gate: complex64 passes run one period.
  const int tb = !cfg.alone() || (4ll << L) >= 3ll * num_sms << 12 ? 12 : 11;
  return L > tb ? tb : 0;
}

std::vector<ResidentRound> resident_rounds(const std::vector<Gate2>& gates, const ResidentShape& sh) {
  std::vector<ResidentRound> out;
  // rounds do not reach across the tables held at a time
  for (size_t at = 0; at < gates.size(); at += kResidentGates) {
    const std::vector<Gate2> part(gates.begin() + at,
                                  gates.begin() + std::min(gates.size(), at + kResidentGates));
    const auto plan = tile_plan(sh.L, part, SV_C64, sh.L, kResidentGates);
    if (plan.size() != 1) return {};
    for (const TileRound& r : plan[0].rounds) {
      ResidentRound o;
      std::memset(&o, 0, sizeof(o));
      int bits[4];
      for (int k = 0; k < 4; ++k) {
        o.sbit[k] = r.sbit[k];
        o.remote |= sh.local(r.sbit[k]) ? 0 : 1;
      }
      for (int k = 0; k < 4; ++k) {
        bits[k] = o.remote ? r.sbit[k] : sh.place(r.sbit[k]);
        o.off[k] = o.remote ? 1u << bits[k] : tile_byte8(1u << bits[k]);
      }
      std::sort(bits, bits + 4);
      for (int k = 0; k < 4; ++k) o.ins[k] = ~0u << bits[k];
      o.count = r.count;
      for (int k = 0; k < 2; ++k) {
        o.bond[k] = r.bond[k];
        o.epi[k] = r.epi[k];
        o.egroup[k] = r.egroup[k];
        o.xorder[k] = r.xorder[k];
        if (r.egroup[k] == TILE_E_SWEEP) o.sweep = (uint8_t)(k + 1);
      }
      out.push_back(o);
    }
  }
  for (size_t k = 0; k < out.size(); ++k)
    out[k].cluster = out[k].remote || out[(k + 1) % out.size()].remote ? 1 : 0;
  return out;
}

}  // namespace fsv
