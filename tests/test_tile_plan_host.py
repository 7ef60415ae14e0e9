"""Host plans of the tile passes and of the chains in shared memory, compiled from
their sources: every length, type and device size gets tiles that fit the chain and
passes that apply each gate once, in order."""
import os
import shutil
import subprocess

import pytest

from paper_2111_08044_gb300 import build as b

_MAIN = r"""
#include <algorithm>
#include <cstdio>
#include <vector>
#include "sv_batch.h"
using namespace fsv;

static int failures = 0;
#define CHECK(c, ...)                              \
  do {                                             \
    if (!(c) && ++failures < 20) {                 \
      std::printf("%s: ", #c);                     \
      std::printf(__VA_ARGS__);                    \
      std::printf("\n");                           \
    }                                              \
  } while (0)

static std::vector<Gate2> gates(int L, int K, int first) {
  sv_floquet_params p{};
  p.J = 1; p.hx = 0.9; p.hz = 0.4; p.T = 0.5; p.theta = 0.3;
  p.edge_field_weight = 0.5; p.K = K; p.first_layer = first;
  return period_gates(L, p, p.theta, p.hx);
}

int main() {
  for (int precision : {SV_C64, SV_C128, SV_DF64})
    for (int L = 2; L <= 34; ++L)
      for (int sms : {1, 16, 132, 152, 300})
        for (int alone = 0; alone < 2; ++alone) {
          LaunchCfg cfg;
          cfg.num_sms = sms;
          cfg.min_tiles_per_cta = alone ? 0 : 4;
          const int tb = tile_bits(L, precision, cfg);
          // complex64 passes have no loop over periods: more than one tile
          CHECK(tb == 0 || (precision == SV_C64 ? tb < L : tb <= L), "type %d L %d tb %d", precision, L, tb);
          if (tb == 0 || tb > L) continue;
          for (int first = 0; first < 2; ++first) {
            const auto g = gates(L, 2, first);
            size_t at = 0;
            for (const auto& p : tile_plan(L, g, precision, tb)) {
              CHECK((int)p.bits.size() == tb && p.bits.back() < L && std::is_sorted(p.bits.begin(), p.bits.end()),
                    "type %d L %d tb %d", precision, L, tb);
              for (int k : p.gates) CHECK(k == (int)at++, "type %d L %d", precision, L);
              int in_rounds = 0;
              for (const auto& r : p.rounds) in_rounds += r.count;
              CHECK(in_rounds == (int)p.gates.size(), "type %d L %d", precision, L);
            }
            CHECK(at == g.size(), "type %d L %d first %d: %zu of %zu gates", precision, L, first, at, g.size());
          }
        }
  for (int L = 5; L <= kResidentPlainMaxL; ++L)
    for (int K = 1; K <= 130; ++K)
      for (int first = 0; first < 2; ++first) {
        const auto g = gates(L, K, first);
        for (int kbits = 0; kbits <= 4 && L - kbits >= 5; ++kbits)
          for (int pos : {L - kbits, std::min(L, 9) - kbits}) {
            ResidentShape sh;
            sh.L = L;
            sh.kbits = kbits;
            sh.pos = pos;
            size_t n = 0;
            for (const auto& r : resident_rounds(g, sh)) n += r.count;
            CHECK(n == g.size(), "L %d K %d first %d kbits %d: %zu of %zu gates", L, K, first, kbits, n, g.size());
          }
      }
  std::printf("%d failures\n", failures);
  return failures != 0;
}
"""


def test_plans_fit_the_chain(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(b._nvcc()))), "include")
    src, exe = tmp_path / "plans.cpp", tmp_path / "plans"
    src.write_text(_MAIN)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", b.CSRC, "-I", b.INCLUDE, "-I", cuda, str(src),
                    os.path.join(b.CSRC, "host_tile.cpp"), os.path.join(b.CSRC, "host_model.cpp"),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
