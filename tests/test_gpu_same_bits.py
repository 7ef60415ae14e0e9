"""The plain form's tile passes and chains in shared memory against one pass per gate:
the same state bit for bit (complex64 and complex128).  Evolutions of these lengths no
longer take the per-gate passes, so a small library calls them."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2111_08044_gb300 import build as b
from paper_2111_08044_gb300 import capi, inputs

pytestmark = pytest.mark.gpu

_CODE = r"""
#include <vector>
#include "sv_batch.h"
#include "sv_kernels.h"
using namespace fsv;
// one period of *p on the state, one launch a gate; 0 on success
extern "C" int per_gate_period(int precision, void* psi, int L, const sv_floquet_params* p, double theta,
                               double hx) {
  const auto gates = period_gates(L, *p, theta, hx);
  const size_t n = gates.size() * kGateEntries;
  std::vector<float2> t32(n);
  std::vector<double2> t64(n, make_double2(0, 0));
  gate_tables(gates, t32.data());
  for (size_t g = 0; g < gates.size(); ++g)
    for (int e = 0; e < 16; ++e)
      t64[g * kGateEntries + e] = make_double2(gates[g].m[e].real(), gates[g].m[e].imag());
  const size_t entry = precision == SV_C64 ? sizeof(float2) : sizeof(double2);
  LaunchCfg cfg;
  cudaDeviceGetAttribute(&cfg.num_sms, cudaDevAttrMultiProcessorCount, 0);
  char* tab = nullptr;
  long long* counter = nullptr;
  double* part = nullptr;
  int bad = cudaMalloc(&tab, n * entry) || cudaMalloc(&counter, 8) || cudaMalloc(&part, 64 * cfg.num_sms);
  bad = bad || cudaMemcpy(tab, precision == SV_C64 ? (void*)t32.data() : (void*)t64.data(), n * entry,
                          cudaMemcpyHostToDevice) ||
        cudaMemset(counter, 0, 8) || cudaDeviceSynchronize();
  for (size_t g = 0; g < gates.size() && !bad; ++g) {
    EpiParams ep;
    ep.flags = gates[g].epi;
    ep.partial = ep.flags ? part : nullptr;
    bad = launch_plain_gate(precision, psi, L, gates[g].bond, tab + g * kGateEntries * entry, 0, counter, ep, 1,
                            cfg, 0);
  }
  bad = bad || cudaDeviceSynchronize();
  cudaFree(tab);
  cudaFree(counter);
  cudaFree(part);
  return bad;
}
"""


@pytest.fixture(scope="module")
def per_gate(svlib, tmp_path_factory):
    d = tmp_path_factory.mktemp("per_gate")
    src, lib = d / "per_gate.cu", d / "per_gate.so"
    src.write_text(_CODE)
    subprocess.run([b._nvcc(), *b.ARCH, *b.NVCC_FLAGS, "-shared", "-o", str(lib), str(src), b.LIB_PATH,
                    "-Xlinker", "-rpath=" + os.path.dirname(b.LIB_PATH)], check=True)
    f = ctypes.CDLL(str(lib)).per_gate_period
    f.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_int, ctypes.POINTER(capi.sv_floquet_params),
                  ctypes.c_double, ctypes.c_double]
    return f


@pytest.mark.parametrize("precision,L,K,first,drive", [
    # one block, several table loads, clusters of 2 to 16 blocks
    ("c64", 5, 3, 0, False), ("c64", 6, 4, 1, True), ("c64", 8, 14, 0, False), ("c64", 9, 4, 1, False),
    ("c64", 11, 4, 0, True), ("c64", 12, 4, 0, False), ("c64", 13, 9, 1, False), ("c64", 14, 2, 0, False),
    ("c64", 15, 4, 1, True),
    # tiles of 2^11 and 2^12, tables as parameters and in memory
    ("c64", 16, 4, 0, False), ("c64", 17, 3, 1, True), ("c64", 18, 4, 1, False), ("c64", 19, 2, 0, True),
    ("c64", 20, 4, 0, False), ("c64", 22, 1, 1, False),
    ("c128", 5, 4, 0, False), ("c128", 8, 14, 1, True), ("c128", 9, 4, 0, False), ("c128", 13, 4, 1, False),
    ("c128", 15, 2, 0, True), ("c128", 17, 2, 1, False)])
def test_state_of_one_pass_per_gate(per_gate, precision, L, K, first, drive):
    import torch
    from paper_2111_08044_gb300.sim import FloquetSimulator, chain_params
    P = 3
    cfg = inputs.ChainConfig(L=L, K=K, first_layer=first, periods=P, seed=L)
    if drive:
        cfg.theta_p, cfg.hx_p = np.linspace(0.2, 0.4, P), np.linspace(0.7, 0.9, P)
    with FloquetSimulator(L, precision=precision) as sim:
        sim.init_product_state(cfg.spinors())
        psi = sim.state.clone()
        sim.build(**chain_params(cfg))
        sim.evolve(P)
        torch.cuda.synchronize()
        p, _ = capi.make_params(**{k: v for k, v in chain_params(cfg).items() if k not in ("theta_p", "hx_p")})
        for k in range(P):
            assert per_gate(sim.precision, psi.data_ptr(), L, ctypes.byref(p),
                            cfg.theta_p[k] if drive else cfg.theta, cfg.hx_p[k] if drive else cfg.hx) == 0
        assert torch.equal(torch.view_as_real(psi).view(torch.int32 if precision == "c64" else torch.int64),
                           torch.view_as_real(sim.state).view(torch.int32 if precision == "c64" else torch.int64))
