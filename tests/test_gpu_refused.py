"""Calls that are refused while their stream is captured: an error status, nothing
advanced, and the calls after them as if they had not been made."""
import ctypes

import numpy as np
import pytest

from paper_2111_08044_gb300 import capi, inputs

pytestmark = pytest.mark.gpu


class _Capture:
    """The stream's work goes to a graph that is thrown away."""

    def __init__(self, stream):
        self.rt = ctypes.CDLL("libcudart.so.13")
        self.s = ctypes.c_void_p(stream.cuda_stream)

    def __enter__(self):
        assert self.rt.cudaStreamBeginCapture(self.s, 2) == 0  # relaxed

    def __exit__(self, *exc):
        g = ctypes.c_void_p()
        self.rt.cudaStreamEndCapture(self.s, ctypes.byref(g))
        if g.value:
            self.rt.cudaGraphDestroy(g)
        self.rt.cudaGetLastError()


def _sim(L, stream, precision="c64", drive=False, **form):
    from paper_2111_08044_gb300.sim import FloquetSimulator, chain_params
    cfg = inputs.ChainConfig(L=L, seed=L)
    if drive:
        cfg.theta_p, cfg.hx_p = np.linspace(0.2, 0.4, 8), np.linspace(0.7, 0.9, 8)
    sim = FloquetSimulator(L, precision=precision, stream=stream)
    sim.init_product_state(cfg.spinors())
    sim.build(**chain_params(cfg, **form))
    return sim


def test_refused_call_leaves_no_error_behind(svlib):
    import torch
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        sim = _sim(14, s, mode=capi.SV_MODE_BLOCK, block_n=6)
        sim.evolve(1)
        with _Capture(s):
            assert svlib.sv_evolve(sim._ctx, 1, None, None) == capi.SV_ECUDA
        sim.init_product_state(inputs.ChainConfig(L=14).spinors())  # raised here
        sim.close()


def test_refused_batch_run_changes_nothing(svlib):
    """A run of another length after a refused one is of its own length."""
    import torch
    from paper_2111_08044_gb300.sim import FloquetBatch
    chains = [inputs.ChainConfig(L=L, seed=L) for L in (6, 12, 13)]
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        out = []
        for refuse in (False, True):
            with FloquetBatch(chains, form=capi.SV_BATCH_RESIDENT, stream=s) as b:
                parts = [b.evolve(8)]
                if refuse:
                    with _Capture(s):
                        assert svlib.sv_batch_evolve(b._b, 3, None, None) == capi.SV_ECUDA
                parts.append(b.evolve(3))
                out.append([x for p in parts for x in p] + [b.chain_state(c) for c in range(3)])
    for x, y in zip(*out):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("L,kw", [
    (4, {}), (6, {}), (12, {}), (15, {}), (17, {}), (12, dict(drive=True)), (17, dict(drive=True)),
    (19, dict(drive=True)), (9, dict(precision="df64")), (13, dict(precision="df64")),
    (7, dict(precision="c128")), (14, dict(mode=capi.SV_MODE_BLOCK, block_n=6)),
    (14, dict(mode=capi.SV_MODE_MULTIGATE))])
def test_refused_evolution_changes_nothing(svlib, L, kw):
    """An evolution under a capture is refused in every form: the periods of a replay
    would not be those that were captured."""
    import torch
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        out = []
        for refuse in (False, True):
            sim = _sim(L, s, **kw)
            sim.evolve(2)
            if refuse:
                with _Capture(s):
                    assert svlib.sv_evolve(sim._ctx, 2, None, None) == capi.SV_ECUDA
                assert sim.period == 2
            e, n = sim.evolve(3)
            out.append((e, n, sim.host_state()))
            sim.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)
