"""A simulator made, built and run on a stream of its own while another stream is
busy: its tables are uploaded in that order, and it does not wait for the other
stream (whose work a copy on the default stream would follow)."""
import numpy as np
import pytest

from paper_2111_08044_gb300 import capi, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,L,form", [
    ("c64", 4, {}), ("c64", 12, {}), ("c64", 17, {}), ("df64", 9, {}), ("df64", 13, {}), ("c128", 13, {}),
    ("c64", 14, dict(mode=capi.SV_MODE_MULTIGATE)), ("c64", 12, dict(mode=capi.SV_MODE_BLOCK, block_n=5)),
    ("c64", 14, dict(mode=capi.SV_MODE_BLOCK, block_n=6))])
def test_side_stream_beside_a_busy_default_stream(svlib, precision, L, form):
    import torch
    from paper_2111_08044_gb300.sim import FloquetSimulator, chain_params
    cfg = inputs.ChainConfig(L=L, seed=L)
    side = torch.cuda.Stream()
    dtype = torch.complex64 if precision == "c64" else torch.complex128
    state = torch.empty(1 << L, dtype=dtype, device="cuda")
    done = torch.cuda.Event()

    def run(busy):
        torch.cuda.synchronize()
        if busy:  # half a second and more of the default stream
            torch.cuda._sleep(1 << 30)
            done.record()
        sim = FloquetSimulator(L, precision=precision, stream=side, state=state)
        sim.init_product_state(cfg.spinors())
        sim.build(**chain_params(cfg, **form))
        e, n = sim.evolve(3)
        psi = sim.host_state()
        waited = busy and done.query()
        sim.close()
        return e, n, psi, waited

    first, second = run(False), run(True)
    for x, y in zip(first[:3], second[:3]):
        assert np.array_equal(x, y)
    assert not second[3], "the build waited for the default stream"
