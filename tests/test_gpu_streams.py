"""Work of a context stays on the context's own stream."""
import numpy as np
import pytest

from paper_1611_00907_gb300 import LbmError, Simulation, _lib, eos_coexistence, inputs

pytestmark = pytest.mark.gpu


def test_creation_leaves_nothing_behind_on_the_default_stream():
    """A context on a non-blocking stream, made while the default stream has
    work queued: nothing of its creation runs later on the default stream and
    clears what the context's kernels have reported since (here a wait of zero
    cycles that ran out; the sums of lbm_reduce lie beside it)."""
    import torch
    rv, rl, _ = eos_coexistence("cs", 1.0, 4.0, 1.0, 0.85)
    rho = inputs.drop(64, 64, 16, rl, rv)
    lib = _lib.load()

    def make(stream):
        return Simulation(64, 64, "cs", 1.0, 4.0, 1.0, 0.85, tau=1.0, kappa=0.5,
                          precision="f64", stream=stream.cuda_stream)

    stream = torch.cuda.Stream()
    with make(stream) as sim:        # kernels loaded: what follows waits for nothing else
        want = sim.init(rho).step(8).reduce()[:3]
        sim.moments()
    torch.cuda.synchronize()
    torch.cuda._sleep(2_000_000_000)  # a second or so on the default stream
    busy = torch.cuda.Event()
    busy.record()
    sim = make(stream)
    with sim:
        assert lib.lbm_test_set_wait_cycles(sim._ctx, 0) == _lib.LBM_OK
        sim.init(rho).step(8)
        stream.synchronize()
        assert not busy.query()       # the default stream is still at work
        torch.cuda.synchronize()
        with pytest.raises(LbmError) as ei:
            sim.moments()
        assert "timed out" in str(ei.value)
        assert lib.lbm_test_set_wait_cycles(sim._ctx, -1) == _lib.LBM_OK
        got = sim.init(rho).step(8).reduce()[:3]
    assert np.allclose(got, want, rtol=1e-12, atol=1e-12)
