"""Attached memory (rd_attach): its owner reads the time levels without the
library.  Until a tuning is set the reported one steps once per launch, and
the levels stand as it says: the current level by the parity of the steps
since the last field was set, the step before in the other level."""
import numpy as np
import pytest

from paper_1004_0480_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def levels(sim):
    """Both levels of every species, as the owner of the memory reads them."""
    nx, ny, nz = sim.shape
    buf = sim._keep[0]
    off = -buf.data_ptr() % 256
    nbytes = (buf.numel() - 256) // (2 * sim.nspecies)
    pitch = -(-nx // 32) * 32
    out = []
    for k in range(2 * sim.nspecies):
        a = buf[off + k * nbytes:off + k * nbytes + 4 * pitch * ny * nz].cpu().numpy()
        out.append(a.view(np.float32).reshape(nz, ny, pitch)[:, :, :nx])
    return np.stack(out).reshape(2, sim.nspecies, nz, ny, nx)


@pytest.mark.parametrize("cfg", [
    W.brusselator(shape=(97, 21, 10)),              # its own plan: two steps per launch
    W.diffusion_blob(shape=(64, 32, 24)),
    W.ch_front(shape=(40, 18, 12)),                 # one step per launch
], ids=lambda c: c["model"])
def test_levels_follow_one_launch_per_step(cfg):
    from paper_1004_0480_gb300.sim import Sim
    f = W.initial_fields(cfg)
    calls = [1, 2, 2, 3, 4, 5, 6, 7, 8, 9, 1, 40, 71]
    with Sim(cfg) as ref:                           # the library's own memory
        ref.set_fields(f)
        states = {0: ref.get_fields()}
        for n in range(1, sum(calls) + 1):
            ref.step(1)
            states[n] = ref.get_fields()
    with Sim(cfg, torch_memory=True) as sim:
        assert sim.tuning()["tsteps"] == 1
        sim.set_fields(f)
        n = 0
        for k in calls:
            sim.step(k)
            sim.sync()
            n += k
            lv = levels(sim)
            assert np.array_equal(sim.get_fields(), states[n]), (k, n)
            assert np.array_equal(lv[n & 1], states[n]), (k, n)
            assert np.array_equal(lv[n & 1 ^ 1], states[n - 1]), (k, n)
