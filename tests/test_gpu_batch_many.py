"""Batches of more members than a warp has lanes, few work items each (so the
CTAs take every gridDim-th item and pull none): the thread that finds an
item's owner then sits in another warp than the first, and a member stepped
with another's descriptor would show.  Every member must equal the same
problem stepped alone bit for bit, in every step kernel that batches run."""
import numpy as np
import pytest

from paper_1004_0480_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# rows that end inside a vector or a tile, the smallest grids, ragged heights
SHAPES = [(2, 2, 2), (5, 3, 4), (63, 9, 7), (64, 12, 6), (65, 13, 5), (66, 17, 9), (24, 8, 11),
          (31, 6, 3), (8, 16, 13)]
MEMBERS = 44                         # at most 166 work items: one wave of CTAs
T1 = dict(tsteps=1, tile_q=16, tile_y=16, zchunk=64)
TUNINGS = {7: [T1, dict(T1, tsteps=2, tile_y=12), dict(T1, tsteps=3, tile_y=4),
               dict(T1, tile_q=8)],
           19: [T1], "ch": [dict(T1, tile_y=14), dict(T1, tsteps=2, tile_y=4)]}
MAKE = {
    "diffusion": lambda s, i: W.diffusion_blob(shape=s, seed=i),
    "brusselator": lambda s, i: W.brusselator(shape=s, seed=i),
    "air": lambda s, i: W.air(s, src=(s[0] - 1, 0, s[2] - 1), seed=i),
    "ch_front": lambda s, i: W.with_(W.ch_front(shape=s, seed=i), init="uniform_noise"),
}


@pytest.mark.parametrize("model,stencil,storage", [
    ("diffusion", 7, "f32"), ("brusselator", 7, "f32"), ("brusselator", 7, "bf16"),
    ("air", 7, "f32"), ("ch_front", 7, "f32"), ("ch_front", 7, "bf16"),
    ("brusselator", 19, "f32"), ("brusselator", 19, "bf16"), ("ch_front", 19, "f32")])
def test_many_members_equal_their_own_runs(model, stencil, storage):
    from paper_1004_0480_gb300.sim import Batch, Sim
    cfgs = [W.with_(MAKE[model](SHAPES[i % len(SHAPES)], i), stencil=stencil)
            for i in range(MEMBERS)]
    fields = [W.initial_fields(c) for c in cfgs]
    steps = 19                       # a 16-launch graph replay and 3 plain launches

    def run(tuning):
        sims = [Sim(c, storage) for c in cfgs]
        try:
            for s, f in zip(sims, fields):
                s.set_fields(f)
            if tuning is None:       # each alone
                for s in sims:
                    s.step(steps)
                return [s.get_fields() for s in sims]
            b = Batch(model, storage)
            b.set_tuning(**tuning)
            for s in sims:
                b.add(s)
            b.step(steps)
            b.sync()
            b.close()
            return [s.get_fields() for s in sims]
        finally:
            for s in sims:
                s.close()
    ref = run(None)
    for t in TUNINGS["ch" if model == "ch_front" and stencil == 7 else stencil]:
        for i, (a, b) in enumerate(zip(run(t), ref)):
            assert np.array_equal(a.view(np.uint32), b.view(np.uint32)), (t, cfgs[i]["shape"])


@pytest.mark.parametrize("model,stencil,storage", [
    ("diffusion", 7, "f32"), ("diffusion", 7, "bf16"), ("brusselator", 7, "f32"),
    ("brusselator", 7, "bf16"), ("air", 7, "f32"), ("ch_front", 7, "f32"),
    ("diffusion", 19, "f32"), ("brusselator", 19, "f32")])
@pytest.mark.parametrize("tsteps", [1, 2])
def test_a_batch_launches_the_ctas_that_fit(model, stencil, storage, tsteps):
    """A persistent batch kernel with more CTAs than the GPU holds starts the
    surplus after the others have taken their whole lists."""
    import ctypes

    from paper_1004_0480_gb300 import _lib as L
    from paper_1004_0480_gb300.sim import Batch, Sim
    if tsteps == 2 and (stencil == 19 or model == "ch_front"):
        pytest.skip("one step per launch")
    out = (ctypes.c_int64 * 2)()
    lib = L.load()
    for ty in (6, 8, 12, 14):
        # 2 x 512 work items at least: more than the GPU holds
        sims = [Sim(W.with_(MAKE[model]((64, 8 * ty, 64), i), stencil=stencil), storage)
                for i in range(2)]
        b = Batch(model, storage)
        b.set_tuning(tsteps=tsteps, tile_q=16, tile_y=ty, zchunk=1)
        for s in sims:
            b.add(s)
        assert lib.rd_debug_batch_grid(b.b, out) == L.RD_EINVAL      # nothing launched yet
        b.step(tsteps)
        b.sync()
        assert lib.rd_debug_batch_grid(b.b, out) == L.RD_OK
        assert out[0] == min(1024, out[1]), (ty, list(out))
        b.close()
        for s in sims:
            s.close()
