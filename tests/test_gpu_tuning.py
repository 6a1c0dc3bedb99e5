"""The library's own plan (no tiling set) and rd_set_tuning: changing the
graph flag, or writing back what was read, keeps the plan; a tiling replaces
it.  Seen by the launches: the plan of this small grid steps twice per
launch.  The results are the same bits either way."""
import numpy as np
import pytest

from paper_1004_0480_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_the_graph_flag_keeps_the_plan():
    from paper_1004_0480_gb300.sim import Sim
    cfg = W.brusselator(shape=(97, 33, 20))
    f = W.initial_fields(cfg)
    steps = 40

    def run(*tunings):
        with Sim(cfg) as sim:
            read = sim.tuning()
            assert read["tsteps"] == 1
            for t in tunings:
                sim.set_tuning(**(read if t == "read" else t))
            now = sim.tuning()
            sim.set_fields(f)
            before = sim.launches
            sim.step(steps)
            sim.step(1)
            n = sim.launches - before
            return n, now, sim.get_fields()
    n0, t0, ref = run()
    assert n0 == steps // 2 + 1
    for tunings in ([dict(graph=0)], ["read"], [dict(regcap=1)], [dict(graph=0), dict(graph=1)]):
        n, t, got = run(*tunings)
        assert n == n0, tunings
        assert {k: v for k, v in t.items() if k not in ("graph", "regcap")} == \
            {k: v for k, v in t0.items() if k not in ("graph", "regcap")}
        assert np.array_equal(got.view(np.uint32), ref.view(np.uint32))
    for tiling in (dict(tile_y=8), dict(zchunk=t0["zchunk"] + 1), dict(tile_q=8, tile_y=8)):
        n, t, got = run(tiling)
        assert n == steps + 1, tiling
        assert all(t[k] == v for k, v in tiling.items())
        assert np.array_equal(got.view(np.uint32), ref.view(np.uint32))
    # a tiling set once stays set
    assert run(dict(tile_y=8), dict(graph=0))[0] == steps + 1
