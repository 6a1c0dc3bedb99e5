"""The march kernels (rd_march_kernel: one or two steps per launch;
rd_march19_kernel: the 19-point stencil; rd_marchch_kernel: Cahn-Hilliard) where they can go wrong: rows that end inside a vector or a tile, tiles and z-chunks that the
grid does not fill, the smallest grids, wrapped and mirrored halos, held
layers, wind and a source on the faces.  Every launch shape evaluates the
same rounded operations, so results must equal the multi-level kernel's (an
odd tile height) bit for bit."""
import numpy as np
import pytest

from paper_1004_0480_gb300 import workloads as W

pytestmark = pytest.mark.gpu

D, N, P = "dirichlet", "neumann", "periodic"


def problem(kind, shape):
    nx, ny, nz = shape
    if kind == "diffusion":
        return W.diffusion_blob(shape=shape)
    if kind == "turing":
        return W.turing(shape=shape, sigma=0.3)
    if kind == "brusselator":
        return W.brusselator(shape=shape)
    if kind == "held":
        return W.with_(W.brusselator(shape=shape, bc=N),
                       bc=[[D, N, N, D, D, N], [N, D, D, N, N, D]],
                       bc_value=[[3.1, 0, 0, 2.9, 3.3, 0], [0, 3.05, 2.95, 0, 0, 2.8]])
    src = (nx - 1, 0, nz - 1)                     # on three faces
    if kind == "air":
        return W.air(shape, src=src)
    if kind == "air_calm":
        return W.with_(W.air(shape, src=src), wind=None, bc=[[P, P, N, N, P, P]] * 3)
    return W.with_(W.air(shape, src=src), bc=[[N, N, P, P, N, N]] * 3,
                   wind=dict(kind="const", u0=-1.0))


SHAPES = [(2, 2, 2), (5, 3, 4), (63, 9, 7), (64, 12, 6), (65, 13, 5), (66, 17, 9), (127, 8, 11),
          (131, 26, 3)]
TUNINGS = [dict(tsteps=2, tile_y=8, zchunk=1), dict(tsteps=2, tile_y=12, zchunk=4, graph=0),
           dict(tsteps=1, tile_y=14, zchunk=3), None]


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("kind", ["diffusion", "turing", "brusselator", "held", "air", "air_calm",
                                  "air_mixed"])
def test_bits_equal_the_multi_level_kernel(kind, storage):
    from paper_1004_0480_gb300.sim import Sim
    for shape in SHAPES:
        cfg = problem(kind, shape)
        f = W.initial_fields(cfg)

        def run(tuning):
            with Sim(cfg, storage, tuning=tuning) as s:
                s.set_fields(f)
                s.step(5)                         # two pairs and a single step
                s.step(1)
                return s.get_fields()
        ref = run(dict(tsteps=2, tile_y=5, zchunk=3))
        for t in TUNINGS:
            got = run(t)
            assert np.array_equal(got.view(np.uint32), ref.view(np.uint32)), (shape, t)


@pytest.mark.parametrize("kind", ["turing", "brusselator", "held", "air", "air_mixed",
                                  "ch_table1", "plume"])
def test_19_point_tilings_agree_and_match_the_oracle(kind):
    import oracle
    from paper_1004_0480_gb300.sim import Sim
    oracle.build()
    for shape in SHAPES:
        if kind == "ch_table1":
            cfg = W.with_(W.ch_table1(shape=shape), init="uniform_noise")
        elif kind == "plume":
            cfg = W.with_(W.plume(shape, src=(shape[0] - 1, 0, 0)), stencil=19,
                          init="uniform_noise")
        else:
            # one diffusivity per species on this stencil
            cfg = W.with_(problem(kind, shape), stencil=19)
            cfg["D"] = [[d[0]] * 3 for d in cfg["D"]]
        f = W.initial_fields(cfg)
        ref = oracle.run(cfg, f, 5)
        first = None
        for t in (None, dict(tile_y=2, zchunk=1, graph=0), dict(tile_y=8, zchunk=3),
                  dict(tile_y=14, zchunk=64)):
            with Sim(cfg, tuning=t) as s:
                s.set_fields(f)
                s.step(5)
                got = s.get_fields()
            # FP32 rounding of 5 steps: some 20 roundings of 6e-8 a step,
            # amplified at most a few times by the reactions
            for a, b in zip(got, ref):
                assert np.abs(a - b).max() <= 2e-5 * max(np.abs(b).max(), 1e-30), (shape, t)
            first = got if first is None else first
            assert np.array_equal(got.view(np.uint32), first.view(np.uint32)), (shape, t)


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("kind", ["front", "periodic_front", "source_front", "table1"])
def test_cahn_hilliard_bits_equal_the_multi_level_kernel(kind, storage):
    from paper_1004_0480_gb300.sim import Sim
    for shape in SHAPES:
        if kind == "table1":
            cfg = W.with_(W.ch_table1(shape=shape, dt=0.001, stencil=7), init="uniform_noise")
        else:
            cfg = W.with_(W.ch_front(shape=shape), init="uniform_noise")
        if kind == "periodic_front":
            cfg = W.with_(cfg, bc=[[P] * 6] * 3)
        if kind == "source_front":          # the general variant
            nx, ny, nz = shape
            cfg = W.with_(cfg, source=dict(x=nx - 1, y=ny - 1, z=0, species=1, rate=2.0),
                          D=[[1.0, 0.5, 0.25], [0.1] * 3, [0.0] * 3])
        f = W.initial_fields(cfg)

        def run(tuning):
            with Sim(cfg, storage, tuning=tuning) as s:
                s.set_fields(f)
                s.step(4)
                return s.get_fields()
        ref = run(dict(tsteps=2, tile_y=5, zchunk=3))
        for t in (None, dict(tsteps=1, tile_y=12, zchunk=4), dict(tsteps=1, tile_y=5, zchunk=1),
                  dict(tsteps=1, tile_y=26, zchunk=2, graph=0)):
            got = run(t)
            assert np.array_equal(got.view(np.uint32), ref.view(np.uint32)), (shape, t)
