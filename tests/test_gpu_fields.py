"""Fields in and out: device memory that the pack and unpack kernels read and
write themselves (vectors where rows and base allow, single cells otherwise)
and memory that goes through the staging field give the same bits."""
import numpy as np
import pytest

from paper_1004_0480_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("shape", [(2, 2, 2), (4, 3, 2), (5, 4, 3), (64, 5, 7), (255, 6, 3),
                                   (1028, 2, 3)])
def test_device_and_host_buffers_agree(shape, storage):
    import torch
    from paper_1004_0480_gb300.sim import Sim
    D, N = "dirichlet", "neumann"
    cfg = W.with_(W.diffusion_blob(shape=shape), bc=[[D, N, N, D, N, D]],
                  bc_value=[[1.5, 0, 0, 2.5, 0, 3.5]])
    f = W.initial_fields(cfg)
    nx, ny, nz = shape
    n = nx * ny * nz
    dev = torch.from_numpy(f[0]).cuda()
    room = torch.empty(n + 8, device="cuda")
    shifted = room[1:n + 1].view(nz, ny, nx)        # 4-byte aligned only
    shifted.copy_(dev)
    torch.cuda.synchronize()
    with Sim(cfg, storage) as s:
        out = []
        for src in (f[0], dev, shifted):
            s.set_field(0, torch.zeros_like(dev))
            s.set_field(0, src)
            out.append(s.get_field(0))
            for dst in (torch.full_like(dev, -1.0), shifted.clone().fill_(-1.0),
                        room[3:n + 3].view(nz, ny, nx)):
                s.get_field(0, dst)
                out.append(dst.cpu().numpy())
            shifted.copy_(dev)
            torch.cuda.synchronize()
    for o in out[1:]:
        assert np.array_equal(o.view(np.uint32), out[0].view(np.uint32))


def test_buffers_inside_the_context_go_through_staging():
    import torch
    from paper_1004_0480_gb300.sim import Sim
    cfg = W.diffusion_blob(shape=(32, 6, 5))
    f = W.initial_fields(cfg)
    with Sim(cfg, torch_memory=True) as s:
        s.set_fields(f)
        # the state's first level (pitch 32 = nx, so it is a dense field)
        base = s._keep[0]
        off = (-base.data_ptr()) % 256
        inside = base[off:off + 4 * 32 * 6 * 5].view(torch.float32).view(5, 6, 32)
        flipped = torch.flip(torch.from_numpy(f[0]).cuda(), [0])
        torch.cuda.synchronize()
        s.set_field(0, inside)                      # onto itself
        assert np.array_equal(s.get_field(0), f[0])
        s.set_field(0, flipped)
        s.get_field(0, inside)
        assert np.array_equal(inside.cpu().numpy(), flipped.cpu().numpy())
