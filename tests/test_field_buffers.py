"""Buffers that are too short for a field are refused on the host, before a
kernel reads or writes past them: by the element count in the Python binding,
and by the driver's allocation ranges in the library."""
import shutil
import subprocess

import numpy as np
import pytest

from paper_1004_0480_gb300 import build as B
from paper_1004_0480_gb300.sim import Sim


class _Lib:
    """Records the calls that reach the library."""
    def __init__(self):
        self.calls = []

    def _call(self, name):
        return lambda ctx, s, ptr, n: self.calls.append((name, n)) or 0

    def __getattr__(self, name):
        return self._call(name)


@pytest.mark.parametrize("cells", [0, 23])
def test_the_binding_checks_the_element_count(cells):
    torch = pytest.importorskip("torch")
    sim = Sim.__new__(Sim)
    sim.lib, sim.ctx, sim.shape, sim.nspecies = _Lib(), 1, (4, 3, 2), 1
    for good in (np.zeros((2, 3, 4), np.float32), torch.zeros(2, 3, 4)):
        sim.set_field(0, good)
        assert sim.get_field(0, good) is good
    assert sim.get_field(0).shape == (2, 3, 4)
    sim.get_field(0, np.zeros(25, np.float32))       # the first 24 are written
    done = list(sim.lib.calls)
    assert done == [("rd_set_field", 24), ("rd_get_field", 24)] * 2 + [("rd_get_field", 24)] * 2
    for bad in (np.zeros(cells, np.float32), torch.zeros(cells)):
        with pytest.raises(ValueError):
            sim.set_field(0, bad)
        with pytest.raises(ValueError):
            sim.get_field(0, bad)
    assert sim.lib.calls == done
    sim.ctx = None


PROGRAM = r"""
#include <cstdio>
#include "rd_extent.h"
using namespace rdk;

// allocations [base, base + size): two that adjoin, a gap, a third
static const unsigned long long kAlloc[][2] = {{1000, 400}, {1400, 600}, {3000, 100}};

static CUresult fake(CUdeviceptr* base, size_t* size, CUdeviceptr p) {
    for (auto& a : kAlloc)
        if (p >= a[0] && p < a[0] + a[1]) {
            *base = a[0];
            *size = a[1];
            return CUDA_SUCCESS;
        }
    return CUDA_ERROR_NOT_FOUND;
}

int main() {
    struct { CUdeviceptr p; size_t bytes; Extent want; } cases[] = {
        {1000, 400, Extent::kOne},      {1000, 4, Extent::kOne},       {1399, 1, Extent::kOne},
        {1000, 401, Extent::kSeveral},  {1200, 800, Extent::kSeveral}, {1200, 801, Extent::kShort},
        {1400, 600, Extent::kOne},      {1996, 8, Extent::kShort},     {3000, 100, Extent::kOne},
        {3096, 5, Extent::kShort},      {1000, (size_t)-1, Extent::kShort},
        {500, 4, Extent::kSeveral}};    // unknown to the driver: the runtime decides
    int bad = 0;
    for (auto& c : cases)
        if (extent_of(fake, c.p, c.bytes) != c.want) {
            std::printf("[%llu, +%zu)\n", (unsigned long long)c.p, c.bytes);
            ++bad;
        }
    return bad != 0;
}
"""


def test_the_library_walks_the_driver_allocations(tmp_path):
    try:
        nvcc = B.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    src = tmp_path / "extent.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "extent")
    subprocess.run([nvcc, *B.ARCH, "-std=c++17", f"-I{B.INCLUDE}", f"-I{B.CSRC}", str(src),
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
