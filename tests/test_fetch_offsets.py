"""Where the step kernels copy from: the offset of every fetch within a plane,
on the host, against 64-bit arithmetic.  Planes of 2^31 cells and more (two
such planes are within the accepted 2^34 cells) must not overflow, planes past
the offsets' range are refused, and the smallest and odd planes keep their
rules: wrapped rows and columns on periodic axes, mirrored (march kernels) or
clamped (8-cell kernel) rows beyond zero-flux faces, nothing where no stored
cell needs a vector."""
import ctypes
import shutil
import subprocess

import pytest

from paper_1004_0480_gb300 import _lib as L
from paper_1004_0480_gb300 import build as B
from paper_1004_0480_gb300 import workloads as W

PROGRAM = r"""
#include <cstdio>
#include "rd_step19_kernel.cuh"
using namespace rdk;
typedef long long ll;

static int bad = 0;

// one fetch of ``w`` cells from column xs of a row whose mapped index is ``row``
static void check(const char* what, const Fetch& f, int w, ll row, int xs, int nx, ll pitch,
                  bool px) {
    const bool none = !px && (xs + w <= 0 || xs >= nx || (w == kVEC && xs < 0));
    const ll x = px ? ((ll)xs % nx + nx) % nx : xs;
    // no single copy: wraps round, straddles a face (8-cell kernel)
    const bool split = px ? x % w || x + w > nx : w == kW8 && x + w > nx;
    bool ok;
    if (none) ok = f.mode == 0 && own_offset(f) == kNone;   // not the plane's first vector
    else if (split) ok = f.mode == 2 && own_offset(f) == kElems && (ll)f.goff * kVEC == row * pitch && f.xs == xs;
    else ok = f.mode == 1 && own_offset(f) == f.goff && (ll)f.goff * kVEC == row * pitch + x && x + w <= pitch;
    if (!ok && bad++ < 5)
        std::printf("%s: row %lld of pitch %lld, x %d of %d: mode %d, offset %u\n", what, row,
                    pitch, xs, nx, f.mode, f.goff);
}

int main() {
    struct { int nx, ny; } planes[] = {
        {2, 2}, {5, 3}, {64, 9}, {67, 18}, {256, 256}, {46342, 46342}, {46400, 46400},
        {32, 1 << 27}, {92681, 92681}, {1 << 30, 7}, {2, 1 << 28}, {16, (1 << 28) - 9}};
    for (auto p : planes)
        for (int align : {32, 64})
            for (int per = 0; per < 4; ++per) {
                const bool px = per & 1, py = per & 2;
                const int nx = p.nx, ny = p.ny;
                const int pitch = (nx + align - 1) / align * align;
                if (!plane_fits((ll)pitch * ny)) continue;     // refused by rd_create
                for (int y : {-2, -1, 0, 1, ny / 2, ny - 2, ny - 1, ny, ny + 1})
                    for (int v : {-1, 0, 1, nx / 8, nx / 4 - 1, nx / 4, nx / 4 + 1}) {
                        const int xs = v * kVEC;
                        if (xs > nx + 1 || (!py && (y < -ny || y >= 2 * ny))) continue;
                        const ll wrap = ((ll)y % ny + ny) % ny;
                        const ll mirror = y < 0 ? -1 - y : (y >= ny ? 2LL * ny - 1 - y : y);
                        check("march", make_fetch_h<float>(y, xs, nx, ny, pitch, px, py, 0), kVEC,
                              py ? wrap : mirror, xs, nx, pitch, px);
                        const ll clamp = y < 0 ? 0 : (y >= ny ? ny - 1 : y);
                        const int x8 = v * kW8;
                        if (x8 > nx + 1) continue;
                        check("8-cell", make_fetch8<float>(y, x8, nx, ny, pitch, px, py, 0), kW8,
                              py ? wrap : clamp, x8, nx, pitch, px);
                    }
            }
    std::printf("%d wrong\n", bad);
    return bad != 0;
}
"""


def test_fetch_offsets_on_the_host(tmp_path):
    try:
        nvcc = B.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    src = tmp_path / "fetch.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "fetch")
    subprocess.run([nvcc, *B.ARCH, "-std=c++17", f"-I{B.INCLUDE}", f"-I{B.CSRC}", str(src),
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_planes_past_the_offsets_are_refused():
    from paper_1004_0480_gb300.sim import make_config
    B.build()
    lib = L.load()

    def query(shape, storage):
        c = make_config(W.diffusion_blob(shape=(8, 8, 8)), storage)
        c.nx, c.ny, c.nz = shape
        return lib.rd_query_sizes(ctypes.byref(c), None, None)
    for storage in ("f32", "bf16"):
        assert query((46342, 46342, 2), storage) == L.RD_OK       # 2^31 cells a plane
        assert query((92681, 92681, 2), storage) == L.RD_OK       # the largest two planes
        assert query((2, 2**28 - 9, 2), storage) == L.RD_OK       # 2^34 padded elements in BF16
        assert query((92683, 92683, 2), storage) == L.RD_EINVAL   # more than 2^34 cells
        assert query((2, 2**29, 2), storage) == L.RD_EINVAL
        assert query((2**31 - 1, 2, 2), storage) == L.RD_EINVAL   # padded past an int
        assert query((2**31 - 64, 2, 2), storage) == L.RD_OK
    assert query((2, 2**28, 2), "f32") == L.RD_OK
    assert query((2, 2**28, 2), "bf16") == L.RD_EINVAL
