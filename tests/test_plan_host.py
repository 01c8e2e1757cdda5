"""Plans on the host: the library's own plan code compiled for a made-up device
(152 SMs, 227 KB of shared memory), so that box shapes, caps and units are
checked without a GPU over more grids than a GPU test would run."""
import ctypes
import itertools
import math
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
pytestmark = pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")

SOURCE = r"""
#include <cuda_runtime.h>
static cudaError_t attribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 232448;
    return cudaSuccess;
}
#define cudaDeviceGetAttribute attribute
#include "api.cu"
extern "C" int plan_fields(const int *desc, long *out) {
    tetra_plan_t p;
    const int st = tetra_plan(&p, reinterpret_cast<const tetra_desc_t *>(desc), 0);
    if (st) return st;
    const long v[] = {p->BX, p->BY, p->BZ, p->n_boxes, p->nbx, p->nby, p->nbz, p->grid_x, p->items_per_box, p->fixed_bits,
                      p->fast_cap, p->flush_bits, p->copies, p->n_chunks, p->chunk_w, (long)p->smem_bytes};
    for (unsigned i = 0; i < sizeof v / sizeof *v; ++i) out[i] = v[i];
    return tetra_plan_destroy(p);
}
extern "C" int drop(float wmax, double cells) { return tetra::fermi_drop(wmax, cells); }
"""
NAMES = "BX BY BZ n_boxes nbx nby nbz grid items bits cap flush copies chunks width smem".split()
POINT, BIN, INTEGRATED = 0, 1, 2


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, so = d / "plan.cu", d / "plan.so"
    src.write_text(SOURCE)
    csrc = os.path.join(ROOT, "paper_1710_10789_gb300", "csrc")
    subprocess.run([NVCC, "-std=c++17", "-O1", "-shared", "-Xcompiler", "-fPIC", "-I", csrc, "-gencode",
                    "arch=compute_103a,code=sm_103a", str(src), "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so), mode=os.RTLD_LAZY)
    L.drop.argtypes = [ctypes.c_float, ctypes.c_double]
    return L


def fields(lib, n, bands, orbitals, energies, mode):
    out = (ctypes.c_long * len(NAMES))()
    st = lib.plan_fields((ctypes.c_int * 10)(*n, bands, orbitals, energies, mode, 0, 0, 0), out)
    return None if st else dict(zip(NAMES, out))


@pytest.mark.parametrize("n", [(1, 1, 1), (60, 60, 10), (2048, 2048, 2048), (4096, 4096, 4096), (4096, 3, 4095)])
def test_boxes_cover_the_grid(lib, n):
    for bands, energies, mode in ((1, 400, POINT), (1, 4000, BIN), (8, 200, INTEGRATED)):
        p = fields(lib, n, bands, 1, energies, mode)
        assert p["n_boxes"] == p["nbx"] * p["nby"] * p["nbz"] and 1 <= p["grid"] <= min(p["n_boxes"], 152)
        for side, box, count in zip(n, (p["BX"], p["BY"], p["BZ"]), (p["nbx"], p["nby"], p["nbz"])):
            assert (count - 1) * box < side <= count * box


def test_larger_boxes_keep_unit_weights_in_the_tile(lib, monkeypatch):
    """In bin and integrated mode the chosen box never sends items of weights up
    to one past the int32 tile where the default box keeps them; a box's items
    and the flush bound stay below 2^31 together; and the plan fits."""
    cases = itertools.product((16, 32, 48, 64, 96, 128, 256), (1, 2, 3, 4, 8, 12), (1, 3, 8, 16), (50, 200, 600, 1000, 2600, 4000),
                              (BIN, INTEGRATED))
    for side, bands, orbitals, energies, mode in cases:
        p = fields(lib, (side,) * 3, bands, orbitals, energies, mode)
        if p is None:
            continue
        for axis, size in zip("XYZ", (4, 4, max(1, min(4, 1536 // (16 * (3 if orbitals <= 8 else 6) * bands))))):
            monkeypatch.setenv("TETRA_BOX_" + axis, str(size))
        base = fields(lib, (side,) * 3, bands, orbitals, energies, mode)
        for axis in "XYZ":
            monkeypatch.delenv("TETRA_BOX_" + axis)
        unit = (2.02 if orbitals <= 8 else 1.01) * 2.0 ** p["bits"]
        assert p["bits"] == base["bits"]
        assert p["cap"] >= unit or base["cap"] < unit, (side, bands, orbitals, energies, mode, p, base)
        assert p["cap"] * p["items"] + 2 ** p["flush"] < 2 ** 31 and p["cap"] <= 2 ** 21
        assert p["smem"] <= 232448 and 1 <= p["copies"] <= 16


def test_fermi_unit(lib):
    """The scale of the weights keeps every sum of the count below 2^62 and
    every cube's value below 2^48, and is not larger than that takes: ordinary weights
    are not scaled, at 1024^3 points and 8 bands neither."""
    assert lib.drop(0.0, 1e9) == 0
    assert lib.drop(1.0, 8.0 * 1024 ** 3) == 0
    for cells in (1.0, 1e4, 8.0 * 256 ** 3, 64.0 * 1024 ** 3):
        for power in range(-20, 128):
            w = 1.5 * 2.0 ** (power - 1)
            d = lib.drop(w, cells)
            value = 6.0 * w * 2.0 ** (26 - d)
            assert value * cells <= 2.0 ** 62 and value <= 2.0 ** 48
            assert d == 0 or 2 * value * cells > 2.0 ** 61 or 2 * value > 2.0 ** 47
            assert math.isfinite(value)
