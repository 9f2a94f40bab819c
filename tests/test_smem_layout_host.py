"""A CTA's dynamic shared memory over the lattice sizes that a context accepts (csrc/dqmc_layout.h, compiled alone with
g++): within the 227 KB of the architecture up to the sizes that fitted before the staging buffers and the QR's panels
were part of it (1735 sites in FP64, FP32 and MIXED, 1296 in MIXED_TC), with two stages wherever the split products are
used and two columns at least for the QR's panels."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1704_00131_gb300", "csrc")

SHIM = r"""
#include "dqmc_layout.h"
using namespace dqmc;
extern "C" long shim_total(int ld, int mv, long ab, int n, int digits) { return (long)smem_total(ld, mv, ab, n, digits); }
extern "C" long shim_offset(int ld, int mv) { return (long)smem_stage_offset(ld, mv); }
extern "C" int shim_fits(int ld, int mv, int n, int digits) { return split_fits(ld, mv, n, digits); }
extern "C" int shim_cols(int n, long bytes) { return qr_panel_cols(n, bytes); }
extern "C" int shim_rows(int n) { return umma_rows(n); }
extern "C" int shim_tiles(int n) { return umma_row_tiles(n); }
extern "C" int shim_exp_len(int ld) { return exp_len(ld); }
"""

LIMIT = 227 * 1024
SIZES = list(range(1, 200)) + [255, 256, 257, 400, 576, 900, 1023, 1024, 1025, 1104, 1105, 1156, 1296, 1440, 1441, 1447,
                               1500, 1550, 1551, 1560, 1561, 1600, 1672, 1673, 1734, 1735]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("layout")
    (d / "shim.cpp").write_text(SHIM)
    so = d / "libshim.so"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, "-o", str(so), str(d / "shim.cpp")])
    lib = ctypes.CDLL(str(so))
    for f in ("shim_total", "shim_offset"):
        getattr(lib, f).restype = ctypes.c_long
    lib.shim_total.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_long, ctypes.c_int, ctypes.c_int]
    lib.shim_cols.argtypes = [ctypes.c_int, ctypes.c_long]
    return lib


@pytest.mark.parametrize("vertices", ["all", "one"])
def test_every_size_fits(lib, vertices):
    for n in SIZES:
        ld, mv = (n + 3) // 4 * 4, n if vertices == "all" else 1
        off = lib.shim_offset(ld, mv)
        for digits in (7, 8):
            d = digits if lib.shim_fits(ld, mv, n, digits) else 0
            total = lib.shim_total(ld, mv, 0, n, d)
            assert total <= LIMIT, (n, digits)
            region = total - off  # what a kernel finds behind its vectors
            cols = lib.shim_cols(n, region)
            assert cols >= 2 and 2 * cols * (n | 1) * 8 <= region, n
            assert 2 * (n | 1) * 8 <= region  # the LU's panels: one column each at least
            if d:
                assert region >= 2 * d * 32 * (lib.shim_rows(n) + 32), (n, digits)
            if off + 2 * 4 * (ld + 1) * 8 + 128 <= LIMIT:  # four columns fit
                assert cols == 4, n
        assert lib.shim_rows(n) * lib.shim_tiles(n) <= lib.shim_exp_len(ld)


def test_split_products_wherever_two_stages_fit(lib):
    """FP64 to 1560 sites and float pairs to 1672."""
    for n in SIZES:
        ld = (n + 3) // 4 * 4
        assert lib.shim_fits(ld, n, n, 8) == (n <= 1560), n
        assert lib.shim_fits(ld, n, n, 7) == (n <= 1672), n
