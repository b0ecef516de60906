"""Tiles of the FP64 general kernel: 32 x 4 nodes where they leave the fullest SM with
fewer rows of 32 nodes than 32 x 8 tiles, else 32 x 8, and the results of either."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2208_03562_gb300 import inputs as I

L = pytest.importorskip("paper_2208_03562_gb300.lbm")

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if not nvcc:
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("host_plan") / "libhost_plan.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17",
                    "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2208_03562_gb300", "csrc"), os.path.join(HERE, "host_plan.cu"),
                    "-o", out], check=True, capture_output=True)
    return C.CDLL(out).host_f64_tile_rows


# on 152 SMs, the faster shape as measured
@pytest.mark.parametrize("nx,ny,want", [(64, 64, 4), (100, 150, 4), (512, 64, 8), (152, 152, 8), (96, 300, 8),
                                        (512, 128, 8), (300, 300, 4), (512, 192, 8), (256, 500, 4), (304, 380, 4),
                                        (200, 650, 8), (700, 300, 4), (512, 400, 4), (500, 500, 8), (512, 512, 8),
                                        (640, 480, 8), (724, 724, 8), (1024, 1024, 8)])
def test_the_faster_shape(rows, nx, ny, want):
    assert rows(nx, ny, 152) == want


def test_without_a_device_the_shape_with_fewer_sums(rows):
    assert rows(64, 64, 0) == 8     # the allocation-free step's scratch holds the sums of 32 x 8 tiles


# one wave and several of either shape, partial tiles in both directions
@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(152, 152), (513, 130), (301, 299), (257, 501), (701, 375)])
def test_results_do_not_depend_on_the_shape(nx, ny):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    p = L.lbm_params_init(nx, ny, 0.7, 0.4, 0.02, 0.02, L.F64)
    h, b = L.Lbm(p), L.Batch(1, L.F64)
    assert h.variant == L.VARIANT_GENERAL
    s = b.add(p, 0.0, 10 ** 6)
    h.init_fields(*I.random_fields(nx, nx, ny, 5e-3, 5e-3))
    b.set_populations(s, h.populations())
    h.set_populations(b.populations(s))
    for n in (20, 23, 37):     # a batch keeps 32 x 8 tiles
        h.step(n)
        b.run(n)
        info = b.query(s)[0]
        assert (info.residual, info.mass) == (h.residual(), h.info().mass)
        assert np.array_equal(h.populations(), b.populations(s))
    h.close()
    b.close()
