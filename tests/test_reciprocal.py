"""FP64 reciprocals and quotients of the CUDA path.

``vrcp(double)`` refines the hardware's approximation y by one cubic step.  The
approximation takes the upper 32 bits of the operand (20 of the mantissa) and
gives as many: its relative error is at most three units of 2^-20 (operand, result,
approximation).  The step leaves the cube of that, 27 x 2^-60, and one rounding:
at most 0.5 + 27 x 2^-60 x 2^53 < 0.75 units in the last place.  At the ends of the
exponent range it divides, exactly as numpy does."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import stepper as S
from paper_2208_03562_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = pytest.importorskip("paper_2208_03562_gb300.lbm")
torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2208_03562_gb300", "csrc")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    L.load()


@pytest.fixture(scope="module")
def vrcp(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if not nvcc:
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("vrcp") / "libvrcp.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, "device_vrcp.cu"), "-o", out], check=True, capture_output=True)
    lib = C.CDLL(out)
    lib.device_vrcp.argtypes = [C.c_void_p, C.c_void_p, C.c_int]

    def call(a):
        a = np.ascontiguousarray(a, dtype=np.float64)
        y = np.empty_like(a)
        assert lib.device_vrcp(a.ctypes.data, y.ctypes.data, a.size) == 0
        return y
    return call


def split(a):
    c = 134217729.0 * a     # 2^27 + 1: the upper 26 bits and the rest
    h = c - (c - a)
    return h, a - h


def ulps(a, y):
    """|y - 1/a| in units in the last place of y, from the exact product (Dekker 1971)."""
    m, e = np.frexp(np.abs(a))
    z = np.ldexp(np.abs(y), e)              # y of the operand m in [1/2, 1)
    p = m * z
    (mh, ml), (zh, zl) = split(m), split(z)
    low = ((mh * zh - p) + mh * zl + ml * zh) + ml * zl
    return np.abs((1 - p) - low) / m / np.spacing(z)


def test_reciprocal_is_within_three_quarters_of_an_ulp(vrcp):
    g = I.rng(77)
    m = np.concatenate([1 + g.random(1 << 20), 1 + np.arange(4096) * 2.0 ** -52, 2 - (1 + np.arange(4096)) * 2.0 ** -52,
                        1 + np.arange(1 << 20) * 2.0 ** -20, 1 + (np.arange(1 << 20) + 1) * 2.0 ** -20 - 2.0 ** -52])
    m = m[m < 2]
    e = g.integers(64 - 1023, 1984 - 1023, m.size)
    e[::7] = 64 - 1023
    e[1::7] = 1983 - 1023
    e[2::7] = 0
    a = np.ldexp(m, e) * g.choice([-1.0, 1.0], m.size)
    y = vrcp(a)
    err = ulps(a, y)
    print("largest error %.4f ulp, correctly rounded %.5f" % (err.max(), np.mean(y == 1 / a)))
    assert np.array_equal(np.signbit(y), np.signbit(a)) and err.max() < 0.75


def test_reciprocal_divides_at_the_ends_of_the_range(vrcp):
    g = I.rng(78)
    m = 1 + g.random(20000)
    e = np.concatenate([g.integers(1, 64, 10000), g.integers(1984, 2047, 10000)]) - 1023
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.0 ** -1030, 1.7976931348623157e308])
    a = np.concatenate([np.ldexp(m, e) * g.choice([-1.0, 1.0], m.size), special])
    with np.errstate(all="ignore"):
        assert np.array_equal(vrcp(a), 1 / a, equal_nan=True)


@pytest.mark.parametrize("noise", [1e-3, 0.2])
def test_fp64_fields_round_their_quotients_once(noise):
    """The sums of the stored deviations in the kernel's order, then the quotient."""
    nx, ny, r = 131, 67, 0.7
    p = L.lbm_params_init(nx, ny, r, 0.4, 0.02, 0.03, L.F64)
    w = S.rest_weights(S.OracleParams(nx=nx, ny=ny, r=r, gamma=0.4, nu=0.02, u_lid=0.03))
    h = L.Lbm(p, torch_workspace=True)
    h.set_populations(w[:, None, None] + I.noise(5, (9, ny, nx), noise))
    pitch = (nx + 31) // 32 * 32
    base = (-h._ws.data_ptr()) % 256
    g = h._ws[base:base + 9 * pitch * ny * 8].view(torch.float64).reshape(9, ny, pitch)[:, :, :nx].cpu().numpy()
    rho, ux, uy = h.fields()
    h.close()
    p56, p78 = g[5] + g[6], g[7] + g[8]
    want = 1 + ((g[0] + (p56 + p78)) + ((g[1] + g[3]) + (g[2] + g[4])))
    assert np.array_equal(rho, want)
    assert np.array_equal(ux, ((g[1] - g[3]) + ((g[5] - g[6]) + (g[8] - g[7]))) / want)
    assert np.array_equal(uy, r * ((g[2] - g[4]) + (p56 - p78)) / want)
