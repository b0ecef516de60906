"""Fields in and out of a handle (k_init_fields, k_fields): the integer
conversions between FP64 and FP32, the reciprocal and the shared sums, at values
where they can go wrong (zeros of both signs, subnormal, very small and very
large values, infinities, NaN, ties), against plain FP64 numpy."""
import numpy as np
import pytest

from paper_2208_03562_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = pytest.importorskip("paper_2208_03562_gb300.lbm")

EX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1.0])
EY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1.0])


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    L.load()


def rest(p):
    c2 = min(1.0, p.r) ** 2 / 3
    a, b, cc = c2, c2 / p.r ** 2, c2 * c2 / p.r ** 2
    return np.array([1 - a - b + cc] + [(a - cc) / 2, (b - cc) / 2] * 2 + [cc / 4] * 4)


@pytest.mark.parametrize("nx,ny", [(3, 3), (127, 5), (128, 4), (129, 3)])
@pytest.mark.parametrize("dtype", [L.F64, L.F32, L.F16])
def test_fields_of_special_populations(nx, ny, dtype):
    p = L.lbm_params_init(nx, ny, 0.5, 0.4, 0.02, 0.0, dtype, fx=1e-3, fy=-2e-3, bc=L.BC_PERIODIC)
    h = L.Lbm(p)
    w = rest(p)
    f = w[:, None, None] + I.noise(nx, (9, ny, nx), 1e-2)
    special = [0.0, -0.0, 1e-30, -1e-30, 1e-45, 3e-39, -3e-39, 1.0, 60000.0, 1e30, 1e300, np.inf, -np.inf, np.nan]
    flat = f.reshape(9, -1)
    for k, v in enumerate(special[:min(len(special), nx * ny)]):
        flat[k % 9, k] = v
    h.set_populations(f)
    with np.errstate(all="ignore"):
        g = h.populations() - w[:, None, None]   # stored deviations
        rho = 1 + g.sum(0)
        ux = (np.tensordot(EX, np.where(EX[:, None, None] == 0, 0, g), 1) - p.fx / (2 * p.gamma)) / rho
        uy = (p.r * np.tensordot(EY, np.where(EY[:, None, None] == 0, 0, g), 1) - p.fy / (2 * p.gamma)) / rho
    got = h.fields()
    h.close()
    plain = np.ones(nx * ny, bool)
    plain[:len(special)] = False
    # twelve FP64 roundings of terms of at most about 1, and the 1e-16 of the shift by w
    for a, b in zip(got, (rho, ux, uy)):
        assert np.max(np.abs(a.reshape(-1)[plain] - b.reshape(-1)[plain]), initial=0.0) < 5e-15
        assert np.array_equal(np.isfinite(a), np.isfinite(b))
        fin = np.isfinite(b)
        # special nodes: the sums are ill-conditioned, each population's rounding counts
        assert np.all(np.abs(a[fin] - b[fin]) <= 1e-13 * (1 + np.abs(b[fin]) + np.nanmax(
            np.where(np.isfinite(g), np.abs(g), 0), axis=0)[fin]))


@pytest.mark.parametrize("dtype", [L.F32, L.F16])
def test_init_fields_rounds_to_nearest(dtype):
    """A node at u = 0 stores c drho for known constants: rounded once to FP32
    (then to FP16), for magnitudes from subnormal to large, ties included."""
    nx, ny = 130, 7
    p = L.lbm_params_init(nx, ny, 1.0, 0.5, 0.05, 0.0, dtype)
    rng = I.rng(3)
    mag = 2.0 ** rng.integers(-52, 20, (ny, nx))
    rho = 1 + mag * rng.choice([1.0, 1 + 2.0 ** -24, 1 + 3 * 2.0 ** -24, 1.5, 1 + 2.0 ** -12], (ny, nx))
    z = np.zeros_like(rho)
    h = L.Lbm(p)
    h.init_fields(rho, z, z)
    w = rest(p)
    g = h.populations() - w[:, None, None]
    h.close()
    drho = rho - 1
    for i in range(9):
        want = (w[i] * drho).astype(np.float32)
        eps = 2.0 ** -23
        if dtype == L.F16:
            with np.errstate(over="ignore"):
                want = want.astype(np.float16)
            eps = 2.0 ** -10
        want = want.astype(np.float64)
        fin = np.isfinite(want)
        assert np.array_equal(fin, np.isfinite(g[i]))
        # one unit in the last place (the FP64 values differ in their last bits), FP16's smallest step, and
        # the rounding of the shift by w
        assert np.all(np.abs(g[i][fin] - want[fin]) <= eps * np.abs(want[fin]) + 2.0 ** -24 * (dtype == L.F16) + 2.3e-16)


def test_init_fields_of_nan_and_infinity():
    h = L.Lbm(L.lbm_params_init(40, 9, 0.5, 0.5, 0.02, 0.0, L.F32))
    rho, ux, uy = np.ones((9, 40)), np.zeros((9, 40)), np.zeros((9, 40))
    rho[2, 3], ux[4, 5], uy[6, 7], ux[0, 39] = np.nan, np.nan, np.inf, 1e200
    h.init_fields(rho, ux, uy)
    bad = ~np.isfinite(h.populations()).all(0)
    h.close()
    assert sorted(map(tuple, np.argwhere(bad))) == [(0, 39), (2, 3), (4, 5), (6, 7)]
