"""Engines of small grids at the edges of their ranges.

The cluster engine's two-nodes-per-thread kernel (FP32 / FP16) resolves pulls,
walls and seams into addresses once per launch; the FP64 general kernel cuts
small grids into smaller tiles.  Both make the operations of the general body in
the same order, so populations are compared bitwise between the engines."""
import numpy as np
import pytest

from paper_2208_03562_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = pytest.importorskip("paper_2208_03562_gb300.lbm")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    L.load()


def compare(nx, ny, dtype, bc, drho, fx, model, steps=(1, 20, 23)):
    u = 0.02
    p = L.lbm_params_init(nx, ny, 0.7, 0.4, 0.02, u, dtype, bc=bc, drho=drho, fx=fx, fy=-0.5 * fx, model=model)
    a, b = L.Lbm(p), L.Lbm(p)
    a.variant, b.variant = L.VARIANT_CLUSTER, L.VARIANT_GENERAL
    f = I.random_fields(7 * nx + ny, nx, ny, 5e-3, 0.3 * u)
    for h in (a, b):
        h.init_fields(*f)
    for n in steps:
        a.step(n)
        b.step(n)
        assert np.array_equal(a.populations(), b.populations()), n
    ia, ib = a.info(), b.info()
    assert ia.residual_step == ib.residual_step == 40
    assert abs(ia.residual - ib.residual) <= 1e-9 * ib.residual
    a.close()
    b.close()


# slabs of 1 to 1024 nodes: odd node counts, a short last slab, rows wider than half the threads (more ring
# nodes than threads), 512 x 2 rows (exactly two nodes per thread), one slab only
SLABS = [(3, 3), (4, 5), (33, 47), (101, 150), (128, 128), (512, 32), (511, 31), (300, 45), (73, 200), (340, 3)]


@pytest.mark.parametrize("nx,ny", SLABS)
@pytest.mark.parametrize("bc", [L.BC_CAVITY, L.BC_CHANNEL, L.BC_PERIODIC])
@pytest.mark.parametrize("dtype", [L.F32, L.F16])
def test_cluster_pairs_equal_general(nx, ny, bc, dtype):
    compare(nx, ny, dtype, bc, L.DRHO_CURRENT, 0.0, L.MODEL_PRC)


@pytest.mark.parametrize("drho", [L.DRHO_CURRENT, L.DRHO_OFF])
@pytest.mark.parametrize("fx", [0.0, 2e-6])
@pytest.mark.parametrize("model", [L.MODEL_PRC, L.MODEL_PRNR])
def test_cluster_pairs_every_scheme(drho, fx, model):
    compare(97, 101, L.F32, L.BC_CHANNEL, drho, fx, model)


@pytest.mark.parametrize("nx,ny", [(8, 4), (9, 5), (64, 64), (65, 33), (100, 150), (127, 90)])
@pytest.mark.parametrize("bc", [L.BC_CAVITY, L.BC_PERIODIC])
def test_fp64_small_tiles_equal_cluster(nx, ny, bc):
    compare(nx, ny, L.F64, bc, L.DRHO_CURRENT, 1e-6 if bc == L.BC_PERIODIC else 0.0, L.MODEL_PRC)


@pytest.mark.parametrize("nx,ny", [(64, 64), (100, 150), (33, 9), (300, 47)])
@pytest.mark.parametrize("variant", [L.VARIANT_GENERAL, L.VARIANT_CLUSTER])
@pytest.mark.parametrize("dtype", [L.F64, L.F32])
def test_mass_between_residual_steps(nx, ny, variant, dtype):
    """lbm_mass sums the current state only, whatever partial sums a residual
    step left in the workspace."""
    h = L.Lbm(L.lbm_params_init(nx, ny, 0.7, 0.4, 0.02, 0.02, dtype, bc=L.BC_CHANNEL, fx=1e-5))
    h.variant = variant
    f = I.random_fields(nx, nx, ny, 5e-2, 5e-3)
    h.init_fields(*f)
    h.step(23)
    # sums of nx ny values of about 1: numpy's and the library's order differ
    assert abs(h.mass() - h.populations().sum()) <= 1e-13 * nx * ny * 10
    assert abs(h.info().mass - f[0].sum()) <= (1e-12 if dtype == L.F64 else 1e-7) * nx * ny
    h.close()


@pytest.mark.parametrize("nx,ny", [(64, 64), (100, 150), (33, 9), (300, 47), (512, 128)])
def test_fp64_sums_do_not_depend_on_the_tile(nx, ny):
    """Small tiles sum the rows of the 32 x 8 tiling, so a single handle's
    residual is bitwise that of a batch slot, which keeps 32 x 8 tiles."""
    p = L.lbm_params_init(nx, ny, 0.7, 0.4, 0.02, 0.02, L.F64)
    h, b = L.Lbm(p), L.Batch(1, L.F64)
    h.variant = L.VARIANT_GENERAL
    s = b.add(p, 0.0, 10 ** 6)
    h.init_fields(*I.random_fields(nx, nx, ny, 5e-3, 5e-3))
    b.set_populations(s, h.populations())
    h.set_populations(b.populations(s))
    for _ in range(2):
        h.step(20)
        b.run(20)
        info = b.query(s)[0]
        assert info.residual == h.residual() and info.mass == h.info().mass
    h.close()
    b.close()
