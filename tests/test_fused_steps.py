"""The fused two-step kernel (k_step2_tma) against single steps.

Both make the same operations per node, the rounding of the stored populations
between the steps included, so the populations must be bitwise the same; the
residual and the mass differ by the order of their FP64 sums only.  Grids at the
edges of the tiles (64 x 32, and 64 x 16 for grids of few tiles): a tile or less,
one node more or less than whole tiles, remainders that end inside the rings of
the neighbouring tile."""
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


SMALL = [(70, 12), (71, 13), (128, 16), (129, 17), (127, 15), (130, 18), (131, 19), (132, 20), (192, 35), (195, 67),
         (70, 200), (1000, 14), (257, 131)]
LARGE = [(1280, 1024), (1283, 1027), (1219, 1057), (4099, 317)]


@pytest.mark.parametrize("nx,ny", SMALL + LARGE)
def test_fused_steps_equal_single_steps_bitwise(nx, ny):
    u = 0.03
    a, b = (L.Lbm(L.lbm_params_init(nx, ny, 0.7, 0.3, 0.02, u, L.F32)) for _ in range(2))
    fields = I.random_fields(nx + ny, nx, ny, 5e-3, 0.3 * u)
    for h in (a, b):
        h.variant = 0
        h.init_fields(*fields)
    done = 0
    for n in (1, 2, 5, 12, 20, 3, 40, 17):  # odd starts, whole blocks of 20, a fused residual step off a block
        a.step(n)
        for _ in range(n):
            b.step(1)
        done += n
        assert np.array_equal(a.populations(), b.populations()), done
        ia, ib = a.info(), b.info()
        assert (ia.step, ia.residual_step) == (ib.step, ib.residual_step) == (done, done // 20 * 20)
        if ia.residual_step:
            # FP32 pair sums of up to 5e6 terms: 48 bits, then FP64
            assert abs(ia.residual - ib.residual) <= 1e-11 * ib.residual
            assert abs(ia.mass - ib.mass) <= 1e-12 * ib.mass
    # a checkpoint taken after an odd number of fused launches resumes bitwise
    a.step(2)
    blob = a.save()
    a.step(20)
    want = a.populations()
    a.load(blob)
    a.step(20)
    assert np.array_equal(a.populations(), want)
    # another engine continues from the same set
    a.variant = L.VARIANT_GENERAL
    b.step(22)
    a.step(3)
    b.step(3)
    assert np.array_equal(a.populations(), b.populations())
    a.close()
    b.close()


def test_run_stops_where_single_steps_stop():
    p = L.lbm_params_init(320, 160, 0.5, 0.5, 0.05, 0.02, L.F32)
    a, g = L.Lbm(p), L.Lbm(p)
    a.variant, g.variant = 0, L.VARIANT_GENERAL
    a.step(3)
    g.step(3)
    ra, rg = a.run(2e-3, 20000), g.run(2e-3, 20000)
    assert ra == rg and ra[0] == L.OK and (3 + ra[1]) % 20 == 0
    assert np.array_equal(a.populations(), g.populations())
    a.step(7)
    g.step(7)
    assert np.array_equal(a.populations(), g.populations())
