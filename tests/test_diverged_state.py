"""A handle that diverges inside an lbm_step call: the launches after the residual
step that found it do nothing, so what is read afterwards is the state of that step,
whatever number of steps follow and whichever engine makes them."""
import numpy as np
import pytest

from oracle import stepper as S
from paper_2208_03562_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = pytest.importorskip("paper_2208_03562_gb300.lbm")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    L.load()


def handle(dtype, nx, ny, variant):
    p = L.lbm_params_init(nx, ny, 0.7, 0.4, 0.02, 0.02, dtype)
    w = S.rest_weights(S.OracleParams(nx=nx, ny=ny, r=0.7, gamma=0.4, nu=0.02, u_lid=0.02))
    f = w[:, None, None] + I.noise(nx, (9, ny, nx), 1e-3)
    f[:, 5, 7] = np.nan   # spreads by a node a step; far corners stay finite
    h = L.Lbm(p)
    h.variant = variant
    h.set_populations(f)
    return h


# fused pairs, interior kernel (FP16), cluster engine (pairs, one node a time), general kernel
@pytest.mark.parametrize("dtype,nx,ny,variant", [(L.F32, 400, 100, 0), (L.F16, 400, 100, 0), (L.F32, 128, 120, -2),
                                                 (L.F32, 160, 100, -2), (L.F64, 64, 64, -2), (L.F64, 100, 70, -1),
                                                 (L.F32, 200, 80, -1)])
@pytest.mark.parametrize("calls", [(21,), (22,), (23,), (41,), (17, 5), (22, 22), (22, 1, 2), (40, 2), (7, 20, 30, 2)])
def test_state_of_the_step_that_diverged(dtype, nx, ny, variant, calls):
    a, b = (handle(dtype, nx, ny, variant) for _ in range(2))
    b.step(20)
    want = b.populations()
    assert np.isnan(want).any() and np.isfinite(want).any() and b.info().diverged
    done = 0
    for n in calls:
        a.step(n)
        done += n
    i = a.info()
    assert (i.step, i.residual_step, i.diverged) == (done, 20, 1)
    assert np.array_equal(a.populations(), want, equal_nan=True)
    for f, g in zip(a.fields(), b.fields()):
        assert np.array_equal(f, g, equal_nan=True)
    blob = a.save()
    c = handle(dtype, nx, ny, variant)
    c.step(1)
    c.load(blob)
    c.step(3)
    assert np.array_equal(c.populations(), want, equal_nan=True)
    with pytest.raises(L.LbmError) as e:
        a.mass()
    assert e.value.status == L.EDIVERGED
    # a new start forgets it
    a.set_populations(np.where(np.isnan(want), 0.1, want))
    b.set_populations(np.where(np.isnan(want), 0.1, want))
    a.step(3)
    b.step(1)
    b.step(2)
    assert np.array_equal(a.populations(), b.populations())
    for h in (a, b, c):
        h.close()


def test_run_of_a_diverged_handle():
    a, b = (handle(L.F32, 400, 100, 0) for _ in range(2))
    b.step(20)
    a.step(23)
    for _ in range(2):
        with pytest.raises(L.LbmError) as e:
            a.run(1e-9, 100)
        assert e.value.status == L.EDIVERGED
        assert np.array_equal(a.populations(), b.populations(), equal_nan=True)
    a.close()
    b.close()
