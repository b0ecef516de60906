"""Slots that leave a batch launch of fused pairs of steps on their own: by their
residual, after an odd and an even number of passes, and by the step limit.  The
tolerances come from the residuals of the same slots stepped one at a time, so that
each slot leaves at a chosen residual step.  The kernels that ran are looked up in a
trace of the device."""
import numpy as np
import pytest

from oracle import stepper as S
from paper_2208_03562_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = pytest.importorskip("paper_2208_03562_gb300.lbm")
torch = pytest.importorskip("torch")

SIZES = [(64, 24), (130, 60), (90, 130)]


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    L.load()


def batch(dtype, tols, max_steps):
    b = L.Batch(len(SIZES), dtype)
    for k, (nx, ny) in enumerate(SIZES):
        r, gamma, nu, u = (0.5, 1.0, 1.7)[k], (0.3, 1.0)[k % 2], 0.02, 0.03
        w = S.rest_weights(S.OracleParams(nx=nx, ny=ny, r=r, gamma=gamma, nu=nu, u_lid=u))
        s = b.add(L.lbm_params_init(nx, ny, r, gamma, nu, u, dtype), tols[k], max_steps)
        b.set_populations(s, w[:, None, None] + I.noise(900 + k, (9, ny, nx), 1e-3))
    return b


def kernels(call):
    """Names of the kernels that call() launches (None where the box does not trace)."""
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    names = [e.key for e in prof.key_averages()]
    return names if any("k_" in n for n in names) else None


def ran(names, kernel):
    return names is None or any(kernel in n for n in names)


@pytest.mark.parametrize("dtype", [L.F32, L.F16])
@pytest.mark.parametrize("before", [2, 4])   # 19 and 18 passes to the residual step 40
def test_slots_leave_fused_launches_by_residual_and_limit(dtype, before):
    limit = 70
    h = batch(dtype, [0.0] * 3, limit)
    res = {}
    for t in range(1, 61):
        h.run(1)
        if t % 20 == 0:
            res[t] = [h.query(k)[0].residual for k in range(3)]
    assert res[20][0] > 1.2 * res[40][0] and res[40][1] > 1.2 * res[60][1]
    tols = [(res[20][0] * res[40][0]) ** 0.5, (res[40][1] * res[60][1]) ** 0.5, 0.0]
    a, b = batch(dtype, tols, limit), batch(dtype, tols, limit)
    a.run(before)
    names = kernels(lambda: a.run(limit - before))
    assert ran(names, "k_batch2_tma"), names
    for _ in range(limit):
        b.run(1)
    assert [a.query(k)[1] for k in range(3)] == [L.SLOT_CONVERGED, L.SLOT_CONVERGED, L.SLOT_MAXSTEPS]
    assert [a.query(k)[0].step for k in range(3)] == [40, 60, limit]
    for k in range(3):
        (ia, sa), (ib, sb) = a.query(k), b.query(k)
        assert (sa, ia.step, ia.residual_step, ia.residual, ia.mass) == (sb, ib.step, ib.residual_step, ib.residual,
                                                                         ib.mass)
        assert np.array_equal(a.populations(k), b.populations(k))
        for f, g in zip(a.fields(k), b.fields(k)):
            assert np.array_equal(f, g)


def test_which_launches_are_fused():
    """An odd number of steps, an odd step count and an odd step limit within the
    launch take single steps; a single handle takes pairs in blocks of 20."""
    b = batch(L.F32, [0.0] * 3, 45)
    for n, fused in ((4, True), (3, False), (2, False), (1, False), (20, True), (16, False)):
        names = kernels(lambda: b.run(n))
        if names is None:
            pytest.skip("no trace of the device here")
        assert ran(names, "k_batch2_tma") == fused and ran(names, "k_batch_tma") != fused, (n, names)
    h = L.Lbm(L.lbm_params_init(400, 100, 0.7, 0.4, 0.02, 0.03, L.F32))
    assert ran(kernels(lambda: h.step(20)), "k_step2_tma") and ran(kernels(lambda: h.step(2)), "k_step2_tma")
    names = kernels(lambda: h.step(1))
    assert ran(names, "k_step_tma") and not ran(names, "k_step2_tma")
    h.close()
