"""lbm_batch_autotune where a launch makes whole pairs of steps: its grid is one CTA
to an SM whatever the launch shape, so the shape set for other launches must stay,
and only launches that depend on it are tuned."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L = pytest.importorskip("paper_2208_03562_gb300.lbm")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    L.load()


@pytest.mark.parametrize("dtype", [L.F32, L.F16])
def test_pairs_of_steps_leave_the_launch_shape(dtype):
    b = L.Batch(3, dtype)
    for nx, ny in ((300, 200), (130, 64), (64, 24)):
        b.add(L.lbm_params_init(nx, ny, 0.7, 0.4, 0.02, 0.03, dtype), 0.0, 10 ** 6)
    b.run(2)
    before = [b.populations(k) for k in range(3)]
    most = b.max_ctas_per_sm
    assert most > 1
    for choice in range(most + 1):        # 0: the maximum
        b.ctas_per_sm = choice
        best, ms = b.autotune(4)
        assert best == b.ctas_per_sm == (choice or most)
        assert len(ms) == most and ms[0] > 0 and all(m == ms[0] for m in ms)
    b.ctas_per_sm = 0
    best, ms = b.autotune(5)              # single steps: every shape is timed
    assert ms[best - 1] == min(ms) > 0 and b.ctas_per_sm == best
    for k in range(3):
        assert np.array_equal(b.populations(k), before[k]) and b.query(k)[0].step == 2
