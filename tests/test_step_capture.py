"""Steps that a caller captures into a CUDA graph of its own.  An even number of
steps ends in the buffer that it started from, so k replays advance the state by
k times as many steps, on every engine; blocks of 20 steps are captured like any
other."""
import numpy as np
import pytest

from paper_2208_03562_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = pytest.importorskip("paper_2208_03562_gb300.lbm")
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    L.load()


# fused pairs (400x100, 1023x511), cluster engine (128x128), general kernel (the rest)
@pytest.mark.parametrize("dtype,nx,ny,bc", [(L.F32, 400, 100, L.BC_CAVITY), (L.F32, 1023, 511, L.BC_CAVITY),
                                            (L.F32, 128, 128, L.BC_CAVITY), (L.F64, 64, 64, L.BC_CAVITY),
                                            (L.F16, 512, 257, L.BC_CAVITY), (L.F32, 256, 65, L.BC_CHANNEL)])
@pytest.mark.parametrize("before,n", [(0, 2), (0, 4), (1, 2), (17, 2), (18, 6), (0, 20), (3, 38), (0, 42)])
def test_replays_of_captured_steps(dtype, nx, ny, bc, before, n):
    p = L.lbm_params_init(nx, ny, 0.7, 0.3, 0.02, 0.02, dtype, bc=bc)
    fields = I.random_fields(nx + n, nx, ny, 5e-3, 0.01)
    a, b = L.Lbm(p), L.Lbm(p)
    stream = torch.cuda.Stream()
    for h in (a, b):
        h.init_fields(*fields)
        h.step(before)
    assert L.load().lbm_set_stream(a.h, stream.cuda_stream) == L.OK
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        a.step(n)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    b.step(3 * n)
    assert np.array_equal(a.populations(), b.populations())
    a.step(5)  # the handle goes on from where the replays ended
    b.step(5)
    assert np.array_equal(a.populations(), b.populations())
    a.close()
    b.close()
