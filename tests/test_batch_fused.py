"""Batch launches of whole pairs of steps (two fused steps per pass) against the
same steps one at a time.

A launch of an odd number of steps, or from an odd step count, takes the
single-step body.  Each node goes through the same operations in the same order on
both, and the residual's terms are added up in the same order, so everything is
compared for equality.
"""
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


# tiles are 64 x 24 with a ring of three: one tile and one node less and more, the
# smallest grid, walls a ring or less beyond a tile, interior tiles, odd sizes
SIZES = [(64, 24), (63, 23), (65, 25), (3, 3), (68, 28), (66, 51), (128, 48), (131, 47), (200, 90), (517, 211), (300, 121)]


def batch(dtype, sizes, tol=0.0, max_steps=10 ** 6, noise=1e-3):
    b = L.Batch(len(sizes), dtype)
    for k, (nx, ny) in enumerate(sizes):
        r, gamma, nu, u = (0.5, 1.0, 1.7)[k % 3], (0.3, 1.0)[k % 2], 0.02, 0.03
        w = S.rest_weights(S.OracleParams(nx=nx, ny=ny, r=r, gamma=gamma, nu=nu, u_lid=u))
        s = b.add(L.lbm_params_init(nx, ny, r, gamma, nu, u, dtype), tol, max_steps)
        b.set_populations(s, w[:, None, None] + I.noise(900 + k, (9, ny, nx), noise))
    return b


def same(a, b, n):
    for s in range(n):
        (ia, sa), (ib, sb) = a.query(s), b.query(s)
        assert (sa, ia.step, ia.residual_step) == (sb, ib.step, ib.residual_step), s
        assert (ia.residual, ia.mass) == (ib.residual, ib.mass), s
        assert np.array_equal(a.populations(s), b.populations(s)), s
        for f, g in zip(a.fields(s), b.fields(s)):
            assert np.array_equal(f, g), s


@pytest.mark.parametrize("dtype", [L.F32, L.F16])
def test_pairs_of_steps_equal_single_steps(dtype):
    a, b = batch(dtype, SIZES), batch(dtype, SIZES)
    # an odd number of passes leaves the state in the other set for what follows
    for n, parts in ((2, (1, 1)), (40, (1, 39)), (18, (17, 1)), (62, (31, 31)), (1, (1,)), (3, (3,)), (20, (9, 11))):
        a.run(n)
        for p in parts:
            b.run(p)
        same(a, b, len(SIZES))
    masses = [a.mass(0), b.mass(0)]
    assert masses[0] == masses[1]
    best, ms = a.autotune(4)  # every shape is one CTA of this body to an SM: the largest stands for them
    assert best == a.max_ctas_per_sm and all(m > 0 for m in ms)
    same(a, b, len(SIZES))


@pytest.mark.parametrize("max_steps", [44, 45])
def test_slots_retire_at_the_same_step(max_steps):
    """By the residual (the first slots) and by an even and an odd step limit."""
    sizes, tols = [(64, 24), (130, 60), (90, 130)], 1e-3
    a, b = batch(L.F32, sizes, tols, max_steps), batch(L.F32, sizes, tols, max_steps)
    a.run(60)
    while b.run(1):
        pass
    same(a, b, len(sizes))
    assert a.query(0)[0].step <= max_steps
