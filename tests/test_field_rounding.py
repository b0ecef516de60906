"""What k_init_fields stores, compared bit by bit: the equilibria of Eq. 12 formed in
FP64 as they are written, rounded once to FP32 (then to FP16).

The FP64 values of two orders of operations differ in their last bits, so each
reference value carries a bound E on its own error, and a stored value has to lie
between the rounded ref - E and the rounded ref + E: the same number but where the
reference itself is next to a midpoint.  A population is a sum of at most four
moments, each a product or a sum of products of at most eight roundings, each of
2^-53 of the largest moment: E = 64 x 2^-53 of that moment."""
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


def equilibria(r, gamma, rho, ux, uy):
    """Rest-shifted populations of Eq. 12 and the bound on their error."""
    c2, ig, ir = min(1.0, r) ** 2 / 3, 1 / gamma, 1 / r
    d = rho - 1
    d10, d01, d11 = rho * ux, rho * uy, rho * ux * uy * ig
    d20, d02 = c2 * d + rho * ux * ux * ig, c2 * d + rho * uy * uy * ig
    d21, d12 = rho * (c2 + ux * ux * ig * ig) * uy, rho * (c2 + uy * uy * ig * ig) * ux
    d22 = c2 * c2 * d + rho * c2 * (ux * ux + uy * uy) + rho * ux * ux * uy * uy
    e01, e02, e11, e21, e12, e22 = d01 * ir, d02 * ir * ir, d11 * ir, d21 * ir, d12 * ir * ir, d22 * ir * ir
    f = np.stack([d - d20 - e02 + e22, 0.5 * (d10 + d20 - e12 - e22), 0.5 * (e01 + e02 - e21 - e22),
                  0.5 * (-d10 + d20 + e12 - e22), 0.5 * (-e01 + e02 + e21 - e22), 0.25 * (e11 + e21 + e12 + e22),
                  0.25 * (-e11 + e21 - e12 + e22), 0.25 * (e11 - e21 - e12 + e22), 0.25 * (-e11 - e21 + e12 + e22)])
    top = np.max(np.abs(np.stack([d, d10, d01, d11, d20, d02, d21, d12, d22, e01, e02, e11, e21, e12, e22])), axis=0)
    return f, 64 * 2.0 ** -53 * top


def stored(p, fields):
    """The handle's populations as they lie in memory, and its snapshot of u_x."""
    h = L.Lbm(p, torch_workspace=True)
    h.init_fields(*fields)
    pitch, half = (p.nx + 31) // 32 * 32, p.dtype == L.F16
    base = (-h._ws.data_ptr()) % 256
    n = 9 * pitch * p.ny
    raw = h._ws[base:base + n * (2 if half else 4)].view(torch.float16 if half else torch.float32)
    f = raw.reshape(9, p.ny, pitch)[:, :, :p.nx].cpu().numpy()
    at = base + 2 * (-(-n * (2 if half else 4) // 256) * 256)
    snap = h._ws[at:at + 4 * pitch * p.ny].view(torch.float32).reshape(p.ny, pitch)[:, :p.nx].cpu().numpy()
    h.close()
    return f, snap


def narrowed(v, dtype):
    with np.errstate(over="ignore", under="ignore"):
        v = v.astype(np.float32)
        return v.astype(np.float16) if dtype == L.F16 else v


def check(p, fields):
    f, snap = stored(p, fields)
    ref, err = equilibria(p.r, p.gamma, *fields)
    lo, hi = narrowed(ref - err, p.dtype), narrowed(ref + err, p.dtype)
    bad = ~((lo <= f) & (f <= hi))
    assert not bad.any(), (np.argwhere(bad)[:4], f[bad][:4], lo[bad][:4], hi[bad][:4])
    assert np.array_equal(snap, fields[1].astype(np.float32))   # ties to even included
    return ref, lo == hi


def params(dtype, nx=257, ny=256, r=0.7, gamma=0.3):
    return L.lbm_params_init(nx, ny, r, gamma, 0.05, 0.0, dtype)


@pytest.mark.parametrize("r,gamma", [(1.0, 1.0), (0.5, 0.25), (1.7, 0.6)])
@pytest.mark.parametrize("dtype", [L.F32, L.F16])
def test_random_flow_is_rounded_once(dtype, r, gamma):
    p = params(dtype, r=r, gamma=gamma)
    fields = list(I.random_fields(11, p.nx, p.ny, 1e-2, 0.05))
    # u_x on midpoints of FP32 numbers (the snapshot)
    m = np.float32(0.03) * (1 + np.arange(p.nx) * 2.0 ** -20)
    fields[1][3] = m.astype(np.float32).astype(np.float64) + 2.0 ** -30
    _, same = check(p, fields)
    assert same.mean() > 0.999


@pytest.mark.parametrize("dtype", [L.F32, L.F16])
@pytest.mark.parametrize("i", range(9))
def test_next_to_midpoints(dtype, i):
    """Densities that put population i on and a few 2^-53 beside a midpoint between
    FP32 numbers (at u = 0, where f_i is w_i drho)."""
    p = params(dtype)
    w = equilibria(p.r, p.gamma, np.float64(2.0), 0.0, 0.0)[0][i]
    rng = I.rng(50 + i)
    v = (w * rng.uniform(0.05, 0.4, (p.ny, p.nx))).astype(np.float32)
    mid = 0.5 * (v.astype(np.float64) + np.nextafter(v, np.float32(1)).astype(np.float64))
    off = rng.integers(-400, 401, v.shape) * 2.0 ** -52 / w
    rho = 1 + (mid / w + off)
    z = np.zeros_like(rho)
    ref, same = check(p, (rho, z, z))
    near = np.abs(ref[i] - mid) < 2.0 ** -43      # 400 x 2^-52 and the rounding of rho
    assert near.mean() > 0.9 and (near & same[i]).mean() > 0.5


@pytest.mark.parametrize("dtype", [L.F32, L.F16])
def test_nodes_at_rest_among_others(dtype):
    p = params(dtype)
    rng = I.rng(8)
    fields = I.random_fields(12, p.nx, p.ny, 1e-2, 0.05)
    at_rest = rng.random(fields[0].shape) < 0.5
    at_rest[100:140] = True                       # whole warps
    sign = rng.choice([0.0, -0.0], fields[0].shape)
    fields = [np.where(at_rest, v, f) for v, f in zip((1.0, sign, -sign), fields)]
    fields[1][200:] = 0.0                         # one component only
    check(p, fields)
    f, _ = stored(p, fields)
    zero = f[:, at_rest]
    assert not zero.any() and not np.signbit(zero).any()
    # and out again: exactly at rest
    h = L.Lbm(p)
    h.init_fields(*fields)
    rho, ux, uy = h.fields()
    h.close()
    assert np.all(rho[at_rest] == 1) and not ux[at_rest].any() and not uy[at_rest].any()


def best_ms(call, n=10):
    best = np.inf
    for _ in range(n):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        call()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("dtype", [L.F32, L.F16])
def test_a_fluid_at_rest_costs_no_more(dtype):
    """Zeros take no slower form of the transfers than other values: measured
    2.9 and 1.3 times where zeros took the conversion instructions."""
    nx, ny = 4096, 2048
    h = L.Lbm(L.lbm_params_init(nx, ny, 0.5, 0.5, 0.05, 0.01, dtype))
    g = torch.Generator(device="cuda").manual_seed(2)
    moving = [1e-2 * torch.randn((ny, nx), dtype=torch.float64, device="cuda", generator=g) for _ in range(3)]
    moving[0] += 1.0
    zero = torch.zeros_like(moving[0])
    out = [torch.empty_like(zero) for _ in range(3)]
    t = {}
    for name, f in (("moving", moving), ("rest", [zero + 1, zero, zero]), ("u=0", [moving[0], zero, zero])):
        torch.cuda.synchronize()
        t[name] = (best_ms(lambda: L.load().lbm_init_fields(h.h, *[v.data_ptr() for v in f], 1)),
                   best_ms(lambda: L.lbm_fields_device(h.h, *[v.data_ptr() for v in out])))
    h.close()
    for name in ("rest", "u=0"):
        assert t[name][0] < 1.15 * t["moving"][0] and t[name][1] < 1.15 * t["moving"][1], t


@pytest.mark.parametrize("dtype", [L.F32, L.F16])
def test_very_slow_flow_is_rounded_once(dtype):
    """Populations around the smallest normal FP32 number, subnormal ones among them."""
    p = params(dtype)
    g = I.rng(4)
    u = [2.0 ** g.uniform(-132, -118, (p.ny, p.nx)) * g.choice([-1, 1], (p.ny, p.nx)) for _ in range(2)]
    check(p, (np.ones((p.ny, p.nx)), *u))
