"""One step of the FP64-arithmetic stream-collide kernel on odd sizes beyond
one grid pass (128-thread blocks, several nodes per thread, a ragged tail) and
around the change from one-warp blocks, every storage, near and far nodes
(max |x| above and below the series' range) in the same warps.

Reference: the step of the stored state in vectorised FP64 with logarithms.
Tolerances, per population: FORMULA FP64 1e-12 f; ROOT and SECANT 1e-9 of the
largest f (a stop-rule edge within rounding moves alpha by the width of the
stop interval); FP32 storage adds alpha's rounding down, 2^-22 |n|, and the
stored value's, 2^-23 of it; binary16 2^-10 of the stored deviation plus its
smallest step 2^-24."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def elbm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1904_00866_gb300 as e
    if not os.path.exists(e.LIB_PATH):
        import __graft_entry__ as g
        g.build()
    e.lib()
    return e


def _phi(y):
    p = np.full_like(y, -1 / 272)
    for k in range(16, 1, -1):
        p = p * y + (-1.0) ** k / (k * (k - 1))
    z = np.maximum(1 + y, 1e-300)
    return np.where(np.abs(y) < 0.1, y * y * p, z * np.log(z) - y)


def _alpha(f, x, mode):
    with np.errstate(divide="ignore"):
        amax = np.where(x < 0, -1 / x, np.inf).min(0)
    ln = np.log1p(x)
    b, d1 = (f * x * ln).sum(0), (f * (ln - x)).sum(0)

    def dh(a):
        return (f * _phi(a * x)).sum(0) - a * b

    if mode == "root":
        lo, hi = np.ones_like(amax), amax.copy()
        a, todo = hi.copy(), dh(hi) > 0
        for _ in range(64):
            mid = 0.5 * (lo + hi)
            d = dh(mid)
            done = todo & (d >= -1e-13) & (d <= 0)
            a = np.where(done, mid, a)
            todo &= ~done
            hi = np.where(todo & (d > 0), mid, hi)
            lo = np.where(todo & ~(d > 0), mid, lo)
        return np.where(todo, lo, a)
    star = np.minimum(2, amax)
    ds = dh(star)
    if mode == "secant":
        a, da, go = np.ones_like(star), d1, np.ones(star.shape, bool)
        for _ in range(4):
            an = star + ds / (ds - da) * (a - star)
            dn = dh(an)
            go &= ~(dn > 0)
            a, da = np.where(go, an, a), np.where(go, dn, da)
            go &= ~(da >= -1e-13)
    else:
        a = star + ds / (ds - d1) * (1 - star)
    return np.where(ds <= 0, star, np.where(ds - d1 > 0, a, 1.0))


SIZES = [("D2Q9", (1, 139, 140)), ("D2Q9", (1, 331, 257)),
         ("D3Q27", (26, 27, 28)), ("D3Q27", (47, 43, 41))]


@pytest.mark.parametrize("dtype,mode", [
    ("fp64", "formula"), ("fp64", "root"), ("fp64", "secant"),
    ("fp32_shifted", "root"), ("fp32_shifted", "secant"), ("fp32", "root"),
    ("fp16_shifted", "secant"), ("fp16_shifted", "root")])
@pytest.mark.parametrize("far", [0.0, 0.02, 0.6])
@pytest.mark.parametrize("lat,shape", SIZES)
def test_one_step(elbm, lat, shape, far, dtype, mode):
    import oracle
    c, w = oracle.lattice(lat)
    d = oracle.dim(lat)
    nz, ny, nx = shape
    rng = np.random.default_rng([nx, int(100 * far)])
    nu = 1e-3
    g = elbm.Lattice(lat, nx, ny, nz, nu=nu, dtype=dtype)
    g.init_fields(1 + 0.02 * rng.uniform(-1, 1, shape),
                  0.1 * rng.uniform(-1, 1, (d,) + shape))
    f = g.populations()
    amp = np.where(rng.uniform(0, 1, shape) < far, 0.2,
                   10 ** rng.uniform(-4, -1.8, shape))
    g.set_populations(f * (1 + amp * rng.uniform(-1, 1, f.shape)))
    f = g.populations()
    rho = f.sum(0)
    fe = rho * w.reshape(-1, 1, 1, 1)
    for a in range(d):
        ca = c[:, a].reshape(-1, 1, 1, 1)
        u = (ca * f).sum(0) / rho
        s = 3 * u * u / (1 + np.sqrt(1 + 3 * u * u))
        fe = fe * np.where(ca == 0, 1 - s, 1 + 3 * ca * u + 2 * s)
    n = fe - f
    x = n / f
    xm = np.abs(x).max(0)
    assert np.mean(xm > 1 / 32) >= 0.8 * far and np.any(xm < 1 / 48)
    alpha = _alpha(f, x, mode)
    want = f + alpha / (6 * nu + 1) * n
    g.set_diagnostics(diag_every=1, alpha_map_every=1)
    g.step(1, mode)
    st = g.entropy_stats()
    assert st["n_nodes"] == g.n and st["n_degenerate"] == 0
    got = g.populations()
    tol = np.abs(want) * 1e-12
    if mode != "formula":
        tol += 1e-9 * np.abs(want).max()
    dev = np.abs(want - w.reshape(-1, 1, 1, 1) * g.rho0)
    if dtype != "fp64":
        tol += 2.0 ** -22 * np.abs(n)
    if dtype == "fp32":
        tol += 2.0 ** -23 * np.abs(want)
    elif dtype == "fp32_shifted":
        tol += 2.0 ** -23 * dev
    elif dtype == "fp16_shifted":
        tol += 2.0 ** -10 * dev + 2.0 ** -24
    for i in range(len(w)):
        shift = (-c[i, 2], -c[i, 1], -c[i, 0])
        post = np.roll(got[i], shift, (0, 1, 2))
        assert np.all(np.abs(post - want[i]) <= tol[i]), i
    m = np.array([f.sum(), *(c[:, :d].T.astype(float) @ f.reshape(
        len(w), -1)).sum(1)])
    assert abs(st["mass"] - m[0]) <= 1e-12 * m[0]
    assert np.all(np.abs(np.array(st["momentum"][:d]) - m[1:]) <= 1e-12 * m[0])
    assert abs(st["alpha_sum"] - alpha.sum()) <= 1e-6 * alpha.sum()
