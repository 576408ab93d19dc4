"""alpha of FP64 FORMULA steps against 50-digit arithmetic, up to and across
the end of the FP64 series' range (max |x| = 1/48): one-node lattices, whose
alpha the statistics return in FP64.

Tolerance 2^-47 = 64 u, u = 2^-53: with x off by a few u of f and the terms of
Delta H(2) summed in FP64, the logarithm form is off by ~15 u in these states
and at most 200 u (100 u M_2 over Delta H(2) - Delta H(1) >= M_2 / 2)."""
import os
from decimal import Decimal, getcontext

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


def _alpha(f, c, d):
    """Eqs. (8) and (9) of the populations f in 50 digits, and max |x|."""
    getcontext().prec = 50
    f = [Decimal(float(v)) for v in f]
    rho = sum(f)
    fe = []
    for k in range(len(f)):
        v = rho
        for a in range(d):
            v *= Decimal(2) / 3 if c[k][a] == 0 else Decimal(1) / 6
        fe.append(v)
    for a in range(d):
        u = sum(int(c[k][a]) * f[k] for k in range(len(f))) / rho
        s = 3 * u * u / (1 + (1 + 3 * u * u).sqrt())
        psi = {0: 1 - s, 1: 1 + 3 * u + 2 * s, -1: 1 - 3 * u + 2 * s}
        fe = [fe[k] * psi[int(c[k][a])] for k in range(len(f))]
    x = [e / v - 1 for e, v in zip(fe, f)]
    ln = [(1 + y).ln() for y in x]
    d1 = sum(v * (m - y) for v, y, m in zip(f, x, ln))
    b = sum(v * y * m for v, y, m in zip(f, x, ln))
    d2 = sum(v * ((1 + 2 * y) * (1 + 2 * y).ln() - 2 * y)
             for v, y in zip(f, x)) - 2 * b
    return (Decimal(2) if d2 <= 0 else 2 - d2 / (d2 - d1),
            float(max(abs(y) for y in x)))


@pytest.mark.parametrize("amp", [1e-9, 1e-6, 1e-4, 3e-3, 0.012, 0.016, 0.02,
                                 0.024, 0.028])
@pytest.mark.parametrize("lat", ["D2Q9", "D3Q27"])
def test_alpha_fp64(elbm, lat, amp):
    import oracle
    c, w = oracle.lattice(lat)
    d = oracle.dim(lat)
    rng = np.random.default_rng(11)
    g = elbm.Lattice(lat, 1, 1, 1, nu=1e-3, dtype="fp64")
    g.set_diagnostics(diag_every=1)
    formula = 0
    for _ in range(32):
        u = 0.1 * rng.uniform(-1, 1, d)
        f = w.copy()
        for a in range(d):
            s = 3 * u[a] ** 2 / (1 + np.sqrt(1 + 3 * u[a] ** 2))
            ca = c[:, a]
            f = f * np.where(ca == 0, 1 - s, 1 + 3 * ca * u[a] + 2 * s)
        f = f * (1 + amp * rng.uniform(-1, 1, len(w)))
        g.set_populations(f.reshape(-1, 1, 1, 1))
        f = g.populations().ravel()
        g.step(1, "formula")
        want, x = _alpha(f, c, d)
        got = g.entropy_stats()["alpha_min"]
        assert abs(Decimal(got) - want) <= Decimal(2) ** -47, (x, got, want)
        formula += want != 2
    assert formula > 0
