"""Nodes at equilibrium to FP64 rounding, in the FP64-arithmetic kernels: the
logarithm form decides them, whatever else the kernel does.

A fluid at rest: f_i = fl(W_i rho), and the logarithm form finds
f^eq == f (n_degenerate, alpha = 2) exactly where no fl(fl(sum f) W_i) lies
below f_i; at u = 0 these are all its operations, so the expected count is
formed here with the same FP64 operations in the same order.

Initialised flows: one step with the FP64 entropy check and one without give
the same populations, alpha maps and counters, bit for bit."""
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


SHAPES = [("D2Q9", (1, 7, 9)), ("D3Q27", (3, 4, 5))]


@pytest.mark.parametrize("mode", ["formula", "root", "secant"])
@pytest.mark.parametrize("rho", [1.0, 1.1, 0.9, 1.7, 3.3, 0.07, 12.9])
@pytest.mark.parametrize("lat,shape", SHAPES)
def test_fluid_at_rest(elbm, lat, shape, rho, mode):
    nz, ny, nx = shape
    d = 2 if lat == "D2Q9" else 3
    g = elbm.Lattice(lat, nx, ny, nz, nu=1e-3, dtype="fp64")
    g.init_fields(np.ones(shape), np.zeros((d,) + shape))
    w = g.populations()[:, 0, 0, 0]          # fl(W_i 1)
    g.init_fields(np.full(shape, rho), np.zeros((d,) + shape))
    f = g.populations()[:, 0, 0, 0]
    assert np.array_equal(f, w * rho)
    s = 0.0
    for v in f:
        s += v
    equal = all(s * wi >= fi for wi, fi in zip(w, f))
    g.set_diagnostics(diag_every=1)
    g.step(1, mode)
    st = g.entropy_stats()
    assert st["n_nodes"] == g.n
    assert st["n_degenerate"] == (g.n if equal else 0)


@pytest.mark.parametrize("mode", ["formula", "root", "secant"])
@pytest.mark.parametrize("umax", [0.0, 0.05, 0.24])
@pytest.mark.parametrize("uniform", [True, False])
@pytest.mark.parametrize("lat,shape", SHAPES)
def test_first_step_and_checked_first_step(elbm, lat, shape, uniform, umax,
                                           mode):
    nz, ny, nx = shape
    d = 2 if lat == "D2Q9" else 3
    rng = np.random.default_rng(7)
    one = (1,) * 3 if uniform else shape
    rho = np.ones(shape) + 0.02 * rng.uniform(-1, 1, one)
    u = np.zeros((d,) + shape) + umax * rng.uniform(-1, 1, (d,) + one)
    got = []
    for check in (0, 1):
        g = elbm.Lattice(lat, nx, ny, nz, nu=1e-3, dtype="fp64")
        g.set_diagnostics(diag_every=1, check_every=check, alpha_map_every=1)
        g.init_fields(rho, u)
        g.step(1, mode)
        s = g.entropy_stats()
        got.append((g.populations(), g.alpha_map(), [
            s[k] for k in ("n_nodes", "n_degenerate", "n_accept_two",
                           "n_accept_star", "n_formula", "n_root_iters",
                           "n_no_root", "alpha_min", "alpha_max")]))
    assert np.array_equal(got[0][0], got[1][0])
    assert np.array_equal(got[0][1], got[1][1])
    assert got[0][2] == got[1][2]
