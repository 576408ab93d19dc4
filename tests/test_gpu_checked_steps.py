"""The FP64 entropy check judges the alpha that ordinary steps use: steps with
check_every = 1 and steps without it take the same arithmetic, so their
populations, alpha maps and counters agree bit for bit, and the check finds no
violation of Eq. (7) and the FP64 FORMULA's alpha.

Near-equilibrium nodes and, for the FP64-arithmetic kernels, a tenth of the
nodes far from it (the logarithm form), on sizes with one and with several
nodes per thread.  The FP32 / FP16 FORMULA gets flows without far nodes: those
take the logarithms one per lane under the check, so that a tie is not counted
as a mismatch, and one per warp otherwise.

alpha_dev_max: FORMULA in FP64 within 1e-12 of the check's own logarithm form
(the two forms are off by 1e-15 and 3e-15 near equilibrium; at |x| ~ 1e-3 and
1e-15 of M_2 it compares rounding), with alpha rounded down to FP32 2^-22."""
import os

import numpy as np
import pytest

import elbm_workloads as W

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


COUNTS = ("n_nodes", "n_accept_two", "n_accept_star", "n_formula",
          "n_degenerate", "n_root_iters", "n_root_cap", "n_no_root", "n_band",
          "n_far", "alpha_min", "alpha_max")


@pytest.mark.parametrize("dtype,mode", [
    ("fp64", "formula"), ("fp64", "root"), ("fp64", "secant"),
    ("fp32_shifted", "root"), ("fp32", "secant"), ("fp16_shifted", "root"),
    ("fp32_shifted", "formula"), ("fp32", "formula"),
    ("fp16_shifted", "formula")])
@pytest.mark.parametrize("lat,shape", [
    ("D2Q9", (1, 23, 37)), ("D2Q9", (1, 331, 257)), ("D3Q27", (11, 13, 19)),
    ("D3Q27", (47, 43, 41))])
def test_checked_steps(elbm, lat, shape, dtype, mode):
    nz, ny, nx = shape
    if lat == "D2Q9":
        rho, u = W.random_phase_2d(nx, seed=3, umax=0.1, ny=ny)
    else:
        rho, u = W.random_phase_3d(nx, seed=3, umax=0.1, ny=ny, nz=nz)
    far = dtype == "fp64" or mode != "formula"
    first = []
    for check in (0, 1):
        g = elbm.Lattice(lat, nx, ny, nz, nu=2e-4, dtype=dtype)
        g.init_fields(rho, u)
        g.set_diagnostics(diag_every=0)
        g.step(3, "formula")
        if far:
            rng = np.random.default_rng(4)
            f = g.populations()
            f *= 1 + 0.2 * rng.uniform(-1, 1, f.shape) * (
                rng.uniform(0, 1, f.shape[1:]) < 0.1)
            g.set_populations(f)
        g.set_diagnostics(diag_every=1, check_every=check, alpha_map_every=1)
        got = []
        for _ in range(1 if far else 3):
            g.step(1, mode)
            s = g.entropy_stats()
            assert s["checked"] == check
            if check:
                assert s["n_violations"] == 0
                if mode == "formula":
                    assert s["n_decision_mismatch"] == 0
                    assert s["alpha_dev_max"] <= (
                        1e-12 if dtype == "fp64" else 2.0 ** -16 + 2.0 ** -22)
            got.append((g.populations(), g.alpha_map(),
                        [s[k] for k in COUNTS]))
        if first:
            for (f0, a0, c0), (f1, a1, c1) in zip(first, got):
                assert np.array_equal(f0, f1)
                assert np.array_equal(a0, a1)
                assert c0 == c1
        first = got
        g.close()
