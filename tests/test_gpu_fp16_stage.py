"""D2Q9 binary16 lattices run the second stage of undecided nodes inside the
stream-collide kernel up to 2^19 nodes and from a record buffer beyond: a flow
and its periodic repetition, on either side of the limit, evolve bit for bit
alike, right after initialisation and later.  (Flows without symmetry planes:
at a tie the branch is rounding, and the logarithms' rounding depends on the
length of their queue.)"""
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


@pytest.mark.parametrize("seed", [2, 3])
@pytest.mark.parametrize("n", [(723, 725), (724, 725), (601, 603)])
def test_repeated_flow(elbm, n, seed):
    ny, nx = n   # 2^19 = 524,288: 524,175 and 524,900; and 362,403
    rho, u = W.random_phase_2d(nx, seed=seed, umax=0.05, ny=ny)
    got = []
    for k in (1, 2):
        g = elbm.Lattice("D2Q9", nx, k * ny, 1, nu=1e-3, dtype="fp16_shifted")
        g.set_diagnostics(diag_every=1, alpha_map_every=1)
        g.init_fields(np.tile(rho, (1, k, 1)), np.tile(u, (1, 1, k, 1)))
        runs = []
        for steps in (1, 1, 6):
            g.step(steps, "formula")
            s = g.entropy_stats()
            runs.append((g.populations(), g.alpha_map(), np.array(
                [s[c] for c in ("n_nodes", "n_accept_two", "n_formula",
                                "n_band", "n_degenerate")])))
        got.append((g.rho0, runs))
        g.close()
    assert got[0][0] == got[1][0]
    band = 0
    for (f1, a1, c1), (f2, a2, c2) in zip(got[0][1], got[1][1]):
        assert np.array_equal(np.tile(f1, (1, 1, 2, 1)), f2)
        assert np.array_equal(np.tile(a1, (1, 2, 1)), a2)
        assert np.array_equal(2 * c1, c2)
        band += c1[3]
    assert band > 0
