"""FP64-arithmetic stream-collide against the oracle, one step from the same
state, over the range of its series path and across its edges: relative
non-equilibrium parts from rounding to 20 % (the path ends at 1/32),
velocities on both sides of its limit 1/4, densities far from one, ragged
sizes around a warp and a block.

Tolerances: FORMULA populations within 1e-12 relative, as for every FP64
path (alpha is off by less than 1e-13 and enters through n_i = f_i x_i);
ROOT and SECANT within 1e-9 of the largest population (a stop-rule edge
within rounding can move alpha by the width of the stop interval)."""
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


@pytest.mark.parametrize("mode", ["formula", "root", "secant"])
@pytest.mark.parametrize("noise,umax,scale", [
    (0.0, 0.0, 1.0), (1e-13, 0.05, 1.0), (1e-6, 0.2, 1e-6), (1e-3, 0.05, 1e6),
    (0.015, 0.1, 1.0), (0.03, 0.26, 1.0), (0.2, 0.05, 1.0)])
@pytest.mark.parametrize("lat,shape", [("D2Q9", (1, 1, 1)),
                                       ("D2Q9", (1, 31, 33)),
                                       ("D3Q27", (3, 5, 7)),
                                       ("D3Q27", (8, 9, 16))])
def test_one_step_matches_oracle(elbm, lat, shape, noise, umax, scale, mode):
    import oracle
    nz, ny, nx = shape
    d = 2 if lat == "D2Q9" else 3
    rng = np.random.default_rng([nx, int(1e6 * umax)])
    rho = scale * (1.0 + 0.02 * rng.uniform(-1, 1, shape))
    u = umax * rng.uniform(-1, 1, (d,) + shape)
    g = elbm.Lattice(lat, nx, ny, nz, nu=1e-3, dtype="fp64")
    g.init_fields(rho, u)
    f = g.populations()
    g.set_populations(f * (1.0 + noise * rng.uniform(-1, 1, f.shape)))
    g.set_diagnostics(diag_every=1, alpha_map_every=1)
    loaded = g.populations()
    o = oracle.Lattice(lat, nx, ny, nz, nu=1e-3)
    o.set_populations(loaded)
    o.step(1, mode, secant_iters=4)
    g.step(1, mode)
    f = g.populations()
    if mode == "formula":
        assert np.all(np.abs(f - o.f) <= 1e-12 * o.f)
    else:
        assert np.abs(f - o.f).max() <= 1e-9 * np.abs(o.f).max()
    s = g.entropy_stats()
    assert s["n_nodes"] == g.n
    assert abs(s["mass"] / loaded.sum() - 1) < 1e-12
    c = oracle.lattice(lat)[0][:, :d].astype(float)
    j = np.tensordot(c, loaded, (0, 0))
    ke = 0.5 * ((j ** 2).sum(0) / loaded.sum(0)).sum()
    assert abs(s["kinetic_energy"] - ke) <= 1e-12 * ke + 1e-28 * scale * g.n
    a = g.alpha_map()
    assert s["alpha_min"] <= a.min() * (1 + 1e-6)
    assert s["alpha_max"] >= a.max() * (1 - 1e-6)

