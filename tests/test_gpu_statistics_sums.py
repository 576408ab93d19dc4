"""Statistics of FP32 steps whose nodes all take the second stage: one state at
every node, so that the sums are N times one node's values and show the
rounding of the summation alone.

The second stage knows rho - rho0, j and rho of a node as FP32 numbers and
sums them, and the kinetic energy formed from them, as FP64 sums would: the
mean momentum is an FP32 number and the mean kinetic energy is
|j|^2 / (2 rho) of FP32 numbers, to 2^-40.  (N / threads < 64 additions of a
thread, each off by at most 2^-47 of the thread's sum, and two double-float
operations of 2^-44; the sums over threads are FP64.)  Nodes that go on to
the FP64 series give the FP64 moments of the stored state instead, to 1e-12."""
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


@pytest.mark.parametrize("dtype", ["fp32_shifted", "fp32", "fp16_shifted"])
@pytest.mark.parametrize("lat,shape", [("D2Q9", (1, 1500, 2000)),
                                       ("D3Q27", (80, 90, 101))])
def test_sums_of_second_stage_nodes(elbm, lat, shape, dtype):
    import oracle
    c, w = oracle.lattice(lat)
    d = oracle.dim(lat)
    nz, ny, nx = shape
    n = nx * ny * nz
    g = elbm.Lattice(lat, nx, ny, nz, nu=1e-3, dtype=dtype)
    g.set_diagnostics(diag_every=1)
    seen = 0
    for seed in range(6):
        rng = np.random.default_rng(seed)
        u = 0.1 * rng.uniform(-1, 1, d)
        f = w * 1.03
        for a in range(d):
            s = 3 * u[a] ** 2 / (1 + np.sqrt(1 + 3 * u[a] ** 2))
            ca = c[:, a]
            f = f * np.where(ca == 0, 1 - s, 1 + 3 * ca * u[a] + 2 * s)
        noise = 1e-3 if dtype == "fp16_shifted" else 1e-7
        f = f * (1 + noise * rng.uniform(-1, 1, len(w)))
        g.set_populations(np.broadcast_to(
            f.reshape((-1,) + (1,) * 3), (len(w),) + shape).copy())
        f = g.populations()[:, 0, 0, 0]
        g.step(1, "formula")
        st = g.entropy_stats()
        assert st["n_nodes"] == n
        if st["n_band"] < n:
            continue
        seen += 1
        mass, ke = st["mass"] / n, st["kinetic_energy"] / n
        mom = np.array(st["momentum"][:d]) / n
        j = c[:, :d].T.astype(float) @ f
        rho = f.sum()
        exact = (abs(mass - rho) <= 1e-12 and
                 np.all(np.abs(mom - j) <= 1e-12) and
                 abs(ke - 0.5 * (j @ j) / rho) <= 1e-12 * ke)
        j32 = mom.astype(np.float32)
        near = np.float32(mass)
        cand = [np.nextafter(near, np.float32(0)), near,
                np.nextafter(near, np.float32(9))]
        j64 = j32.astype(float)
        tol = 2.0 ** -40
        fp32 = (np.all(np.abs(mom - j64) <= tol * np.abs(j64)) and
                any(abs(ke - 0.5 * (j64 @ j64) / float(r)) <= tol * ke
                    for r in cand))
        assert exact or fp32, (seed, mass - rho, mom - j, mom - j64, ke)
        # either way within the FP32 rounding of one node's moments
        assert abs(mass - rho) <= 2e-7
        assert np.all(np.abs(mom - j) <= 2e-7)
    assert seen > 0 or dtype == "fp16_shifted"
