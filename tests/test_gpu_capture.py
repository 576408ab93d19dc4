"""elbm_step captured into a CUDA graph by its caller: the kernels of a call
are chained by programmatic dependent launch, which a capture turns into
programmatic edges, and replays advance the lattice as plain calls do, bit for
bit."""
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


@pytest.mark.parametrize("diag", [0, 1])
@pytest.mark.parametrize("lat,dtype,mode", [
    ("D2Q9", "fp64", "formula"), ("D3Q27", "fp64", "root"),
    ("D2Q9", "fp32_shifted", "formula"), ("D3Q27", "fp32_shifted", "formula"),
    ("D3Q27", "fp16_shifted", "formula"), ("D2Q9", "fp16_shifted", "secant")])
def test_captured_steps(elbm, lat, dtype, mode, diag):
    import torch
    if lat == "D2Q9":
        shape = (1, 45, 61)
        rho, u = W.random_phase_2d(61, seed=3, umax=0.1, ny=45)
    else:
        shape = (13, 17, 23)
        rho, u = W.random_phase_3d(23, seed=3, umax=0.1, ny=17, nz=13)
    nz, ny, nx = shape
    s = torch.cuda.Stream()
    got = []
    for captured in (False, True):
        g = elbm.Lattice(lat, nx, ny, nz, nu=1e-3, dtype=dtype,
                         stream=s.cuda_stream)
        g.set_diagnostics(diag_every=diag)
        g.init_fields(rho, u)
        g.step(2, mode)
        g.sync()
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=s):
                g.step(4, mode)   # an even number: back in the same buffer
            for _ in range(3):
                graph.replay()
            torch.cuda.synchronize()
        else:
            g.step(12, mode)
        got.append(g.populations())
        g.close()
    assert np.array_equal(got[0], got[1])
