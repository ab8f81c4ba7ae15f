"""Applies captured in a CUDA graph."""
import numpy as np
import pytest

from paper_1709_09347_gb300 import synth
from tests._gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("atoms", [0, 3])
@pytest.mark.parametrize("dtype", ["complex128", "complex64"])
def test_captured_apply_follows_the_potential(atoms, dtype):
    """V_loc is replaced in place, so a replay applies the present one: potentials whose largest
    value moves the fixed-point unit of the weights up and down, and one that no unit holds.  A
    handle made with that V_loc gives the reference; where the unit has moved, the replay takes the
    FP64 formula, which may differ by the rounding of a few dozen terms."""
    torch = need_gpu()
    from paper_1709_09347_gb300 import cbs
    wl = synth.tiny_workload(nx=9, ny=10, nz=16, h=0.4, fd_order=8, n_atoms=max(atoms, 1), r_c=0.75, sigma=0.3,
                             projectors=atoms > 0, L=6)
    dt = getattr(torch, dtype)
    H = cbs.Hamiltonian(wl.grid, wl.vloc, wl.projectors)
    z, E = np.array([2 * np.exp(0.3j), 0.5 * np.exp(-1.2j)]), np.array([0.3, -0.45])
    g = torch.Generator(device="cuda").manual_seed(2)
    X = torch.randn((2, wl.grid.n, 6), dtype=dt, device="cuda", generator=g)
    Y = torch.empty_like(X)
    plan = cbs.ApplyPlan(H, z, E, 6, dt)
    plan(X, Y)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan(X, Y)
    for factor in (1.0, 40.0, 3000.0, 0.01, 1e52 if dtype == "complex128" else 1.0, 1.0):
        v = wl.vloc * factor
        H.set_vloc(v)
        Y.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        ref = cbs.apply(cbs.Hamiltonian(wl.grid, v, wl.projectors), z, E, X)
        if factor == 1.0 or dtype == "complex64":
            assert torch.equal(Y, ref), factor
        else:
            assert float((Y - ref).abs().max()) <= 1e-14 * float(ref.abs().max()), factor
