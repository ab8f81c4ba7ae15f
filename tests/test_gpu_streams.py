"""Solves beside work of other owners of the GPU."""
import threading

import numpy as np
import pytest

from paper_1709_09347_gb300 import synth
from tests._gpu_common import need_gpu

pytestmark = pytest.mark.gpu


class _BusyDefaultStream:
    """Keeps the legacy default stream occupied from another thread: kernels of a few
    milliseconds, at most four in flight, while the block runs."""

    def __enter__(self):
        import torch
        self.stop = False

        def work():
            flight = []
            while not self.stop:
                torch.cuda._sleep(5_000_000)
                ev = torch.cuda.Event()
                ev.record()
                flight.append(ev)
                if len(flight) == 4:
                    flight.pop(0).synchronize()

        self.thread = threading.Thread(target=work)
        self.thread.start()
        return self

    def __exit__(self, *exc):
        self.stop = True
        self.thread.join()


def _dirty_memory(torch):
    """Leaves memory that a later allocation may be given full of ones."""
    t = torch.full((64 << 20,), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    del t
    torch.cuda.empty_cache()


@pytest.mark.parametrize("precision,multi_shift", [("fp64", 0), ("fp32_refine", 0), ("fp64", 1), ("fp32_refine", 1)])
def test_solves_beside_a_busy_default_stream(precision, multi_shift):
    """The solver runs on a stream of its own, which nothing orders against the default stream: the
    results are those of a quiet GPU, bit for bit (every reduction has a fixed order)."""
    torch = need_gpu()
    from paper_1709_09347_gb300 import cbs
    wl = synth.tiny_workload(nx=6, ny=5, nz=4, h=0.45, fd_order=4, n_atoms=2, r_c=0.8, sigma=0.3, L=8, M=4, n_int=16,
                             energies=(0.2, -0.3))
    H = cbs.Hamiltonian(wl.grid, wl.vloc, wl.projectors)
    o = cbs.options(tol=1e-11, precision=precision, multi_shift=multi_shift)

    def go():
        res = cbs.solve(H, wl.energies, wl.lambda_min, wl.n_int, wl.L, wl.M, wl.V, o)
        J, g, gE = cbs.objective(H, 0.2, wl.lambda_min, wl.n_int, wl.L, wl.M, wl.V, o, grad=True)
        return [e[k] for e in res.energies for k in ("mu", "iters", "lam")] + [np.asarray(J), np.asarray(g), np.asarray(gE)]

    quiet = go()
    for _ in range(3):
        _dirty_memory(torch)
        with _BusyDefaultStream():
            beside = go()
        assert all(np.array_equal(a, b) for a, b in zip(quiet, beside))
