"""One-call applies: scratch kept with the handle, several threads on one handle."""
import threading
import time

import numpy as np
import pytest

from paper_1709_09347_gb300 import synth
from tests._gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def _cell(atoms=2):
    return synth.tiny_workload(nx=9, ny=10, nz=6, h=0.4, fd_order=8, n_atoms=atoms, r_c=0.75, sigma=0.3, L=1)


def test_threads_share_a_handle():
    """Four threads, each on a stream of its own, with batches that grow and shrink: every result is
    that of the same call alone, bit for bit."""
    torch = need_gpu()
    from paper_1709_09347_gb300 import cbs
    wl = _cell()
    H = cbs.Hamiltonian(wl.grid, wl.vloc, wl.projectors)
    gen = torch.Generator(device="cuda").manual_seed(4)
    jobs = []
    for n, L, dt in ((1, 3, torch.complex128), (7, 16, torch.complex128), (2, 40, torch.complex64), (16, 64, torch.complex128)):
        X = torch.randn((n, wl.grid.n, L), dtype=dt, device="cuda", generator=gen)
        z, E = 1.8 * np.exp(1j * np.arange(n)), np.linspace(-0.5, 0.5, n)
        jobs.append((z, E, X, cbs.apply(H, z, E, X)))
    torch.cuda.synchronize()
    wrong = []

    def work(k):
        with torch.cuda.stream(torch.cuda.Stream()):
            for i in range(40):
                z, E, X, ref = jobs[(k + i) % len(jobs)]
                if not torch.equal(cbs.apply(H, z, E, X), ref):
                    wrong.append((k, i))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


def test_scratch_goes_with_the_handle():
    """16 MiB at most stay with a handle, and they are given back with it."""
    torch = need_gpu()
    from paper_1709_09347_gb300 import cbs
    wl = _cell()
    X = torch.randn((64, wl.grid.n, 64), dtype=torch.complex128, device="cuda")
    z, E = np.full(64, 1.5 + 0.5j), np.zeros(64)

    def once():
        H = cbs.Hamiltonian(wl.grid, wl.vloc, wl.projectors)
        cbs.apply(H, z[:4], E[:4], X[:4].contiguous())
        cbs.apply(H, z, E, X)
        torch.cuda.synchronize()
        held = torch.cuda.mem_get_info()[0]
        H.close()
        return held, torch.cuda.mem_get_info()[0]

    once()
    held, free = once()
    assert once()[1] == free
    assert 0 <= free - held <= 24 << 20


def test_time_does_not_follow_the_allocator():
    """The same apply beside more and more other small allocations.  With scratch from the allocator
    the calls that opened a page of device memory took three times the others'; the quietest of
    several medians leaves the host's own noise out."""
    torch = need_gpu()
    from paper_1709_09347_gb300 import cbs
    g = synth.Grid(8, 8, 4, 0.4, 0.4, 0.4, 4)
    X = torch.randn((300, g.n, 64), dtype=torch.complex64, device="cuda")
    z, E = np.full(300, 1.5 + 0.5j), np.zeros(300)
    keep, times = [], []
    for _ in range(40):
        H = cbs.Hamiltonian(g, np.zeros(g.n))
        keep.append((H, cbs.Hamiltonian(synth.Grid(16, 16, 16, 0.4, 0.4, 0.4, 4), np.zeros(4096))))
        best = np.inf
        for k in range(8):
            if k >= 3 and best < 1.5 * min(times, default=best):
                break       # what the allocations cause stays however often it is timed
            t = []
            for _ in range(9):
                torch.cuda.synchronize()
                a = time.perf_counter()
                cbs.apply(H, z, E, X)
                torch.cuda.synchronize()
                t.append(time.perf_counter() - a)
            best = min(best, float(np.median(t)))
        times.append(best)
    assert max(times) < 1.8 * min(times), (min(times), max(times))
