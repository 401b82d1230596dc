"""The device memory of contexts that come and go: given back but for a bounded rest, sound for contexts of several
threads at once, each on its own stream."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

from paper_1701_06658_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1701_06658_gb300 import lsgg
    lsgg.lib()
    return lsgg


def _run(L, seed):
    n = 24 + 8 * (seed % 4)
    with L.Microstructure(n, n + 2, n + 4, 12, seeds=I.voronoi_seeds(seed, 12, (n, n + 2, n + 4))) as ms:
        ms.step(4, 1.0)
        ms.sync()
        return ms.boxes(), L.get_phi(ms.ctx), ms.grain_volumes()


def test_threads_reuse_each_other_s_memory(L):
    want = {s: _run(L, s) for s in range(8)}
    got, errors = {}, []

    def work(first):
        try:
            for k in range(3):
                for s in range(8):
                    got[first, k, s] = _run(L, (s + first) % 8)
        except Exception as e:                       # seen by the asserting thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for (first, _, s), r in got.items():
        for a, b in zip(r, want[(s + first) % 8]):
            assert np.array_equal(a, b)


def test_memory_is_given_back(L):
    import torch
    _run(L, 1)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    n, G = 128, 600
    mss = [L.Microstructure(n, n, n, G, seeds=I.voronoi_seeds(k, G, (n, n, n))) for k in range(6)]
    held = sum(ms.stats().device_bytes for ms in mss)
    for ms in mss:
        ms.close()
    torch.cuda.synchronize()
    assert held > 2 << 30                            # more than the pool keeps without contexts
    assert torch.cuda.mem_get_info()[0] >= free - (1 << 30) - (64 << 20)


def test_a_thread_new_to_cuda_destroys_contexts(L):
    """Contexts made by this thread and destroyed by one that has called nothing of CUDA: their memory is back."""
    import torch
    _run(L, 1)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    n, G = 128, 600
    mss = [L.Microstructure(n, n, n, G, seeds=I.voronoi_seeds(k, G, (n, n, n))) for k in range(6)]
    assert sum(ms.stats().device_bytes for ms in mss) > 2 << 30

    def close():
        for ms in mss:
            ms.close()

    t = threading.Thread(target=close)
    t.start()
    t.join()
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= free - (1 << 30) - (64 << 20)


def test_growth_from_the_pool_to_plain_allocations(L):
    """An arena grows past the size up to which buffers come from the pool, with room for the new ones only if the
    old ones, just freed into the pool, are given back: the room left holds three of the four new buffers."""
    import torch
    dims, G = (96, 96, 96), 60
    e = 4e-2 * I.u01(5, 7, np.arange(G))
    old_cap, new_cap = 110 << 20, 150 << 20          # elements of four bytes: 440 and 600 MiB a buffer
    with L.Microstructure(*dims, G, seeds=I.voronoi_seeds(5, G, dims), energy=e, physics=L.PHYSICS_MAGNETIC) as a, \
            L.Microstructure(*dims, G, seeds=I.voronoi_seeds(5, G, dims), energy=e, physics=L.PHYSICS_MAGNETIC) as b:
        a.step(4, 1.0)
        a.sync()
        L.debug_set_capacity(b.ctx, old_cap)
        b.step(2, 1.0)
        b.sync()
        torch.cuda.synchronize()
        room = 3 * 4 * new_cap + (256 << 20)
        ballast = torch.empty(max(0, torch.cuda.mem_get_info()[0] - room), dtype=torch.uint8, device="cuda")
        try:
            L.debug_set_capacity(b.ctx, new_cap)     # raises when it runs out
        finally:
            del ballast
            torch.cuda.empty_cache()
        b.step(2, 1.0)
        b.sync()
        assert b.stats().arena_capacity == new_cap
        assert np.array_equal(a.boxes(), b.boxes())
        assert np.array_equal(L.get_phi(a.ctx), L.get_phi(b.ctx))


RESET = """
import ctypes, numpy as np
from paper_1701_06658_gb300 import inputs as I, lsgg as L
L.lib()
rt = ctypes.CDLL("libcudart.so.13")

def run(keep=False):
    ms = L.Microstructure(40, 36, 44, 12, seeds=I.voronoi_seeds(3, 12, (40, 36, 44)))
    ms.step(4, 1.0)
    ms.sync()
    out = ms.boxes(), L.get_phi(ms.ctx), ms.grain_volumes()
    if keep:
        return ms, out
    ms.close()
    return out

want = run()
old, _ = run(keep=True)
for k in range(2):
    assert rt.cudaDeviceReset() == 0
    ms, got = run(keep=True)
    assert all(np.array_equal(a, b) for a, b in zip(want, got))
    old.close()                                      # of the CUDA context before: nothing of the new one goes with it
    assert all(np.array_equal(a, b) for a, b in zip(want, run()))
    assert np.array_equal(want[1], L.get_phi(ms.ctx))
    old = ms
print("same after the reset")
"""


def test_contexts_after_a_device_reset():
    """The process ends its own CUDA context (cudaDeviceReset) with a microstructure in it and makes new ones."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", RESET], cwd=root, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "same after the reset" in r.stdout, r.stderr[-2000:]
