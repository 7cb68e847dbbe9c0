"""Batches at the edges of what a process and a device hold: several host threads, device memory."""
import ctypes
import threading

import numpy as np
import pytest

from paper_2403_11167_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    import __graft_entry__

    __graft_entry__.build()
    from paper_2403_11167_gb300 import lbm as L

    return L


def _spec(lbm, nx, ny, nsteps, seed):
    p = lbm.lbm_params_default(lbm.LBM_PSEUDOPOTENTIAL, precision=lbm.LBM_F32, a=0.25, Tr=0.85, tau_nu=0.8)
    _, th = lbm.lbm_resolve_params(p)
    return (dict(nx=nx, ny=ny, geometry=0, nsteps=nsteps, params=p),
            inputs.spinodal_noise(nx, ny, 0.5 * (th.rho_l + th.rho_v), 0.01, seed=seed))


def test_threads_with_resident_batches_of_different_sizes(lbm):
    """Two host threads run batches whose resident lattices need the same kernel with different amounts of
    shared memory, 3000 times each: no launch of either is refused, and the states are those of one thread."""
    sizes = [(64, 64), (48, 50)]
    batches = [lbm.Batch(*zip(_spec(lbm, nx, ny, 2, seed=nx))) for nx, ny in sizes]
    for b in batches:
        b.run()
    want = [b.populations(0) for b in batches]
    errors = []

    def work(b):
        try:
            for _ in range(3000):
                b.run()
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(b,)) for b in batches]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for b, w in zip(batches, want):
        assert np.array_equal(b.populations(0), w)
        b.close()


def test_batch_that_fills_the_device(lbm):
    """With room for the buffers and the scratch (88 bytes per cell) but not for the initial densities too
    (96), a batch still runs, and runs again, to the bits of one with room."""
    import torch

    nx, ny = 8192, 4096
    specs, rhos = zip(_spec(lbm, nx, ny, 3, seed=1), _spec(lbm, 40, 40, 3, seed=2))

    def outputs():
        b = lbm.Batch(specs, rhos)
        out = []
        for _ in range(2):
            b.run()
            out.append((b.observables(), b.populations(0), b.populations(1)))
        b.close()
        return out

    want = outputs()
    torch.cuda.synchronize()
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - 92 * nx * ny, dtype=torch.uint8, device="cuda")
    got = outputs()
    del hold
    torch.cuda.empty_cache()
    for g, w in zip(got, want):
        assert repr(g[0]) == repr(w[0])
        assert np.array_equal(g[1], w[1]) and np.array_equal(g[2], w[2])


def test_run_after_a_failed_run(lbm):
    """A run that fails between the resident launch and the tiled one (the caller has left the batch's stream in
    capture, so its graph cannot be captured) does not spoil the next: the resident kernel of the failed run,
    20,000 steps long, stores its last state before the next run's initial state is written."""
    specs, rhos = zip(_spec(lbm, 64, 64, 20000, seed=1), _spec(lbm, 100, 60, 10, seed=2))
    want = []
    for s, r in zip(specs, rhos):
        ctx = lbm.Context(s["params"], s["nx"], s["ny"])
        ctx.set_density(r)
        ctx.step(s["nsteps"])
        want.append(ctx.populations())
        ctx.close()
    b = lbm.Batch(specs, rhos)
    cudart = ctypes.CDLL("libcudart.so.13")
    stream = ctypes.c_void_p(lbm._lib().lbm_batch_stream(b.h))
    assert cudart.cudaStreamBeginCapture(stream, 2) == 0  # relaxed
    with pytest.raises(lbm.LBMError):
        b.run()
    graph = ctypes.c_void_p()
    cudart.cudaStreamEndCapture(stream, ctypes.byref(graph))
    if graph:
        cudart.cudaGraphDestroy(graph)
    cudart.cudaGetLastError()
    b.run()
    for i, w in enumerate(want):
        assert np.array_equal(b.populations(i), w), i
    b.close()
