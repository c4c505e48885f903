"""Contexts of different widths stepped from several threads at once, each on a
stream of its own: they run the same kernels with different amounts of shared
memory, and each gets the bits that it gets alone."""
import threading

import numpy as np
import pytest

from paper_1710_09472_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09472_gb300.build import build

    build()


def _steps(nx, calls, out):
    from paper_1710_09472_gb300.lbm import LBM

    try:
        stream = torch.cuda.Stream()
        shape = (16, 16, nx)
        solid, _ = wl.boolean_obstacles(shape, 2.5, 0.8, seed=17)
        sim = LBM("D3V19", (nx, 16, 16), 0.8, E=(1e-4, 0, 0), stream=stream)
        sim.set_geometry(solid.reshape(-1))
        sim.init_equilibrium()
        rho = torch.empty(sim.N, device="cuda")
        for _ in range(calls):
            sim.step(1)
            sim.moments(rho, None, totals=False)
        w = torch.ones(sim.N, device="cuda")
        torch.cuda.synchronize()
        loss = sim.adjoint(0, 4, w, None)["loss"]
        out[nx] = (sim.populations(), loss)
        sim.close()
    except Exception as e:  # the thread's failure is the test's
        out[nx] = e


def test_contexts_of_different_widths():
    # run-time strides: 64 to 180 KB of shared memory in one kernel
    widths, calls = (96, 160, 224, 320), 1500
    alone, together = {}, {}
    for nx in widths:
        _steps(nx, calls, alone)
    threads = [threading.Thread(target=_steps, args=(nx, calls, together)) for nx in widths]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for nx in widths:
        assert not isinstance(together[nx], Exception), together[nx]
        np.testing.assert_array_equal(together[nx][0], alone[nx][0])
        assert together[nx][1] == alone[nx][1]
