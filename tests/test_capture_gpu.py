"""lbm_step under stream capture: an even number of captured steps ends in the
buffer it started from, so a replayed graph steps on from the state that the
replay before it left, whichever kernel takes the steps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09472_gb300.build import build

    build()


# a cluster's box (one launch), a cooperative grid's, and one that is stepped launch by launch
@pytest.mark.parametrize("vel,dims", [("D2V9", (32, 64)), ("D2V9", (331, 100)), ("D3V19", (64, 48, 40))])
@pytest.mark.parametrize("calls", [(2,), (10,), (3, 3)])
def test_replayed_steps(vel, dims, calls):
    from paper_1710_09472_gb300.lbm import LBM

    def box(stream=None):
        sim = LBM(vel, dims, 0.8, E=(1e-4, 0.0, 0.0), stream=stream)
        solid = np.zeros(sim.N, dtype=np.uint8)
        solid[:: 7] = 1
        sim.set_geometry(solid)
        sim.init_equilibrium()
        return sim

    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        sim = box(stream)
        for n in calls:  # every kernel has been launched once
            sim.step(n)
        sim.init_equilibrium()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        for n in calls:
            sim.step(n)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    plain = box()
    plain.step(3 * sum(calls))
    np.testing.assert_array_equal(sim.populations(), plain.populations())
    sim.close()
    plain.close()
