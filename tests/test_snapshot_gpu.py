"""States kept in device memory (LBM.snapshot / restore, used by the autograd
function): the same bits as through save_state, on the context's own stream."""
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


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("side", [False, True])
def test_snapshot_round_trip(storage, side):
    from paper_1710_09472_gb300._lib import LBMError
    from paper_1710_09472_gb300.lbm import LBM

    shape = (9, 53)
    solid, _ = wl.boolean_obstacles(shape, 2.0, 0.8, seed=5)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream() if side else None
    sim = LBM("D2V9", (53, 9), 0.8, E=(1e-4, 0, 0), storage=storage, stream=stream)
    with pytest.raises(LBMError):
        sim.snapshot()  # no state yet
    sim.set_geometry(solid.reshape(-1))
    sim.init_equilibrium()
    sim.step(7)
    blob, snap = sim.save_state(), sim.snapshot()
    sim.step(6)
    after = sim.populations()
    sim.restore(snap)
    assert sim.info()["steps"] == 7 and sim.save_state() == blob
    sim.step(6)  # the rounding stream goes on from step 7
    np.testing.assert_array_equal(sim.populations(), after)
    with pytest.raises(LBMError):
        sim.restore((snap[0][:-16], 7))
    sim.close()


def test_gradient_with_the_state_on_the_host(monkeypatch):
    """Without room on the device the start state goes through the host, with
    the same gradients."""
    from paper_1710_09472_gb300.autograd import WindowCurrent
    from paper_1710_09472_gb300.lbm import LBM

    def gradients():
        sim = LBM("D2V9", (40, 12), 0.8, storage="f32")
        sim.init_equilibrium()
        E = torch.full((2, 12, 40), 1e-3, device="cuda", requires_grad=True)
        B = torch.tensor([0.0, 0.0, 1e-3], device="cuda", requires_grad=True)
        tau = torch.tensor(0.8, device="cuda", requires_grad=True)
        WindowCurrent.apply(E, B, tau, sim, 5, 10, 3)[1].backward()
        sim.close()
        return E.grad, B.grad, tau.grad

    device = gradients()

    def full(self):
        raise torch.cuda.OutOfMemoryError()

    monkeypatch.setattr(LBM, "snapshot", full)
    for a, b in zip(device, gradients()):
        assert torch.equal(a, b)
