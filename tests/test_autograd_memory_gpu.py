"""WindowCurrent.backward() where the device has no room beside the start state
that forward() kept there: for its own tensors, for lbm_adjoint's buffers or for
the result.  The start state then goes through the host, with the same gradients,
also for a second backward() over the same graph."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09472_gb300.build import build

    build()


def _gradients():
    from paper_1710_09472_gb300.autograd import WindowCurrent
    from paper_1710_09472_gb300.lbm import LBM

    sim = LBM("D2V9", (41, 12), 0.8, storage="f16")
    sim.init_equilibrium()
    E = torch.full((2, 12, 41), 1e-3, device="cuda").requires_grad_()
    B = torch.tensor([0.0, 0.0, 1e-3], device="cuda", requires_grad=True)
    tau = torch.tensor(0.8, device="cuda", requires_grad=True)
    loss = WindowCurrent.apply(E, B, tau, sim, 5, 10, 3)[1]
    got = []
    for _ in range(2):
        got += list(torch.autograd.grad(loss, (E, B, tau), retain_graph=True))
    assert sim.info()["steps"] == 10  # both leave the run at its end
    sim.close()
    return got


def _once(real, error, calls):
    def call(*a, **k):
        calls.append(1)
        if len(calls) == 1:
            raise error
        return real(*a, **k)
    return call


@pytest.mark.parametrize("where", ["tensors", "adjoint", "result"])
def test_backward_without_room(where, monkeypatch):
    from paper_1710_09472_gb300 import _lib
    from paper_1710_09472_gb300.lbm import LBM

    want = _gradients()
    calls, saves = [], []
    full = torch.cuda.OutOfMemoryError("no room")
    place, name, error = {"tensors": (torch.Tensor, "repeat_interleave", full),
                          "adjoint": (LBM, "adjoint", _lib.LBMError(_lib.LBM_ERR_OOM, "no room")),
                          "result": (torch.Tensor, "to", full)}[where]  # after lbm_adjoint has run
    monkeypatch.setattr(place, name, _once(getattr(place, name), error, calls))
    real = LBM.save_state
    monkeypatch.setattr(LBM, "save_state", lambda self: (saves.append(1), real(self))[1])
    got = _gradients()
    assert len(saves) == 1 and len(calls) == 3
    for a, b in zip(want, got):
        assert torch.equal(a, b)


def test_other_errors_are_raised(monkeypatch):
    from paper_1710_09472_gb300 import _lib
    from paper_1710_09472_gb300.lbm import LBM

    monkeypatch.setattr(LBM, "adjoint", _once(LBM.adjoint, _lib.LBMError(5, "non-finite gradient"), []))
    with pytest.raises(_lib.LBMError):
        _gradients()
