"""Waits that run out inside the kernels (lbm_selftest_withhold keeps units from
being staged, or a grid barrier from completing): the kernel ends, takes nothing
from a stage that was not filled and writes nowhere else, the call reports
LBM_ERR_TIMEOUT, and the context works again from a new state."""
import numpy as np
import pytest

from paper_1710_09472_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CLOCKS = 1 << 22  # about 2 ms
GUARD, MARK = 4096, -12345.0


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09472_gb300.build import build

    build()


# whole rows (ragged and exact) and ragged segments, with a unit for every SM at least
BOXES = [("D3V19", (16, 10, 40), "f32"), ("D3V19", (16, 10, 50), "f16"), ("D3V19", (10, 16, 256), "f32"),
         ("D2V9", (80, 1025), "f32"), ("D3V27", (10, 16, 250), "bf16")]


def _box(vel, shape, storage):
    from paper_1710_09472_gb300.lbm import LBM

    solid, _ = wl.boolean_obstacles(shape, 2.5, 0.8, seed=31)
    sim = LBM(vel, tuple(reversed(shape)), 0.8, E=(1e-4, 0, 0), storage=storage)
    sim.set_geometry(solid.reshape(-1))
    sim.init_equilibrium()
    return sim


def _guarded(n, dtype=torch.float32):
    whole = torch.full((n + 2 * GUARD,), MARK, dtype=dtype, device="cuda")
    return whole, whole[GUARD:GUARD + n]


def _intact(whole):
    return bool((whole[:GUARD] == MARK).all() and (whole[-GUARD:] == MARK).all())


def _times_out(call):
    from paper_1710_09472_gb300._lib import LBMError

    with pytest.raises(LBMError, match="LBM_ERR_TIMEOUT"):
        call()


def _good_as_new(sim, *box):
    sim.selftest_withhold(-1)
    fresh = _box(*box)
    sim.init_equilibrium()
    for s in (sim, fresh):
        for _ in range(3):
            s.step(1)
    np.testing.assert_array_equal(sim.populations(), fresh.populations())
    assert sim.moments()[0] == fresh.moments()[0]
    fresh.close()


@pytest.mark.parametrize("vel,shape,storage", BOXES)
@pytest.mark.parametrize("part", [0.0, 0.5])
def test_fields_of_unstaged_units(vel, shape, storage, part):
    box = (vel, shape, storage)
    sim = _box(*box)
    sim.step(1)
    want, want_j = torch.empty(sim.N, device="cuda"), torch.empty(sim.D * sim.N, device="cuda")
    sim.moments(want, want_j)
    rows = sim.N // shape[-1]
    units = int(part * rows)
    sim.selftest_withhold(units, CLOCKS)
    (whole, rho), (whole_j, j) = _guarded(sim.N), _guarded(sim.D * sim.N)
    _times_out(lambda: sim.moments(rho, j))
    assert _intact(whole) and _intact(whole_j)
    # rows of whole units: the staged ones as they are, the others zero or untouched
    if shape[-1] < 1000:
        done = units * shape[-1]
        assert torch.equal(rho[:done], want[:done])
        assert bool(((rho[done:] == MARK) | (rho[done:] == 0)).all())
        jd = j.view(sim.D, -1)
        assert torch.equal(jd[:, :done], want_j.view(sim.D, -1)[:, :done])
        assert bool(((jd[:, done:] == MARK) | (jd[:, done:] == 0)).all())
    _good_as_new(sim, *box)
    sim.close()


@pytest.mark.parametrize("vel,shape,storage", BOXES)
def test_steps_and_reverse_steps(vel, shape, storage):
    box = (vel, shape, storage)
    sim = _box(*box)
    sim.selftest_withhold(0, CLOCKS)
    sim.step(1)
    _times_out(lambda: sim.moments())  # the step's wait, or the fields' own
    whole, dE = _guarded(sim.D * sim.N, torch.float64)
    whole_l, lam0 = _guarded(sim.Q * sim.N)
    _times_out(lambda: sim.adjoint(1, 3, torch.ones(sim.N, device="cuda"), None, dL_dE=dE, dL_df0=lam0))
    assert _intact(whole) and _intact(whole_l)
    _good_as_new(sim, *box)
    sim.close()


def test_grid_barrier():
    box = ("D2V9", (100, 331), "f32")
    sim = _box(*box)
    before = sim.launch_count()
    sim.selftest_withhold(0, CLOCKS)
    sim.step(5)
    assert sim.launch_count() == before + 1  # many steps in one launch
    _times_out(lambda: sim.moments())
    _good_as_new(sim, *box)
    sim.close()


def test_arguments():
    from paper_1710_09472_gb300._lib import LBMError

    sim = _box("D2V9", (8, 40), "f32")
    for clocks in (0, (1 << 31) + 1):
        with pytest.raises(LBMError):
            sim.selftest_withhold(0, clocks)
    sim.step(2)
    sim.moments()
    sim.close()
