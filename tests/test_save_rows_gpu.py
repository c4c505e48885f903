"""Saved states and per-cell fields of rows that are padded or cut into segments:
packed on the device, one copy each way, the same bytes as row by row."""
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


# padded rows (nx no multiple of 8), segments (ragged last ones), more chunks than blocks; a whole row for comparison
BOXES = [("D2V9", (7, 33), "f16"), ("D2V9", (40, 1025), "f32"), ("D3V19", (3, 5, 490), "bf16"),
         ("D3V27", (4, 3, 305), "f32"), ("D1V3", (70001,), "f16"), ("D2V9", (5, 40), "f32")]


@pytest.mark.parametrize("vel,shape,storage", BOXES)
def test_save_and_load(vel, shape, storage):
    from paper_1710_09472_gb300.lbm import LBM

    N, D = int(np.prod(shape)), len(shape)
    solid = (wl.uniform01(3, N) < 0.2).astype(np.uint8)
    u = (0.01 * wl.normal(5, D * N)).astype(np.float32)
    sims = [LBM(vel, tuple(reversed(shape)), 0.8, E=(1e-4, 0, 0), storage=storage) for _ in range(2)]
    for s in sims:
        s.set_geometry(solid)
        s.init_equilibrium(None, u)
    a, b = sims
    for _ in range(3):
        a.step(1)
    before, blob = a.populations(deviation=True), a.save_state()
    np.testing.assert_array_equal(a.populations(deviation=True), before)  # the state is as it was
    assert a.save_state() == blob
    # slot by slot: the populations in the blob are those that the cells pull, rows of nx values (lbm.h)
    eb = 4 if storage == "f32" else 2
    assert len(blob) >= 64 + a.Q * N * eb
    b.load_state(blob)
    np.testing.assert_array_equal(b.populations(deviation=True), before)
    assert b.save_state() == blob
    for s in sims:
        s.step(1)
        s.step(4)
    np.testing.assert_array_equal(a.populations(), b.populations())
    for s in sims:
        s.close()


@pytest.mark.parametrize("vel,shape,storage", BOXES)
def test_field_from_the_host(vel, shape, storage):
    """A host field in the middle of a run acts as the same field on the device."""
    from paper_1710_09472_gb300.lbm import LBM

    N, D = int(np.prod(shape)), len(shape)
    E = (1e-4 * wl.normal(7, D * N)).astype(np.float32)
    out = []
    for field in (E, torch.from_numpy(E).cuda()):
        sim = LBM(vel, tuple(reversed(shape)), 0.8, storage=storage)
        sim.set_E_field(field)  # before there is a state
        sim.init_equilibrium()
        for k in range(3):
            sim.step(1)
            sim.set_E_field(field if k % 2 else E[::-1].copy())
        sim.step(1)
        out.append(sim.populations(deviation=True))
        sim.close()
    np.testing.assert_array_equal(out[0], out[1])
    assert np.abs(out[0]).max() > 0
