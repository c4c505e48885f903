"""The thermal step takes two cells per thread away from the row's ends and
one at them.  A cell has the same bits either way: a run of the fields shifted
by some cells is the shifted run (periodic row, no random rounding)."""
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


# one cell per thread; then (2 x 256 cells for each of 152 SMs and more) pairs, even and odd
@pytest.mark.parametrize("nx", [5, 1031, 77824, 77825, 100002])
@pytest.mark.parametrize("lattice,order", [("D1V7", 4), ("D1V5a", 2)])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_shifted_run(nx, lattice, order, storage):
    from paper_1710_09472_gb300.lbm import Thermal

    rho = (1.0 + 0.01 * wl.normal(5, nx)).astype(np.float32)
    u = (0.01 * wl.normal(6, nx)).astype(np.float32)
    th = (1.0 + 0.01 * wl.normal(7, nx)).astype(np.float32)

    def run(shift):
        t = Thermal(lattice, nx, 0.8, E=1e-4, order=order, storage=storage, stat="mb", theta=1.0, mu=0.0)
        if storage != "f32":
            t.set_rounding(False)
        t.init(*[torch.from_numpy(np.roll(a, shift)).cuda() for a in (rho, u, th)])
        t.step(7)
        f = t.populations(torch.empty(t.Q * nx, device="cuda"), deviation=True).cpu().numpy().reshape(t.Q, nx)
        tot = t.moments()
        t.close()
        return f, tot

    a, ta = run(0)
    assert np.isfinite(a).all()
    for shift in (1, nx // 2):
        b, tb = run(shift)
        np.testing.assert_array_equal(np.roll(a, shift, axis=1), b)
        np.testing.assert_allclose(tb, ta, rtol=1e-12, atol=1e-10)  # FP64 sums in another order
