"""The row-staged kernels on padded rows and on segments of long rows: row
lengths at the edges of both rules (32 cells; three copies of a row within 96
KB), ragged ones among them, against the FP64 oracle; and the saved state,
which holds the rows without their padding."""
import struct

import numpy as np
import pytest

import oracle
from paper_1710_09472_gb300 import workloads as wl
from tests.helpers import THETA, check_storage_error, oracle_run, rel_linf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09472_gb300.build import build

    build()


# (lattice, shape, storage): the longest general row, the shortest staged one, a whole number of 8 columns and one
# more; then whole rows at their longest and the first segmented ones, with ragged last segments
CASES = [("D2V9", (6, 31), "f32"), ("D2V9", (6, 32), "f16"), ("D2V9", (5, 33), "f32"), ("D2V9", (5, 41), "f16"),
         ("D2V9", (5, 904), "f32"), ("D2V9", (5, 905), "f32"), ("D2V9", (3, 1816), "f16"), ("D2V9", (3, 1821), "f16"),
         ("D2V9", (2, 4096), "bf16"), ("D2V9", (700, 1025), "f32"), ("D3V19", (3, 4, 424), "f32"),
         ("D3V19", (3, 4, 433), "f32"), ("D3V19", (3, 3, 865), "f16"), ("D3V27", (3, 4, 305), "f32"),
         ("D3V27", (2, 3, 609), "f16"), ("D1V3", (2040,), "f32"), ("D1V3", (2041,), "f32"), ("D1V3", (2048,), "f16")]


def _case(vel, shape, seed):
    N, D = int(np.prod(shape)), len(shape)
    solid = (wl.uniform01(seed, N) < 0.15).reshape(shape).astype(np.uint8)
    solid[..., -1] = wl.uniform01(seed + 5, N // shape[-1]).reshape(shape[:-1]) < 0.5  # links across the wrap
    rho = (1.0 + 0.02 * (wl.uniform01(seed + 1, N) - 0.5)).reshape(shape).astype(np.float32)
    u = (0.01 * wl.normal(seed + 2, D * N)).reshape((D,) + tuple(shape)).astype(np.float32)
    Ef = (1e-4 * (1.0 + 0.1 * wl.normal(seed + 3, D * N))).reshape((D,) + tuple(shape)).astype(np.float32)
    B = {1: (0, 0, 0), 2: (0, 0, 2e-3), 3: (1e-3, -2e-3, 3e-3)}[D]
    return solid, rho, u, Ef, B


def _run(vel, shape, storage, force, case, calls, local_mu=False, seed=0):
    """A run of the given lbm_step calls; its simulation and the fields after it."""
    from paper_1710_09472_gb300.lbm import LBM

    solid, rho, u, Ef, B = case
    sim = LBM(vel, tuple(reversed(shape)), 0.8, B=B, storage=storage, force=force)
    sim.set_geometry(torch.from_numpy(solid.reshape(-1)).cuda())
    sim.set_E_field(torch.from_numpy(Ef.reshape(-1)).cuda())
    if seed:
        sim.set_rounding_seed(seed)
    if local_mu:
        sim.set_local_mu(True)
    sim.init_equilibrium(torch.from_numpy(rho.reshape(-1)).cuda(), torch.from_numpy(u.reshape(-1)).cuda())
    for n in calls:
        sim.step(n)
    r = torch.empty(sim.N, device="cuda")
    j = torch.empty(sim.D * sim.N, device="cuda")
    tot = sim.moments(r, j)
    return r.cpu().numpy().reshape(shape), j.cpu().numpy().reshape((sim.D,) + tuple(shape)), tot, sim


@pytest.mark.parametrize("vel,shape,storage", CASES)
def test_step_and_totals(vel, shape, storage):
    """Single steps (the staged or general kernel) against the oracle; the same
    steps in one call (small boxes: one launch on a cluster) to the last bit."""
    case = _case(vel, shape, 81)
    solid, rho, u, Ef, B = case
    rg, jg, totg, sim = _run(vel, shape, storage, "term", case, [1] * 30)
    ro, jo, toto, _, _ = oracle_run(vel, shape, solid, 0.8, 30, "term", (0, 0, 0), B, rho, u, Ef)

    def rerun(seed):
        r, j, _, s = _run(vel, shape, storage, "term", case, [1] * 30, seed=seed)
        s.close()
        return rel_linf(r, ro), rel_linf(j, jo)

    check_storage_error(storage, (rel_linf(rg, ro), rel_linf(jg, jo)),
                        dict(vel=vel, shape=shape, solid=solid, tau=0.8, steps=30, force="term", E=(0, 0, 0), B=B,
                             rho=rho, u=u, Efield=Ef, reference=(ro, jo)), label=f"units {vel} {shape}",
                        gpu_rerun=rerun)
    # the FP64 total of FP32 (16-bit) cells: rounding of the stored values only
    assert abs(totg[0] / toto[0] - 1) < {"f32": 1e-6, "f16": 1e-5, "bf16": 1e-4}[storage]
    _, _, _, many = _run(vel, shape, storage, "term", case, [30])
    np.testing.assert_array_equal(many.populations(deviation=True), sim.populations(deviation=True))
    sim.close()
    many.close()


# boxes stepped in one launch: one cell, one block, several blocks and walls across the wrap, every lattice, on a
# cluster and (from the third D2V9 box on, and 24 x 25 x 26) on a cooperative grid, the last one too large for either
SMALL = [("D2V9", (1, 1), "f32"), ("D2V9", (3, 5), "f16"), ("D2V9", (64, 32), "f32"), ("D2V9", (8, 4096), "bf16"),
         ("D2V9", (100, 331), "f32"), ("D3V19", (2, 3, 5), "bf16"), ("D3V19", (24, 25, 26), "f32"),
         ("D3V27", (12, 13, 14), "f16"), ("D1V3", (33,), "f32"), ("D1V3", (40000,), "f16"), ("D1V3", (90001,), "f32"),
         ("D3V27", (17, 30, 31), "bf16"), ("D3V19", (48, 50, 50), "f16")]


@pytest.mark.parametrize("vel,shape,storage", SMALL)
@pytest.mark.parametrize("force", ["term", "shift"])
def test_steps_in_one_launch(vel, shape, storage, force):
    case = _case(vel, shape, 61)
    local = vel in ("D2V9", "D3V19") and force == "shift"
    _, _, _, one = _run(vel, shape, storage, force, case, [1] * 13, local)
    _, _, _, many = _run(vel, shape, storage, force, case, [2, 11], local)
    np.testing.assert_array_equal(many.populations(deviation=True), one.populations(deviation=True))
    before = many.launch_count()
    many.step(6)
    assert many.launch_count() == before + (1 if np.prod(shape) < 90000 or vel == "D1V3" else 6)
    one.step(5)
    one.step(1)
    np.testing.assert_array_equal(many.populations(deviation=True), one.populations(deviation=True))
    one.close()
    many.close()


@pytest.mark.parametrize("vel,shape,storage", [c for c in CASES if c[2] == "f32" and np.prod(c[1]) < 10000])
def test_reverse_step(vel, shape, storage):
    from paper_1710_09472_gb300.lbm import LBM

    solid, rho, u, Ef, B = _case(vel, shape, 91)
    D, N, T = len(shape), int(np.prod(shape)), 6
    wj = wl.normal(95, D * N).reshape((D,) + shape).astype(np.float32)
    wr = wl.normal(96, N).reshape(shape).astype(np.float32)
    sim = LBM(vel, tuple(reversed(shape)), 0.75, B=B, storage=storage)
    sim.set_geometry(torch.from_numpy(solid.reshape(-1)).cuda())
    sim.set_E_field(Ef.reshape(-1))  # from the host
    sim.init_equilibrium(torch.from_numpy(rho.reshape(-1)).cuda(), torch.from_numpy(u.reshape(-1)).cuda())
    dE = torch.empty(D * N, dtype=torch.float64, device="cuda")
    lam0 = torch.empty(sim.Q * N, dtype=torch.float32, device="cuda")
    res = sim.adjoint(2, T, torch.from_numpy(wr.reshape(-1)).cuda(), torch.from_numpy(wj.reshape(-1)).cuda(),
                      checkpoint_every=2, dL_dE=dE, dL_df0=lam0)
    m = oracle.Model(vel, "fd", THETA, 1.0, tau=0.75, B=B, force="term")
    f0 = m.init_equilibrium(shape, solid, rho.astype(np.float64), u.astype(np.float64))
    states = m.trajectory(shape, solid, f0, T, Ef.astype(np.float64))
    ref = m.adjoint(shape, solid, states, 2, T, wr.astype(np.float64), wj.astype(np.float64), Ef.astype(np.float64))
    # 1e-4: the bound of the reverse step in every other test; the loss is a signed sum, so against its terms' size
    assert rel_linf(dE.cpu().numpy().reshape(ref["gE"].shape), ref["gE"]) < 1e-4
    assert rel_linf(lam0.cpu().numpy(), ref["lam0"]) < 1e-4
    assert abs(res["loss"] - ref["loss"]) < 1e-5 * 4 * float(np.abs(wr).sum())
    sim.close()


@pytest.mark.parametrize("shape,storage", [((4, 5, 37), "f32"), ((4, 5, 37), "f16"), ((3, 4, 40), "f32"),
                                           ((2, 3, 301), "f32"), ((3, 4, 20), "f16")])
def test_saved_state_holds_unpadded_rows(shape, storage):
    """The populations of a saved state are the rows in slot order, nx values
    per direction, whatever the pitch in device memory; loading brings the
    state back bit for bit."""
    from paper_1710_09472_gb300.lbm import LBM

    N, dims = int(np.prod(shape)), tuple(reversed(shape))
    _, rho, u, _, B = _case("D3V19", shape, 71)
    sims = [LBM("D3V19", dims, 0.8, E=(1e-4, 0, 0), B=B, storage=storage) for _ in range(2)]
    for s in sims:
        s.init_equilibrium(torch.from_numpy(rho.reshape(-1)).cuda(), torch.from_numpy(u.reshape(-1)).cuda())
    sims[0].step(5)
    blob = sims[0].save_state()
    Q, eb = sims[0].Q, 4 if storage == "f32" else 2
    header = 64
    payload = struct.unpack_from("<Q", blob, 48)[0]
    assert len(blob) == header + payload and payload >= Q * N * eb
    P = np.frombuffer(blob, dtype=np.float32 if eb == 4 else np.float16, count=Q * N, offset=header)
    P = P.astype(np.float32).reshape(shape[0], shape[1], Q, shape[2]) / (1.0 if eb == 4 else 4096.0)
    e = oracle.Model("D3V19", "fd", THETA, 1.0, tau=0.8).e
    order = sorted(range(Q), key=lambda a: (3 * (e[a][1] + 1) + e[a][2] + 1, a))
    h = sims[0].populations(deviation=True).reshape((Q,) + shape)
    for s, a in enumerate(order):  # no solid cells: f_a(x) = P_a(x - e_a)
        np.testing.assert_array_equal(np.roll(P[:, :, s], (e[a][2], e[a][1], e[a][0]), (0, 1, 2)), h[a])
    sims[1].load_state(blob)
    for s in sims:
        s.step(3)
    np.testing.assert_array_equal(sims[0].populations(), sims[1].populations())
    for s in sims:
        s.close()
