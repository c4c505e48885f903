"""Every kind of row-staged kernel against the FP64 oracle, each on a box that
reaches it (a unit for every SM and single steps; smaller boxes, and many steps
in one call, run other kernels), with the kernel that ran asserted: exact rows,
padded rows and segments, compile-time and run-time strides, each storage and
rounding, the four lattices and the local chemical-potential model; the fields
from the same stages; and the reverse steps, staged and general."""
import numpy as np
import pytest

import oracle
from paper_1710_09472_gb300 import workloads as wl
from tests.helpers import THETA, rel_linf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09472_gb300.build import build

    build()


def _inputs(vel, shape, seed):
    N, D = int(np.prod(shape)), len(shape)
    solid, _ = wl.boolean_obstacles(shape, 2.5, 0.75, seed=seed) if D > 1 else (
        (wl.uniform01(seed, N) < 0.15).reshape(shape).astype(np.uint8), None)
    # solid cells at the ends of rows: links across the wrap and beside segments
    solid[..., -1] |= (wl.uniform01(seed + 1, N // shape[-1]).reshape(shape[:-1]) < 0.5).astype(np.uint8)
    rho = (1.0 + 0.02 * (wl.uniform01(seed + 2, N) - 0.5)).reshape(shape).astype(np.float32)
    u = (0.01 * wl.normal(seed + 3, D * N)).reshape((D,) + tuple(shape)).astype(np.float32)
    Ef = (1e-4 * (1.0 + 0.1 * wl.normal(seed + 4, D * N))).reshape((D,) + tuple(shape)).astype(np.float32)
    B = {1: (0, 0, 0), 2: (0, 0, 2e-3), 3: (1e-3, -2e-3, 3e-3)}[D]
    return solid, rho, u, Ef, B


def _sim(vel, shape, storage, force, inputs, efield, tau=0.8, **weight):
    from paper_1710_09472_gb300.lbm import LBM

    solid, rho, u, Ef, B = inputs
    sim = LBM(vel, tuple(reversed(shape)), tau, E=(2e-4, 0, 0), B=B, storage=storage, force=force, **weight)
    sim.set_geometry(torch.from_numpy(solid.reshape(-1)).cuda())
    if efield:
        sim.set_E_field(torch.from_numpy(Ef.reshape(-1)).cuda())
    sim.init_equilibrium(torch.from_numpy(rho.reshape(-1)).cuda(), torch.from_numpy(u.reshape(-1)).cuda())
    return sim


# (lattice, shape, storage, force, per-cell E, kernel)
STEPS = [
    ("D3V19", (16, 10, 256), "f32", "term", False, ("exact", 256)),
    ("D3V19", (16, 10, 256), "f32", "shift", True, ("exact", 256)),
    ("D3V19", (16, 10, 256), "f16", "term", False, ("exact", 256)),
    ("D3V19", (16, 10, 256), "f16", "shift", True, ("exact", 256)),
    ("D3V19", (16, 10, 256), "bf16", "term", True, ("exact", 256)),
    ("D3V19", (16, 10, 250), "f32", "term", True, ("rows", 256)),
    ("D3V19", (16, 10, 250), "f16", "term", False, ("rows", 256)),
    ("D3V19", (16, 10, 250), "f16", "shift", True, ("rows", 256)),
    ("D3V19", (16, 10, 250), "bf16", "term", False, ("rows", 256)),
    ("D3V19", (16, 10, 512), "f16", "term", False, ("exact", 512)),
    ("D3V19", (16, 10, 512), "f32", "term", False, ("segments", 256)),
    ("D3V19", (16, 10, 33), "f16", "shift", False, ("rows", 0)),
    ("D3V19", (16, 10, 200), "f32", "shift", False, ("rows", 0)),
    ("D3V19", (16, 10, 200), "bf16", "term", True, ("rows", 0)),
    ("D3V19", (9, 10, 490), "f32", "shift", True, ("segments", 256)),
    ("D3V19", (9, 9, 433), "f32", "term", False, ("segments", 0)),
    ("D3V19", (6, 10, 1000), "f16", "term", True, ("segments", 256)),
    ("D3V19", (6, 9, 865), "bf16", "shift", False, ("segments", 0)),
    ("D3V27", (16, 10, 256), "f16", "term", True, ("exact", 256)),
    ("D3V27", (16, 10, 256), "bf16", "shift", False, ("exact", 256)),
    ("D3V27", (16, 10, 256), "f32", "term", False, ("rows", 0)),
    ("D3V27", (16, 10, 250), "f16", "shift", False, ("rows", 0)),
    ("D3V27", (9, 10, 305), "f32", "term", True, ("segments", 0)),
    ("D3V27", (6, 9, 609), "f16", "term", False, ("segments", 0)),
    ("D2V9", (160, 256), "f32", "term", False, ("exact", 256)),
    ("D2V9", (160, 256), "f16", "shift", True, ("exact", 256)),
    ("D2V9", (160, 512), "f32", "shift", True, ("exact", 512)),
    ("D2V9", (160, 512), "bf16", "term", False, ("exact", 512)),
    ("D2V9", (160, 200), "f16", "term", True, ("rows", 0)),
    ("D2V9", (160, 903), "f32", "term", False, ("rows", 0)),
    ("D2V9", (80, 1500), "f32", "term", True, ("segments", 512)),
    ("D2V9", (40, 2048), "f16", "term", False, ("segments", 512)),
    ("D2V9", (40, 2047), "bf16", "shift", True, ("segments", 512)),
    ("D2V9", (80, 1025), "f32", "shift", False, ("segments", 0)),
    ("D1V3", (100000,), "f32", "term", True, ("segments", 0)),
    ("D1V3", (100001,), "f16", "shift", False, ("segments", 0)),
]
# the same with nearest rounding, and the local chemical-potential model
NEAREST = [("D3V19", (16, 10, 256), "f16", "term", False, ("exact", 256)),
           ("D3V19", (16, 10, 250), "bf16", "term", True, ("rows", 0)),
           ("D3V27", (16, 10, 256), "f16", "shift", True, ("rows", 0)),
           ("D2V9", (40, 2048), "f16", "term", False, ("segments", 512))]
LOCAL = [("D2V9", (160, 256), "f32", "term", False, ("exact", 256)),
         ("D2V9", (160, 256), "f16", "shift", True, ("exact", 256)),
         ("D2V9", (160, 250), "bf16", "term", True, ("rows", 0)),
         ("D2V9", (80, 1025), "f32", "shift", False, ("segments", 0))]
PARAMS = [c + (None,) for c in STEPS] + [c + ("nearest",) for c in NEAREST] + [c + ("local",) for c in LOCAL]


@pytest.mark.parametrize("vel,shape,storage,force,efield,kernel,option", PARAMS)
def test_one_step_and_fields(vel, shape, storage, force, efield, kernel, option):
    """The whole state after one staged step from a state that the GPU made
    against the oracle's step from the same state, and the fields of it.

    Each value is off by the rounding of its store (an ulp when stochastic, half
    one when nearest: 2^-10 and 2^-7 of the value for FP16 and BF16) and the FP32
    arithmetic (1e-5 of the largest deviation, the bound of the sampled
    one-step tests)."""
    inputs = _inputs(vel, shape, 21)
    solid, rho, u, Ef, B = inputs
    weight = dict(theta=0.5, mu=0.0) if option == "local" else dict(theta=THETA, mu=1.0)
    sim = _sim(vel, shape, storage, force, inputs, efield, **weight)
    if option == "nearest":
        sim.set_rounding(False)
    if option == "local":
        sim.set_local_mu(True)
    for _ in range(3):
        sim.step(1)
    m = oracle.Model(vel, "fd", weight["theta"], weight["mu"], tau=0.8, E=(2e-4, 0, 0), B=B, force=force)
    Q, N, D = sim.Q, sim.N, sim.D
    f0 = (m.w / m.const["I0"])[:, None] * (solid.reshape(1, N) == 0)
    f = f0 + sim.populations(deviation=True).reshape(Q, N).astype(np.float64)
    f = np.ascontiguousarray(f.reshape(-1))
    sim.step(1)
    assert sim.last_kernel("step") == ("staged",) + kernel
    got = sim.populations(deviation=True).reshape(Q, N).astype(np.float64)
    E64 = Ef.astype(np.float64) if efield else None
    if option == "local":
        m.step_local_mu(shape, solid, f, 1, E64, rho_ref=1.0)
    else:
        m.step(shape, solid, f, 1, E64)
    want = f.reshape(Q, N) - f0
    ulp = {"f32": 0.0, "f16": 2.0**-10, "bf16": 2.0**-7}[storage] * (0.5 if option == "nearest" else 1.0)
    err = np.abs(got - want) - ulp * np.abs(want)
    assert err.max() <= 1e-5 * np.abs(want).max(), (err.max(), np.unravel_index(err.argmax(), err.shape))
    # the fields: sums of the stored values in FP32
    r, j = torch.full((N,), -1.0, device="cuda"), torch.full((D * N,), -1.0, device="cuda")
    total, total_j = sim.moments(r, j)
    assert sim.last_kernel("moments") == ("staged", "segments" if kernel[0] == "segments" else "rows", 0)
    fluid = solid.reshape(N) == 0
    r, j = r.cpu().numpy().astype(np.float64), j.cpu().numpy().astype(np.float64).reshape(D, N)
    want_r = np.where(fluid, 1.0 + got.sum(0), 0.0)
    want_j = np.stack([sum(m.e[a][d] * got[a] for a in range(Q)) for d in range(D)]) / m.const["cs"]
    assert np.abs(r - want_r).max() < 1e-6
    assert np.abs(j - want_j).max() < 1e-6 * np.abs(got).sum(0).max()
    assert abs(total - r.sum()) < 1e-10 * N
    assert np.abs(total_j[:D] - j.sum(1)).max() < 1e-10 * N
    sim.close()


@pytest.mark.parametrize("dims,kernel", [((256, 16, 10), ("exact", 256)), ((250, 16, 10), ("rows", 0))])
def test_local_mu_3d(dims, kernel):
    """The local model on D3V19 at the paper's copper values: with a weight whose
    thetabar does not depend on mu it has the default model's states to FP32
    rounding (every cell), and sampled cells of one step agree with the oracle."""
    from tests.test_local_mu_gpu import test_local_mu_3d_sampled_step

    test_local_mu_3d_sampled_step(dims)
    shape = tuple(reversed(dims))
    inputs = _inputs("D3V19", shape, 33)
    states = []
    for local in (False, True):
        sim = _sim("D3V19", shape, "f32", "term", inputs, True, stat="mb", theta=1.0, mu=0.0)
        sim.set_local_mu(local)
        for _ in range(4):
            sim.step(1)
        if local:
            assert sim.last_kernel("step") == ("staged",) + kernel
        states.append(sim.populations(deviation=True))
        sim.close()
    assert rel_linf(states[1], states[0]) < 1e-6


# the reverse step has no smallest number of units: small boxes; rows below 32 cells are the general kernel's
REVERSE = [("D3V19", (2, 3, 256), ("staged", "exact", 256)), ("D3V19", (2, 3, 250), ("staged", "rows", 0)),
           ("D3V19", (2, 3, 512), ("staged", "segments", 256)), ("D2V9", (3, 256), ("staged", "exact", 256)),
           ("D2V9", (3, 512), ("staged", "exact", 512)), ("D2V9", (2, 1500), ("staged", "segments", 512)),
           ("D3V27", (2, 3, 256), ("staged", "rows", 0)), ("D3V27", (2, 3, 305), ("staged", "segments", 0)),
           # narrow rows in numbers: more than eight blocks are resident per SM
           ("D2V9", (2048, 64), ("staged", "rows", 0)), ("D3V19", (64, 64, 32), ("staged", "rows", 0)),
           ("D2V9", (8200, 40), ("staged", "rows", 0)),
           ("D3V19", (4, 5, 31), ("general", None, 0)), ("D3V27", (4, 5, 30), ("general", None, 0)),
           ("D1V3", (31,), ("general", None, 0)), ("D2V9", (9, 31), ("general", None, 0))]


@pytest.mark.parametrize("vel,shape,kernel", REVERSE)
@pytest.mark.parametrize("force", ["term", "shift"])
def test_reverse_step(vel, shape, kernel, force):
    """dL/dE per cell, dL/df_0, dL/dB and dL/dtau to 1e-4, the bound of the other
    reverse tests; the local model too where it has a closed form."""
    inputs = _inputs(vel, shape, 51)
    solid, rho, u, Ef, B = inputs
    D, N, T, tb = len(shape), int(np.prod(shape)), 6, 2
    wr = wl.normal(56, N).reshape(shape).astype(np.float32)
    wj = wl.normal(57, D * N).reshape((D,) + shape).astype(np.float32)
    E64 = Ef.astype(np.float64)
    for local in (False, True) if vel == "D2V9" else (False,):
        weight = dict(theta=0.5, mu=0.0) if local else dict(theta=THETA, mu=1.0)
        sim = _sim(vel, shape, "f32", force, inputs, True, tau=0.75, **weight)
        if local:
            sim.set_local_mu(True)
        dE = torch.empty(D * N, dtype=torch.float64, device="cuda")
        lam0 = torch.empty(sim.Q * N, dtype=torch.float32, device="cuda")
        res = sim.adjoint(tb, T, torch.from_numpy(wr.reshape(-1)).cuda(), torch.from_numpy(wj.reshape(-1)).cuda(),
                          checkpoint_every=3, dL_dE=dE, dL_df0=lam0)
        ran = sim.last_kernel("reverse")
        if local and kernel[0] == "staged":  # run-time strides
            assert ran == ("staged", "segments" if kernel[1] == "segments" else "rows", 0)
        else:
            assert ran == kernel
        m = oracle.Model(vel, "fd", weight["theta"], weight["mu"], tau=0.75, B=B, force=force)
        f = m.init_equilibrium(shape, solid, rho.astype(np.float64), u.astype(np.float64))
        if local:
            states = np.empty((T + 1, f.size))
            states[0] = f
            for t in range(T):
                m.step_local_mu(shape, solid, f, 1, E64, rho_ref=1.0)
                states[t + 1] = f
            ref = m.adjoint_local_mu(shape, solid, states, tb, T, wr.astype(np.float64), wj.astype(np.float64), E64,
                                     rho_ref=1.0)
        else:
            states = m.trajectory(shape, solid, f, T, E64)
            ref = m.adjoint(shape, solid, states, tb, T, wr.astype(np.float64), wj.astype(np.float64), E64)
        assert rel_linf(dE.cpu().numpy().reshape(ref["gE"].shape), ref["gE"]) < 1e-4
        assert rel_linf(lam0.cpu().numpy(), ref["lam0"]) < 1e-4
        # signed sums over cells and steps: against the size of their terms
        terms = float(np.abs(wr).sum() + np.abs(wj).sum()) * (T - tb)
        assert abs(res["loss"] - ref["loss"]) < 1e-6 * terms
        assert abs(res["dL_dtau"] - ref["gtau"]) < 1e-4 * max(abs(ref["gtau"]), 1e-4 * terms)
        for d in range(3) if D == 3 else ([2] if D == 2 else []):
            assert abs(res["dL_dB"][d] - ref["gB"][d]) < 1e-4 * max(abs(ref["gB"][d]), 1e-2 * np.abs(ref["gB"]).max())
        sim.close()


def test_smoke_reaches_the_benchmarked_kernel():
    """What runs a box this size is the exact-row kernel of the benchmark."""
    sim = _sim("D3V19", (20, 20, 256), "f16", "term", _inputs("D3V19", (20, 20, 256), 61), False)
    sim.step(10)
    assert sim.last_kernel("step") == ("staged", "exact", 256)
    sim.close()
