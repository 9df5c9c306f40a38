"""FP64 pushes of particles whose charge, momentum or field lies outside what a pair of FP32
numbers resolves: the units of charge, of a photon's momentum and of the field are the caller's.
One step at a small iter_tol, which takes the push's increment form, against the oracle. Tolerance:
1e-12 relative per step, as for every FP64 push (tests/parity.py); all results scale with the
unit, so the same relative bound holds in each."""
import numpy as np
import pytest

import workloads as W
from oracle import oracle as O
from paper_2511_17701_gb300.binding import J01
from parity import assert_particles, gpu_from_oracle, oracle_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def particles(cfg, n, seed, umag):
    rng = np.random.default_rng(seed)
    pos = dict(i1=rng.integers(3, cfg["n_r"] - 2, n).astype(np.int32),
               i2=rng.integers(1, cfg["n_theta"] - 1, n).astype(np.int32),
               dx1=rng.random(n), dx2=rng.random(n))
    uh = rng.standard_normal((3, n))
    return pos, uh * umag / np.linalg.norm(uh, axis=0)


@pytest.mark.parametrize("k", [-800, -130, -107, -80, 120, 127, 700])
def test_charge_unit(torch_cuda, k):
    """A charge 2^k times as large deposits 2^k times the current: every contribution exactly,
    their sums up to the order of the additions (a few of them per node, 2^-53 each; the nodes'
    sums of absolute values are the oracle's)."""
    cfg = W.grid_config("wald64")
    osim = O.OracleSim(cfg)
    osim.init_fields(O.FIELD_WALD, 1.0)
    n = 4000
    pos, uh = particles(cfg, n, 3, 1.0)
    osim.add_species(pos, uh, 0.1 * np.ones(n), 1.0, -0.2)
    g = gpu_from_oracle(osim, iter_tol=1e-12, sort_every=0)
    J = []
    for scale in (1.0, 2.0 ** k):
        g.set_planes(osim.F)
        g.set_particles(0, osim.species[0].view(), 1.0, -0.2 * scale)
        g.step(1)
        J.append(g.planes()[J01:J01 + 3] / scale)
    osim.predict()
    osim.push(0)
    osim.deposit()
    assert np.abs(J[0]).max() > 0.0
    assert np.all(np.abs(J[1] - J[0]) <= 2.0 ** -50 * osim.F[O.JA1:O.JA1 + 3])


@pytest.mark.parametrize("umag", [1e30, 1e3, 1e-3, 1e-14, 1e-18, 1e-30])
def test_photon_momentum_unit(torch_cuda, umag):
    cfg = W.grid_config("wald64")
    osim = O.OracleSim(cfg)
    osim.init_fields(O.FIELD_WALD, 1.0)
    n = 4000
    pos, uh = particles(cfg, n, 5, umag)
    osim.add_species(pos, uh, 0.1 * np.ones(n), 1.0, 0.0, massless=True)
    g = gpu_from_oracle(osim, iter_tol=1e-12, massless=[0])
    osim.predict()
    g.predict()
    osim.push(0)
    g.push(0)
    assert_particles(g.get_particles(0), osim.species[0].view())


@pytest.mark.parametrize("B0,qm", [(1e-22, 1e20), (1e-27, 1e24), (1e-35, 1e35), (1e25, 1e-25)])
def test_field_unit(torch_cuda, B0, qm):
    cfg = W.grid_config("wald64")
    osim = O.OracleSim(cfg)
    osim.init_fields(O.FIELD_WALD, B0)
    n = 4000
    pos, uh = particles(cfg, n, 7, 0.3)
    osim.add_species(pos, uh, 0.1 * np.ones(n), qm, 0.2)
    g = gpu_from_oracle(osim, iter_tol=1e-12)
    osim.predict()
    g.predict()
    osim.push(0)
    g.push(0)
    assert_particles(g.get_particles(0), osim.species[0].view())


def test_small_moves_next_to_the_corner(torch_cuda):
    """The flux of one slow particle in the first cells, where positions carry up to 53 bits: J^1
    and J^2 summed over their two nodes against the oracle. Both sides take end points rounded to
    absolute positions below 4 (2^-51 apart where they round differently) and a midpoint rounded
    by 2^-52, each times q / dt."""
    cfg = W.grid_config("wald64", metric="ks0", a=0.0, r_min=3.0, r_max=30.0, r_absorb=27.0)
    rng = np.random.default_rng(17)
    sim = None
    for _ in range(60):
        osim = O.OracleSim(cfg)
        osim.init_fields(O.FIELD_WALD, 0.0)
        pos = dict(i1=rng.integers(1, 4, 1).astype(np.int32), i2=rng.integers(2, 4, 1).astype(np.int32),
                   dx1=rng.uniform(0.6, 0.9, 1), dx2=rng.uniform(0.6, 0.9, 1))
        osim.add_species(pos, 1e-3 * rng.standard_normal((3, 1)), np.ones(1), 0.0, 1.0)
        sp = osim.species[0]
        if sim is None:
            sim = gpu_from_oracle(osim, iter_tol=1e-16, sort_every=0)
        sim.set_particles(0, sp.view(), sp.qm, sp.qc)
        q = float(sp.view()["w"][0])
        osim.predict()
        osim.push(0)
        osim.deposit()
        sim.step(1)
        for c in range(2):
            flux = float(sim.plane(J01 + c).sum()), float(osim.F[O.J1 + c].sum())
            assert abs(flux[0] - flux[1]) <= 2.0 ** -50 * q / osim.dt, (c, flux)


def test_continuity(torch_cuda):
    """Full steps of the increment form conserve charge as those of the general push do
    (tests/test_gpu_charge.py, the same bound)."""
    g = gpu_from_oracle(oracle_state(W.grid_config("wald64")), iter_tol=1e-12)
    for _ in range(3):
        g.step(1)
        res, drho, _, scale = g.charge_check(after_step=True)
        assert drho > 1e-3
        assert res / scale < 1e-13, (res, drho, scale)


@pytest.mark.parametrize("n_theta", [48, 64, 1024, 2048])
@pytest.mark.parametrize("massless", [False, True])
def test_rows_on_the_axes(torch_cuda, n_theta, massless):
    """The two rows next to each axis, among them particles closer to theta = pi than
    n_theta 2^-10 cells, which the general routine keeps, and ones on either side of that."""
    cfg = W.grid_config("wald64", n_theta=n_theta)
    osim = O.OracleSim(cfg)
    osim.init_fields(O.FIELD_WALD, 1.0)
    rng = np.random.default_rng(23)
    n = 4000
    near = n_theta * 2.0 ** -10
    d = np.where(rng.random(n) < 0.5, rng.uniform(0.0, 2.0, n), near * rng.uniform(0.5, 1.5, n))
    d = np.clip(d, 0.02, 1.98)
    x2 = np.where(rng.random(n) < 0.7, n_theta - d, d)
    pos = dict(i1=rng.integers(3, cfg["n_r"] - 2, n).astype(np.int32), i2=np.floor(x2).astype(np.int32),
               dx1=rng.random(n), dx2=x2 - np.floor(x2))
    uh = rng.standard_normal((3, n))
    osim.add_species(pos, uh / np.linalg.norm(uh, axis=0), 0.1 * np.ones(n), 1.0, 0.2, massless=massless)
    g = gpu_from_oracle(osim, iter_tol=1e-12, massless=[0] if massless else [])
    osim.predict()
    g.predict()
    osim.push(0)
    g.push(0)
    assert_particles(g.get_particles(0), osim.species[0].view())
