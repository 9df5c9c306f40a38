"""The FP64 push's increment form at the edges of what it covers, against the oracle: one push
of particles on either side of each bound (grids whose offsets exceed the series' range, radii
above FP32's safe range, fields that turn the momentum by more than the form takes, mixed in
one warp with ones that do not, the rows next to the axes, offsets at the corners and halves of
a cell, particles at rest, photons). Tolerance: 1e-12 relative per step, as for every FP64 push
(tests/parity.py); the particle order in memory mixes all kinds, so warps hold several."""
import numpy as np
import pytest

import workloads as W
from oracle import oracle as O
from parity import assert_particles, gpu_from_oracle

pytestmark = pytest.mark.gpu

@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def particles(cfg, massless, n, seed):
    """n particles over the grid, a part of them in the rows and at the offsets where the form
    ends, with momenta of 0.3 to 3 (and a few 0)."""
    rng = np.random.default_rng(seed)
    i1 = rng.integers(3, cfg["n_r"] - 2, n).astype(np.int32)
    i2 = rng.integers(2, cfg["n_theta"] - 2, n).astype(np.int32)
    edge = rng.integers(0, 6, n)
    i2[edge == 0] = rng.choice([1, 2, 3, cfg["n_theta"] - 4, cfg["n_theta"] - 3, cfg["n_theta"] - 2],
                               (edge == 0).sum())
    dx1, dx2 = rng.random(n), rng.random(n)
    dx1[edge == 1] = 0.0
    dx2[edge == 2] = 0.0
    dx1[edge == 3] = 0.5
    dx2[edge == 3] = np.nextafter(0.5, 0.0)
    dx1[edge == 4] = np.nextafter(1.0, 0.0)
    uh = rng.standard_normal((3, n))
    uh *= 10.0 ** rng.uniform(-0.5, 0.5, n) / np.linalg.norm(uh, axis=0)
    if not massless:
        uh[:, :5] = 0.0
    return dict(i1=i1, i2=i2, dx1=dx1, dx2=dx2), uh


@pytest.mark.parametrize("over,qm", [
    (dict(), 1.0),                                    # the form's own ground
    (dict(n_r=20, n_theta=96, r_min=1.0, r_max=40.0), 1.0),  # radial offsets beyond the series
    (dict(n_r=300, n_theta=40), -1.0),                # angular offsets beyond the series
    (dict(n_r=400, n_theta=64, r_max=2000.0, r_absorb=1800.0), 1.0),  # radii above 1024
    (dict(n_r=96, n_theta=96), 40.0),                 # increments around the form's bound
    (dict(n_r=96, n_theta=96), -2e4),                 # far above it
    (dict(n_r=200, n_theta=130, a=0.0, metric="ks0", r_min=3.0, r_max=30.0, r_absorb=27.0), 1.0),
])
@pytest.mark.parametrize("massless", [False, True])
def test_push_against_oracle(torch_cuda, over, qm, massless):
    if massless and abs(qm) > 1.0:
        pytest.skip("photons see no field")
    cfg = W.grid_config("wald64", **over)
    osim = O.OracleSim(cfg)
    osim.init_fields(O.FIELD_WALD, 1.0)
    pos, uh = particles(cfg, massless, 6000, 7)
    osim.add_species(pos, uh, 0.1 * np.ones(6000), qm, 0.2, 0.0, massless=massless)
    g = gpu_from_oracle(osim, iter_tol=1e-12, massless=[0] if massless else [])
    osim.predict()
    g.predict()
    osim.push(0)
    g.push(0)
    assert_particles(g.get_particles(0), osim.species[0].view())


def test_gathered_rest_gives_the_same_bits(torch_cuda):
    """Particles that the increment form leaves to the general routine are gathered over more
    particles per warp in large pushes than in small ones; a particle's result depends on
    neither: one push of 2^19 + 777 particles, and the same in pieces below 2^19."""
    from paper_2511_17701_gb300 import FIELD_WALD, Sim
    cfg = W.grid_config("wald64", n_r=96, n_theta=96, iter_tol=1e-12, sort_every=0)
    n = (1 << 19) + 777
    pos, uh = particles(cfg, False, n, 21)
    w0 = 0.1 * np.ones(n)

    def push(sel):
        g = Sim(cfg, [len(w0[sel])])
        g.init_metric()
        g.init_fields(FIELD_WALD, 1.0)
        g.load_particles(0, {k: v[sel] for k, v in pos.items()}, uh[:, sel], w0[sel], 3.0, 0.2)
        g.push(0)
        return g.get_particles(0)

    whole = push(slice(0, n))
    for a in range(0, n, 200001):
        sel = slice(a, min(n, a + 200001))
        part = push(sel)
        for k in ("i1", "i2", "dx1", "dx2", "u1", "u2", "u3", "phi", "tag"):
            assert np.array_equal(part[k], whole[k][sel]), k
