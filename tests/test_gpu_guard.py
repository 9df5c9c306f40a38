"""The mixed push's guard zones (metric in pairs of floats next to the horizon and the axes, the
whole push in pairs in the rows on the axes) where their series and clamps end, against the FP64
oracle on FP32-rounded inputs: cells wider than the series' range, a small-angle clamp that
reaches into the first rows, quasi-spherical grids, photons. Tolerance 1e-5 per step, as for
every mixed push (test_gpu_mixed.py)."""
import numpy as np
import pytest

import workloads as W
from oracle import oracle as O
from parity import gpu_from_oracle, particle_errors, round_state_fp32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("over", [
    dict(),
    dict(n_r=14, n_theta=18, r_min=0.9, r_max=40.0, r_absorb=36.0),  # series out of range
    dict(small_angle=0.06),                                          # clamped rows
    dict(n_theta=48, r0=0.3, h0=0.5),
    dict(n_r=16, n_theta=20, r_min=0.9, r_max=30.0, r_absorb=27.0, r0=0.2, h0=-0.2),
])
@pytest.mark.parametrize("massless", [False, True])
def test_guard_zones_against_oracle(torch_cuda, over, massless):
    cfg = dict(W.grid_config("wald64", **over), precision="mixed")
    osim = O.OracleSim(cfg)
    osim.init_fields(O.FIELD_WALD, 1.0)
    rng = np.random.default_rng(3)
    n, nt, nr = 4000, cfg["n_theta"], cfg["n_r"]
    i2 = rng.choice([0, 1, 2, 3, 4, nt - 5, nt - 4, nt - 3, nt - 2, nt - 1], n)
    i2[n // 2:] = rng.integers(0, nt, n - n // 2)
    pos = dict(i1=rng.integers(2, nr - 2, n).astype(np.int32), i2=i2.astype(np.int32),
               dx1=rng.uniform(0.0, 1.0, n), dx2=rng.uniform(0.15, 0.85, n))
    uh = rng.standard_normal((3, n))
    osim.add_species(pos, uh, 0.1 * np.ones(n), 1.0, 0.2, 0.0, massless=massless)
    round_state_fp32(osim)
    g = gpu_from_oracle(osim, massless=[0] if massless else [])
    osim.predict()
    g.predict()
    osim.push(0)
    g.push(0)
    err = particle_errors(g.get_particles(0), osim.species[0].view())
    assert max(err.values()) <= 1e-5, err
