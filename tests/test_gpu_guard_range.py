"""The mixed push of the cell rows on the axes, all in pairs of FP32 numbers, where a unit takes
its factors out of FP32's range: photons' momenta, whose squares leave it first, and charges that
only times the weight are of order 1. Against the FP64 oracle on FP32-rounded inputs; tolerance
1e-5 per step, as for every mixed push (test_gpu_mixed.py)."""
import numpy as np
import pytest

import workloads as W
from oracle import oracle as O
from paper_2511_17701_gb300.binding import J01
from parity import gpu_from_oracle, particle_errors, round_state_fp32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def axis_rows(cfg, n, seed):
    rng = np.random.default_rng(seed)
    pos = dict(i1=rng.integers(2, cfg["n_r"] - 2, n).astype(np.int32),
               i2=rng.choice([0, cfg["n_theta"] - 1], n).astype(np.int32),
               dx1=rng.uniform(0.0, 1.0, n), dx2=rng.uniform(0.15, 0.85, n))
    return pos, rng.standard_normal((3, n))


@pytest.mark.parametrize("umag", [1e-30, 1e-22, 1.0, 1e22, 1e30])
@pytest.mark.parametrize("over", [dict(), dict(n_theta=48, r0=0.3, h0=0.5)])
def test_photon_momentum_unit(torch_cuda, umag, over):
    cfg = dict(W.grid_config("wald64", **over), precision="mixed")
    osim = O.OracleSim(cfg)
    osim.init_fields(O.FIELD_WALD, 1.0)
    n = 2000
    pos, uh = axis_rows(cfg, n, 3)
    osim.add_species(pos, uh * umag, 0.1 * np.ones(n), 1.0, 0.0, massless=True)
    round_state_fp32(osim)
    g = gpu_from_oracle(osim, massless=[0])
    osim.predict()
    g.predict()
    osim.push(0)
    g.push(0)
    err = particle_errors(g.get_particles(0), osim.species[0].view())
    assert max(err.values()) <= 1e-5, err


@pytest.mark.parametrize("qc,w", [(0.2, 0.1), (1e-42, 1e36), (1e42, 1e-30)])
def test_charge_unit(torch_cuda, qc, w):
    cfg = dict(W.grid_config("wald64"), precision="mixed")
    osim = O.OracleSim(cfg)
    osim.init_fields(O.FIELD_WALD, 1.0)
    n = 2000
    pos, uh = axis_rows(cfg, n, 5)
    osim.add_species(pos, uh, w * np.ones(n), 1.0, qc)
    round_state_fp32(osim)
    g = gpu_from_oracle(osim, sort_every=0)
    osim.predict()
    osim.push(0)
    osim.deposit()
    g.step(1)
    F = g.planes()
    for c in range(3):
        e = np.abs(F[J01 + c].astype(np.float64) - osim.F[O.J1 + c]).max()
        assert e <= 1e-5 * osim.F[O.JA1 + c].max(), (c, e)
