"""The field kernels at the sizes where a tile or a boundary write can go wrong, against the
oracle: rows and columns around multiples of the 64 x 4 tiles, the fewest rows the mirrors
need, horizon layers of several columns. Every stored point is compared, ghost rows and
horizon columns included. Tolerance: 1e-12 of each plane's maximum per step (both sides carry
rounding errors of ~1e-16 per operation, amplified by condition numbers up to ~1e2)."""
import numpy as np
import pytest

import workloads as W
from oracle import oracle as O
from parity import assert_planes, gpu_from_oracle, oracle_state

pytestmark = pytest.mark.gpu

R_H = W.horizon_radius(0.9)


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("n_r,n_th,n_f,qks", [
    (16, 4, 0, False), (59, 5, 0, False), (60, 7, 3, False), (123, 63, 1, False),
    (61, 64, 0, True), (64, 6, 5, False), (200, 11, 2, True)])
def test_vacuum_steps(torch_cuda, n_r, n_th, n_f, qks):
    over = dict(r0=0.3, h0=0.4) if qks else {}
    cfg = W.grid_config("wald64", n_r=n_r, n_theta=n_th, n_filter=n_f, r_min=0.55 * R_H,
                        r_max=12.0, r_absorb=9.0, **over)
    osim = oracle_state(cfg, species=0)
    rng = np.random.default_rng(n_r * 100 + n_th)
    j = np.arange(n_th)
    bump = 0.05 * rng.standard_normal((n_th, n_r)) * np.sin(np.pi * (j + 0.5) / n_th)[:, None] ** 3
    osim.F[2][O.G:O.G + n_th, O.G:O.G + n_r] += bump
    g = gpu_from_oracle(osim)
    for step in range(3):
        g.step(1)
        osim.step(1)
        assert_planes(g.planes(), osim.F, rtol=1e-12 * (step + 1), what="step %d" % step)
