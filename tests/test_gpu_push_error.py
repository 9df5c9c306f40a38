"""The accuracy of the FP64 push's increment form where a step changes a particle's momentum by
more than a small part of it: cold particles, fields that turn or kick it by order one, the rows
next to the axes. At an iter_tol at FP64's rounding, against the oracle: the root mean square over
the particles of the error in the length of u, relative to it.

Bound: each side rounds u about 30 times (two passes through the tetrad frame, the geodesic
substep) by up to 2^-53 of it or of an increment of its own size, 2^-53 / sqrt(3) rms each, so
the two differ by sqrt(2 * 30 / 3) 2^-53 = 5e-16 of the larger of the two; a factor of 3 on top for the
metric's own rounding (its terms cancel by about that next to the horizon): 1.5e-15."""
import numpy as np
import pytest

import workloads as W
from oracle import oracle as O
from parity import gpu_from_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("umag,qm", [(1.0, 1.0), (0.1, 1.0), (1e-2, 1.0), (1e-3, 1.0), (1e-6, 1.0),
                                     (0.1, 0.0), (1e-3, 0.0), (1.0, 10.0), (1e-2, 10.0),
                                     (1.0, 100.0)])
def test_momentum_error(torch_cuda, umag, qm):
    cfg = W.grid_config("wald64")
    osim = O.OracleSim(cfg)
    osim.init_fields(O.FIELD_WALD, 1.0)
    rng = np.random.default_rng(13)
    n = 8000
    pos = dict(i1=rng.integers(3, cfg["n_r"] - 2, n).astype(np.int32),
               i2=rng.integers(2, cfg["n_theta"] - 2, n).astype(np.int32),
               dx1=rng.random(n), dx2=rng.random(n))
    uh = rng.standard_normal((3, n))
    osim.add_species(pos, uh * umag / np.linalg.norm(uh, axis=0), 0.1 * np.ones(n), qm, 0.2)
    g = gpu_from_oracle(osim, iter_tol=1e-16)
    osim.predict()
    g.predict()
    # the lengths' weights at x^n: 1/f, 1/dtheta, 1/sin(theta) over r
    sp = osim.species[0].view()
    dxi = np.log(cfg["r_max"] / cfg["r_min"]) / cfg["n_r"]
    r = cfg["r_min"] * np.exp((sp["i1"] + sp["dx1"]) * dxi)
    th = (sp["i2"] + sp["dx2"]) * np.pi / cfg["n_theta"]
    wt = np.stack([1.0 / (r * dxi), cfg["n_theta"] / (np.pi * r), 1.0 / (r * np.sin(th))])
    osim.push(0)
    g.push(0)
    pg, po = g.get_particles(0), osim.species[0].view()
    ug, uo = (np.stack([p[k] for k in ("u1", "u2", "u3")]) for p in (pg, po))
    err = np.linalg.norm(wt * (ug - uo), axis=0) / np.linalg.norm(wt * uo, axis=0)
    rms = float(np.sqrt(np.mean(err ** 2)))
    print("u %g qm %g: rms %.2e max %.2e" % (umag, qm, rms, err.max()))
    assert rms <= 1.5e-15
