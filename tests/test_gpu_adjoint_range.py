"""The adjoint with field planes, amplitudes and charges far from 1, where FP32's range ends,
against the general FP64 form, which takes iteration limits below 16. Tolerances as in
test_gpu_adjoint_inc.py; the gradient by the amplitude relative to its own median."""
import numpy as np
import pytest

import workloads as W
from test_gpu_adjoint_inc import STEPS, states

pytestmark = pytest.mark.gpu


def make(B0):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_17701_gb300 import FIELD_WALD, Sim
    g = Sim(W.grid_config("wald64", r_absorb=1e300), [1])
    g.init_metric()
    g.init_fields(FIELD_WALD, B0)
    return g


def both(g, st, v, qm, b0):
    torch = g.torch
    st, v = torch.tensor(st, device="cuda"), torch.tensor(v, device="cuda")
    res = []
    for n_iter in (64, 15):
        out, ck = g.adjoint_forward(st, qm, b0, STEPS, 4, n_iter)
        gin, gpp, _ = g.adjoint_backward(ck, v, qm, b0, STEPS, 4, n_iter)
        res.append([x.cpu().numpy() for x in (out, gin, gpp)])
    return res


@pytest.mark.parametrize("B0,qm,b0", [(1e-25, 1e25, 1e-25), (1e-30, 1.0, 1.0), (1e30, 1.0, 1.0),
                                      (1.0, 1e-30, 1e30), (1e-12, 1e-13, 1e25), (1e-35, 1.0, 1e-35)])
def test_units(B0, qm, b0):
    g = make(B0)
    n = 400
    (o1, g1, p1), (o2, g2, p2) = both(g, states(n, 9), np.random.default_rng(10).standard_normal((6, n)),
                                      qm, b0)
    assert np.array_equal(np.isnan(o1), np.isnan(o2))
    ok = ~np.isnan(o2[0])
    assert ok.sum() >= 300
    assert np.max(np.abs(o1 - o2)[:, ok] / np.maximum(1.0, np.abs(o2[:, ok]))) <= 1e-12
    scale = np.abs(g2[:, ok]).max(axis=0)
    assert np.max(np.abs(g1 - g2)[:, ok] / scale) <= 1e-10
    assert np.max(np.abs(p1 - p2)[ok] / (np.abs(p2[ok]) + np.median(np.abs(p2[ok])))) <= 1e-10
