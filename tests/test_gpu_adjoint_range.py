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


def test_gradient_error():
    """Gradients by u_1 and by the amplitude over 30 steps on 200^2, whose Jacobian entries are not
    small beside a 1: the two forms' difference, rms over the orbits relative to the gradients'
    rms. Against 80-bit arithmetic the general form is off by 1.5e-15 and 1.1e-15 (rounding along
    30 steps of a few hundred operations), entries in pairs of FP32 numbers by 2.7e-15 and
    3.4e-15; the bounds lie between the general form's alone and the two together."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import oracle as O
    from paper_2511_17701_gb300 import FIELD_WALD, Sim
    cfg = W.grid_config("wald64", n_r=200, n_theta=200, r_max=50.0, r_absorb=1e300)
    rng = np.random.default_rng(14)
    n = 2000
    x = 200 * (0.35 + 0.3 * rng.random((2, n)))
    i = np.floor(x).astype(np.int32)
    uh = rng.standard_normal((3, n))
    uh *= 0.5 * rng.random(n) / np.linalg.norm(uh, axis=0)
    osim = O.OracleSim(cfg)
    osim.init_fields(O.FIELD_WALD, 1.0)
    osim.add_species(dict(i1=i[0], i2=i[1], dx1=x[0] - i[0], dx2=x[1] - i[1]), uh, np.ones(n), 1.0, 1.0)
    sp = osim.species[0].view()
    st = np.stack([x[0], x[1], np.zeros(n), sp["u1"], sp["u2"], sp["u3"]])
    g = Sim(cfg, [1])
    g.init_metric()
    g.init_fields(FIELD_WALD, 1.0)
    res = []
    for n_iter in (64, 15):
        s = torch.tensor(st, device="cuda")
        v = torch.tensor(np.random.default_rng(15).standard_normal((6, n)), device="cuda")
        _, ck = g.adjoint_forward(s, 1.0, 1.0, 30, 10, n_iter)
        gin, gpp, _ = g.adjoint_backward(ck, v, 1.0, 1.0, 30, 10, n_iter)
        res.append((gin[3].cpu().numpy(), gpp.cpu().numpy()))
    for a, b, bound in zip(res[0], res[1], (2.3e-15, 2.0e-15)):
        rms = np.sqrt(np.mean((a - b) ** 2) / np.mean(b ** 2))
        print("%.2e" % rms)
        assert rms <= bound
