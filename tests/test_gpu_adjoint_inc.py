"""The adjoint's increment form against its general FP64 form, which takes iteration limits
below 16 (both converge here well before 15 iterations): states and gradients of the same
orbits, over rows next to the axes, at rest and fast, weak and strong fields (the strongest
past what the increment form takes, so its steps mix both forms in one segment).
Tolerances: states 1e-12; gradients 1e-10 of a particle's largest entry (8 steps of a few
hundred operations at ~1e-16, condition numbers up to ~1e2). Cotangents scaled by a power of
two scale the gradients exactly, far outside FP32's range too."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

STEPS = 8


@pytest.fixture(scope="module")
def sim():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_17701_gb300 import FIELD_WALD, Sim
    g = Sim(W.grid_config("wald64", r_absorb=1e300), [1])
    g.init_metric()
    g.init_fields(FIELD_WALD, 1.0)
    return g


def states(n, seed):
    rng = np.random.default_rng(seed)
    s = np.zeros((6, n))
    s[0] = rng.uniform(12.0, 56.0, n)
    s[1] = np.where(np.arange(n) % 8 == 0, rng.uniform(1.2, 3.5, n), rng.uniform(3.0, 61.0, n))
    s[3:] = rng.standard_normal((3, n)) * 10.0 ** rng.uniform(-2.0, 0.3, n)
    s[3] *= 0.05
    s[4] *= 0.1
    s[3:, 1] = 0.0
    return s


@pytest.mark.parametrize("qm", [0.0, 1.0, -8.0, 300.0])
@pytest.mark.parametrize("every", [3, 8])
def test_against_general_form(sim, qm, every):
    torch = sim.torch
    st = torch.tensor(states(500, 5), device="cuda")
    v = np.random.default_rng(6).standard_normal((6, 500))
    res = []
    for n_iter in (64, 15):
        out, ck = sim.adjoint_forward(st, qm, 1.0, STEPS, every, n_iter)
        gin, gpp, gsum = sim.adjoint_backward(ck, torch.tensor(v, device="cuda"), qm, 1.0, STEPS,
                                              every, n_iter)
        res.append([x.cpu().numpy() for x in (out, gin, gpp)])
    (o1, g1, p1), (o2, g2, p2) = res
    assert np.array_equal(np.isnan(o1), np.isnan(o2))
    ok = ~np.isnan(o2[0])
    assert ok.sum() >= 400
    assert np.max(np.abs(o1 - o2)[:, ok] / np.maximum(1.0, np.abs(o2[:, ok]))) <= 1e-12
    scale = np.abs(g2[:, ok]).max(axis=0)
    assert np.max(np.abs(g1 - g2)[:, ok] / scale) <= 1e-10
    assert np.max(np.abs(p1 - p2)[ok] / (np.abs(p2[ok]) + scale)) <= 1e-10


def test_cotangent_scale_is_exact(sim):
    torch = sim.torch
    st = torch.tensor(states(300, 7), device="cuda")
    v = torch.tensor(np.random.default_rng(8).standard_normal((6, 300)), device="cuda")
    out, ck = sim.adjoint_forward(st, 1.0, 1.0, STEPS, 4, 64)
    ok = ~torch.isnan(out[0])
    ref = sim.adjoint_backward(ck, v, 1.0, 1.0, STEPS, 4, 64)
    for k in (600, -600):
        got = sim.adjoint_backward(ck, v * 2.0 ** k, 1.0, 1.0, STEPS, 4, 64)
        assert torch.equal(got[0][:, ok], ref[0][:, ok] * 2.0 ** k)
        assert torch.equal(got[1][ok], ref[1][ok] * 2.0 ** k)
