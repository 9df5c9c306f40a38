"""What a particle's FP64 push gives depends on that particle alone: not on the particles beside
it in memory, whose fields may be strong where its own is weak, nor on how a step is cut into
ranges. Bit for bit, at a small iter_tol (the push's increment form)."""
import numpy as np
import pytest

import workloads as W
from oracle import oracle as O
from parity import gpu_from_oracle, oracle_state
from test_gpu_step_host import STATE, as_numpy, host_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("qm", [1.0, 2.25, 2.5, 9.0])
def test_push_in_another_order(torch_cuda, qm):
    """Where the fields turn the momentum by about the form's bound over a half step, some
    particles are below it and some above (qm = 2.25 for a bound of 1/64, 9 for 1/16)."""
    cfg = W.grid_config("wald64")
    osim = O.OracleSim(cfg)
    osim.init_fields(O.FIELD_WALD, 1.0)
    rng = np.random.default_rng(11)
    n = 20011
    pos = dict(i1=rng.integers(3, cfg["n_r"] - 2, n).astype(np.int32),
               i2=rng.integers(0, cfg["n_theta"], n).astype(np.int32),
               dx1=rng.random(n), dx2=rng.random(n))
    osim.add_species(pos, rng.standard_normal((3, n)), 0.1 * np.ones(n), qm, 0.2)
    osim.predict()
    state = osim.species[0].view()
    sim = gpu_from_oracle(osim, iter_tol=1e-12)

    def push(order):
        sim.set_particles(0, {k: np.ascontiguousarray(v[order]) for k, v in state.items()}, qm, 0.2)
        sim.push(0)
        return sim.get_particles(0)

    ref = push(np.arange(n))
    for order in (rng.permutation(n), np.argsort(state["i1"], kind="stable"), np.arange(5, n, 3)):
        got = push(order)
        for k in ("i1", "i2", "dx1", "dx2", "u1", "u2", "u3", "phi", "tag"):
            assert np.array_equal(got[k], ref[k][order]), k


@pytest.mark.parametrize("qm", [1.0, 2.25, 10.0])
def test_step_host_bits(torch_cuda, qm):
    """The streamed step pushes each species in four ranges that no multiple of a warp bounds."""
    osim = oracle_state(W.grid_config("wald64", sort_every=0))
    n_keep = 8191
    a, b = (gpu_from_oracle(osim, iter_tol=1e-12) for _ in range(2))
    for g in (a, b):
        for s in range(2):
            sp = osim.species[s]
            g.set_particles(s, {k: v[-n_keep:] for k, v in sp.view().items()}, sp.qm * qm, sp.qc)
    states, counts = host_state(b)
    a.step(1)
    counts = b.step_host(states, counts)
    for s in range(2):
        pa = a.get_particles(s)
        hb = as_numpy(states[s], counts[s])
        for k in STATE:
            assert np.array_equal(pa[k], hb[k]), (s, k)
