"""The current filter's two tile sizes: 64 x 32 on grids with enough of them for every SM, 16 x 8
below, ragged on both sides of the line, against the oracle (assert_currents' bound)."""
import pytest

import workloads as W
from parity import assert_currents, gpu_from_oracle, oracle_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_r,n_th,n_f", [(90, 37, 1), (130, 65, 8), (530, 300, 2), (600, 517, 9)])
def test_filter_tiles(n_r, n_th, n_f):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfg = W.grid_config("wald64", n_r=n_r, n_theta=n_th, ppc=1, n_filter=n_f,
                        r_min=0.6 * W.horizon_radius(0.9))
    osim = oracle_state(cfg)
    osim.predict()
    for s in range(2):
        osim.push(s)
    g = gpu_from_oracle(osim)
    g.deposit()
    osim.deposit()
    osim.filter_currents()
    assert_currents(g.planes(), osim.F)
