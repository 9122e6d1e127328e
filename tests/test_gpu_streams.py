"""What a handle's own stream has to order by itself, whatever the caller has on other streams."""
import numpy as np
import pytest

import paper_2303_00689_gb300 as kx
from tests.test_gpu_eigen import lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [kx.SIM_PREC_FP64, kx.SIM_PREC_MIXED])
@pytest.mark.parametrize("n", [40, 300])
def test_a_handle_is_ready_while_the_default_stream_is_busy(n, precision):
    """The error word of the tensor-core products lies in memory that other handles have used."""
    torch = pytest.importorskip("torch")
    h = lattice(n, precision)
    D = kx.sim_get_state(h, n)[3]
    kx.sim_destroy(h)
    for other in (n + 31, 2 * n, n + 7):                # leave nothing in the pool as it was
        kx.sim_destroy(lattice(other, precision))
    torch.cuda._sleep(400_000_000)                      # ~ 0.2 s on the legacy default stream
    h = lattice(n, precision)
    try:
        assert np.array_equal(kx.sim_get_state(h, n)[3], D)
    finally:
        kx.sim_destroy(h)
        torch.cuda.synchronize()
