"""GPU: the CFL radii that the two-kernel FP32-bulk stage reduces cover every
node, also those of a block's last, partly filled warp (n^3 nodes per element
is no multiple of 32 at N = 2, 4, 5 and 6): the first step's time step equals
dg_time_step of the state bit for bit, wherever the fastest node sits."""
import numpy as np
import pytest

from paper_2404_12703_gb300 import workloads as W

from gpu_util import gpu_or_skip, mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7])
@pytest.mark.parametrize("where", ["first", "last"])
def test_radii_cover_every_node(N, where):
    torch, dg = gpu_or_skip()
    m = mesh(N, (3, 3, 3))
    U = W.tgv_state(m["xyz"], Ma=0.5).reshape(m["E"], -1, 5)
    e, v = (0, 0) if where == "first" else (m["E"] - 1, U.shape[1] - 1)
    U[e, v, 1] += 4.0 * U[e, v, 0]  # one fast node
    U[e, v, 4] += 20.0 * U[e, v, 0]
    s = dg.Solver(m, precision=dg.FP32_BULK, mu=1e-6)
    assert s.stage_form() == 2
    s.set_state(U)
    dt = s.time_step()
    assert s.step(1, sync=True) == dt
    assert np.isfinite(dt) and dt > 0
