"""GPU: the FP64 surface flux of a viscous run takes 1 / rho and the pressure of
both sides from the lifting's surface kernel through the flux array; an inviscid
run forms them itself.  The right-hand side is within the parity bound of the
oracle and the same bit for bit whatever the array held before (another state's
flux, an autotuner run)."""
import numpy as np
import pytest

import oracle as O
from paper_2404_12703_gb300 import workloads as W

from gpu_util import gpu_or_skip, mesh, oracle_params, parity_bound, parity_check, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 4, 7])
@pytest.mark.parametrize("nodes", ["lgl", "gauss"])
@pytest.mark.parametrize("viscous", [0, 1])
def test_right_hand_side_does_not_depend_on_the_flux_array(N, nodes, viscous):
    torch, dg = gpu_or_skip()
    m = mesh(N, (4, 3, 5))
    gauss = nodes == "gauss"
    s = dg.Solver(m, nodes=nodes, mu=0.01, viscous=viscous, R=2.5)
    x = s.node_coords()
    U = [W.random_perturbation(W.tgv_state(x, Ma=Ma).reshape(m["E"], -1, 5), 1e-2, 5) for Ma in (0.3, 0.7)]
    d = [torch.from_numpy(u).cuda() for u in U]
    first = s.rhs(d[0]).cpu().numpy()
    prm = oracle_params(s.params)
    ref = O.Mesh(N, m["xyz"], m["period"], quad=True, gauss=gauss).rhs(U[0], prm)
    o64 = O.Mesh(N, m["xyz"], m["period"], gauss=gauss).rhs(U[0], prm)
    parity_check(rel_err(first, ref), *parity_bound(o64, ref))
    s.rhs(d[1])
    np.testing.assert_array_equal(s.rhs(d[0]).cpu().numpy(), first)
    s.set_state(U[1])
    if not gauss:
        s.autotune()
        s.set_config(vol_pairs=1)
    s.step(1, sync=True)
    np.testing.assert_array_equal(s.rhs(d[0]).cpu().numpy(), first)
