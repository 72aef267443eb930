"""GPU: the FP64 CFL reduction's upper bounds in supersonic and hypersonic flow,
where the internal energy is a small part of the total one: the time step is
the oracle's to the rounding of one node's radii.  FP64 forms the pressure as a
difference, so its relative rounding grows with the ratio of the energies:
1e-14 times (1 + kinetic / internal energy)."""
import numpy as np
import pytest

import oracle as O
from paper_2404_12703_gb300 import workloads as W

from gpu_util import gpu_or_skip, mesh, oracle_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ma", [1.5, 3.0, 10.0, 100.0, 3000.0])
@pytest.mark.parametrize("kw", [dict(viscous=0), dict(mu=0.0), dict(mu=0.01, sutherland=1, T_ref=0.7)])
def test_time_step_at_high_mach_numbers(Ma, kw):
    torch, dg = gpu_or_skip()
    N = 4
    m = mesh(N, (16, 12, 10))
    X = m["xyz"].reshape(m["E"], -1, 3)
    r = 1.0 + 0.3 * np.sin(X[..., 0])
    u = 1.0 + 0.2 * np.sin(X[..., 1])
    p = (1.0 + 0.5 * np.sin(X[..., 2])) / (1.4 * Ma ** 2)
    U = W.prim_to_cons(r, u, 0.1 * u, 0.3 * u, p)
    s = dg.Solver(m, **kw)
    s.set_state(U)
    ref, bad = O.Mesh(N, m["xyz"], m["period"]).dt(U, oracle_params(s.params))
    assert not bad
    ratio = 0.5 * (1.4 * 0.4 * 1.1 * 1.44 * Ma ** 2) / 0.5
    assert abs(s.time_step() - ref) <= 1e-14 * (1.0 + ratio) * ref
