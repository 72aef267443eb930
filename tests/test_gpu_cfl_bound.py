"""GPU: the FP64 CFL reduction evaluates a node only if its FP32 upper bound
exceeds the largest radius so far.  The time step equals the oracle's to the
rounding of one node's radii (a few FP64 operations: 1e-14) wherever the node
that sets it sits and whatever the units, and a node without a sound speed is
reported wherever it sits."""
import numpy as np
import pytest

import oracle as O
from paper_2404_12703_gb300 import workloads as W

from gpu_util import gpu_or_skip, mesh, oracle_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,nel", [(1, (3, 3, 3)), (4, (16, 12, 10)), (7, (9, 8, 7))])
@pytest.mark.parametrize("kw", [dict(viscous=0), dict(mu=0.5, dfl=0.1), dict(mu=0.01, sutherland=1, T_ref=0.7)])
@pytest.mark.parametrize("scale", [0, 120, -120, -500])
def test_time_step(N, nel, kw, scale):
    torch, dg = gpu_or_skip()
    m = mesh(N, nel)
    U0 = W.random_perturbation(W.tgv_state(m["xyz"], Ma=0.8).reshape(m["E"], -1, 5), 1e-3, 7)
    rng = np.random.Generator(np.random.PCG64(N))
    s = dg.Solver(m, **{**kw, "mu": kw.get("mu", 0.0) * 2.0 ** scale} if kw.get("viscous", 1) else kw)
    om = O.Mesh(N, m["xyz"], m["period"])
    for k in range(3):
        U = U0.copy()
        e, v = int(rng.integers(m["E"])), int(rng.integers(U.shape[1]))
        U[e, v, 1:4] *= 1.0 + k  # from a smooth state to one fast node
        U[e, v, 4] *= 1.0 + k * k
        s.set_state(U * 2.0 ** scale)
        prm = oracle_params(s.params)
        ref, bad = om.dt(U * 2.0 ** scale, prm)
        assert not bad
        assert abs(s.time_step() - ref) <= 1e-14 * ref


@pytest.mark.parametrize("what", ["nan", "inf", "pressure", "density"])
@pytest.mark.parametrize("where", [0, 1, -1])
def test_nodes_without_a_sound_speed_are_reported(what, where):
    torch, dg = gpu_or_skip()
    m = mesh(3, (16, 16, 16))
    U = W.tgv_state(m["xyz"], Ma=0.5).reshape(m["E"], -1, 5)
    e = {0: 0, 1: m["E"] // 2, -1: m["E"] - 1}[where]
    if what == "pressure":
        U[e, where, 4] = 0.5 * (U[e, where, 1:4] ** 2).sum() / U[e, where, 0] * (1 - 1e-9)
    elif what == "density":
        U[e, where, 0] *= -1.0
    else:
        U[e, where, 4] = np.nan if what == "nan" else np.inf
    s = dg.Solver(m, mu=0.01)
    s.set_state(U)
    with pytest.raises(dg.DgError) as err:
        s.step(1, sync=True)
    assert err.value.code == dg.DG_ERR_NONFINITE
