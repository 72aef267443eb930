"""GPU: the fixed-point element kernels on Gauss-Legendre nodes
(dg_fixed64_gl.cuh): the scales of volume and surface sums, groups outside the
fixed-point range and non-finite values.  Bounds as in test_gpu_fixed64.py:
power-of-two units scale the right-hand side bit for bit, the FP64 sums
outside the range are within the parity bound."""
import numpy as np
import pytest

import oracle as O
from paper_2404_12703_gb300 import workloads as W

from gpu_util import gpu_or_skip, mesh, parity_bound, parity_check, rel_err

pytestmark = pytest.mark.gpu


def _state(dg, m, **kw):
    s = dg.Solver(m, nodes="gauss", **kw)
    return s, W.random_perturbation(W.tgv_state(s.node_coords(), Ma=0.4).reshape(m["E"], -1, 5), 1e-2, 5)


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7])
@pytest.mark.parametrize("a,b,exact", [(80, -16, True), (-80, 16, True), (300, 0, False)])
def test_power_of_two_units(N, a, b, exact):
    torch, dg = gpu_or_skip()
    m = mesh(N, (3, 4, 3))
    mu = 0.01
    su = 2.0 ** np.array([a, a + b, a + b, a + b, a + 2 * b])
    sr = 2.0 ** np.array([a + b, a + 2 * b, a + 2 * b, a + 2 * b, a + 3 * b])
    s, U = _state(dg, m, mu=mu)
    R1 = s.rhs(torch.from_numpy(U).cuda()).cpu().numpy()
    s2 = dg.Solver(m, nodes="gauss", mu=mu * 2.0 ** (a + b))
    R2 = s2.rhs(torch.from_numpy(U * su).cuda()).cpu().numpy() / sr
    if exact:
        np.testing.assert_array_equal(R1, R2)
        return
    prm = O.params(mu=mu)
    ref = O.Mesh(N, m["xyz"], m["period"], quad=True, gauss=True).rhs(U, prm)
    o64 = O.Mesh(N, m["xyz"], m["period"], gauss=True).rhs(U, prm)
    bound, floor = parity_bound(o64, ref)
    parity_check(rel_err(R2, ref), bound, floor)


@pytest.mark.parametrize("N", [2, 7])
def test_non_finite_node(N):
    """A NaN at one node of an inviscid run reaches its element and the face
    neighbours only; the other elements are untouched bit for bit."""
    torch, dg = gpu_or_skip()
    m = mesh(N, (4, 4, 4))
    s, U = _state(dg, m, viscous=0)
    R1 = s.rhs(torch.from_numpy(U).cuda()).cpu().numpy()
    e = 17
    Ub = U.copy()
    Ub[e, 1, 4] = np.nan
    R2 = s.rhs(torch.from_numpy(Ub).cuda()).cpu().numpy()
    near = np.concatenate([[e], s.debug("maps")[0][e, :, 0]])
    assert np.isnan(R2[e]).any()
    far = ~np.isin(np.arange(m["E"]), near)
    np.testing.assert_array_equal(R1[far], R2[far])
