"""GPU: the FP64 element kernels' fixed-point arithmetic (dg_fixed64.cuh) at
the places where it can go wrong: the scales of an element's groups, groups
outside the fixed-point range, non-finite values, groups that are all zero.

Bounds.  Scaling density by 2^a (a even), velocity by 2^b and the viscosity by
2^(a + b) multiplies every FP64 operation's result by a power of two, so the
right-hand side scales bit for bit by 2^(a + b) (mass), 2^(a + 2 b) (momentum)
and 2^(a + 3 b) (energy) while no group leaves the range.  Outside it the FP64
loops run: within the parity bound of the long-double oracle (scaled)."""
import numpy as np
import pytest

import oracle as O
from paper_2404_12703_gb300 import workloads as W

from gpu_util import gpu_or_skip, mesh, oracle_params, parity_bound, parity_check, rel_err

pytestmark = pytest.mark.gpu


def _state(m, seed=5):
    return W.random_perturbation(W.tgv_state(m["xyz"], Ma=0.4).reshape(m["E"], -1, 5), 1e-2, seed)


def _scales(a, b):
    return 2.0 ** np.array([a, a + b, a + b, a + b, a + 2 * b]), 2.0 ** np.array(
        [a + b, a + 2 * b, a + 2 * b, a + 2 * b, a + 3 * b])


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7])
@pytest.mark.parametrize("a,b,exact", [(80, -16, True), (-80, 16, True), (300, 0, False), (-320, 20, False)])
def test_power_of_two_units(N, a, b, exact):
    torch, dg = gpu_or_skip()
    m = mesh(N, (3, 4, 3))
    mu = 0.01
    U = _state(m)
    su, sr = _scales(a, b)
    R1 = dg.Solver(m, mu=mu).rhs(torch.from_numpy(U).cuda()).cpu().numpy()
    s = dg.Solver(m, mu=mu * 2.0 ** (a + b))
    R2 = s.rhs(torch.from_numpy(U * su).cuda()).cpu().numpy() / sr
    if exact:
        np.testing.assert_array_equal(R1, R2)
        return
    prm = O.params(mu=mu)
    ref = O.Mesh(N, m["xyz"], m["period"], quad=True).rhs(U, prm)
    o64 = O.Mesh(N, m["xyz"], m["period"]).rhs(U, prm)
    bound, floor = parity_bound(o64, ref)
    parity_check(rel_err(R2, ref), bound, floor)


@pytest.mark.parametrize("N", [2, 5, 7])
def test_non_finite_node_stays_on_its_lines(N):
    """A NaN at one inner node of an inviscid run reaches the nodes of its
    element's three lines through it and of faces beside them only; other
    elements away from it are untouched bit for bit, and the element's other
    nodes hold FP64 values of the same sums."""
    torch, dg = gpu_or_skip()
    n = N + 1
    m = mesh(N, (4, 4, 4))
    U = _state(m)
    s = dg.Solver(m, viscous=0)
    R1 = s.rhs(torch.from_numpy(U).cuda()).cpu().numpy()
    e, i, j, k = 17, 1, 1, 1
    Ub = U.copy()
    Ub[e, i + n * (j + n * k), 4] = np.nan
    R2 = s.rhs(torch.from_numpy(Ub).cuda()).cpu().numpy()
    on = np.zeros((n, n, n), bool)  # [k, j, i]
    on[k, j, :] = on[k, :, i] = on[:, j, i] = True
    on = on.reshape(-1)
    assert np.isnan(R2[e][on]).any(axis=1).all()
    assert np.isfinite(R2[e][~on]).all()
    # the same sums in FP64: each sums 3 (N + 1) terms of at most the element's largest
    scale = np.abs(R1).max(axis=(0, 1))
    assert (np.abs(R2[e][~on] - R1[e][~on]) <= 1e-11 * scale).all()
    far = np.arange(m["E"]) != e
    np.testing.assert_array_equal(R1[far], R2[far])


@pytest.mark.parametrize("N", [1, 4, 7])
def test_groups_that_are_zero_or_span_many_magnitudes(N):
    """Fluid at rest (an all-zero velocity group), and a density ratio of 1e6
    inside elements: within the parity bound."""
    torch, dg = gpu_or_skip()
    m = mesh(N, (3, 3, 4), seed=3)
    X = m["xyz"].reshape(m["E"], -1, 3)
    z = np.zeros(X.shape[:2])
    rho = 10.0 ** (3.0 * np.sin(X[..., 0]) * np.cos(X[..., 1]))
    for u, r in ((z, 1.0 + 0.1 * np.sin(X[..., 2])), (np.sin(X[..., 1]), rho)):
        U = W.prim_to_cons(r, u, z, z, 1.0 + z)
        s = dg.Solver(m, mu=0.01)
        R = s.rhs(torch.from_numpy(U).cuda()).cpu().numpy()
        prm = oracle_params(s.params)
        ref = O.Mesh(N, m["xyz"], m["period"], quad=True).rhs(U, prm)
        o64 = O.Mesh(N, m["xyz"], m["period"]).rhs(U, prm)
        bound, floor = parity_bound(o64, ref)
        parity_check(rel_err(R, ref), bound, floor)
