"""GPU: precision of the fixed-point element kernels where an element's values
span many magnitudes: each node's error against the values on that node's own
lines, not against the largest of the mesh.

Bounds.  A node's volume sums in FP64 have 3 (N + 1) terms of at most 8
rounded factors each, times derivative weights whose absolute row sums stay
below 2 n^2 (n = N + 1): the error is at most (n + 12) 2^-53 times the sum over
the directions of 2 n^2 max |flux . metrics| over the node's line, over J.  The
same again for what both sides share (pressure from the state, metrics), and
once more for the surface terms of Gauss nodes.  Fixed point with one scale
per element would be off by 2^-60 of the element's largest value instead:
hundreds of times these bounds."""
import numpy as np
import pytest

import oracle as O
from paper_2404_12703_gb300 import workloads as W

from gpu_util import gpu_or_skip, mesh, oracle_params

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


def _lines_max(A, n):
    """A[e, node] -> per direction the largest on the node's line, [3, E, node]."""
    B = A.reshape(A.shape[0], n, n, n)  # [e, k, j, i]
    return np.stack([np.broadcast_to(B.max(axis=ax, keepdims=True), B.shape).reshape(A.shape) for ax in (3, 2, 1)])


def _local(s, U, n):
    """The bound's magnitude per node and variable: sum over the directions of the line's largest flux, over J."""
    Ja, J = s.debug("metrics")  # [e, node, direction, component]
    rho, m, E = U[..., 0], U[..., 1:4], U[..., 4]
    u = m / rho[..., None]
    p = (s.params.gamma - 1) * (E - 0.5 * (m * u).sum(-1))
    out = np.zeros(U.shape)
    for d in range(3):
        c = np.abs(Ja[:, :, d])
        fr = rho * (np.abs(u) * c).sum(-1)
        f = np.stack([fr, *(fr * np.abs(u[..., i]) + np.abs(p) * c[..., i] for i in range(3)), fr * (np.abs(E) + np.abs(p)) / rho], -1)
        for k in range(5):
            out[..., k] += _lines_max(f[..., k], n)[d]
    return out / np.abs(J)[..., None]


def _solver(dg, m, nodes, **kw):
    return dg.Solver(m, **({"nodes": "gauss"} if nodes == "gauss" else {}), **kw)


def _inner(n, nodes):
    if nodes == "gauss":
        return np.ones(n ** 3, bool)
    i = np.zeros((n, n, n), bool)
    i[1:-1, 1:-1, 1:-1] = True
    return i.reshape(-1)


# (on Gauss nodes the interpolation of a spike of 1e10 to the faces undershoots
# zero pressure)
@pytest.mark.parametrize("nodes,ratio", [("lgl", 1e6), ("lgl", 1e10), ("gauss", 1e6)])
@pytest.mark.parametrize("N", [2, 3, 5, 7])
def test_pressure_spike_at_a_corner(N, nodes, ratio):
    """A pressure spike at an element corner of a slowly moving gas: nodes whose
    three lines miss the spike keep the precision of their own values."""
    torch, dg = gpu_or_skip()
    n = N + 1
    m = mesh(N, (4, 4, 4), seed=11)
    s = _solver(dg, m, nodes, viscous=0, riemann="lf")
    X = s.node_coords().reshape(m["E"], -1, 3)
    h = 2 * np.pi / 4
    r2 = ((X - m["xyz"].reshape(m["E"], -1, 3)[21, 0]) ** 2).sum(-1)
    p = 1.0 + ratio * np.exp(-np.log(ratio * 1e2) * r2 / (0.5 * h) ** 2)
    one = np.ones(p.shape)
    U = W.prim_to_cons(1.0 + 0.1 * np.sin(X[..., 2]), 0.2 + 0.1 * np.sin(X[..., 1]), -0.1 * one, 0.3 * one, p)
    R = s.rhs(torch.from_numpy(U).cuda()).cpu().numpy()
    ref = O.Mesh(N, m["xyz"], m["period"], quad=True, gauss=nodes == "gauss").rhs(U, oracle_params(s.params))
    local = _local(s, U, n)
    inner = _inner(n, nodes)
    quiet = inner[None, :] & (_lines_max(p, n).max(axis=0) < 1e-5 * ratio)
    near = _lines_max(p, n).max(axis=(0, 2)) > 1e-2 * ratio  # elements that hold the spike
    assert (quiet & near[:, None]).sum() >= 3
    bound = (4 if nodes == "gauss" else 2) * 2 * n * n * (n + 12) * EPS * local
    at = quiet & near[:, None]
    err = np.abs(R - ref)
    assert np.all(err[at] <= bound[at]), (err[at] / bound[at]).max(axis=0)


@pytest.mark.parametrize("nodes", ["lgl", "gauss"])
@pytest.mark.parametrize("N", [2, 5, 7])
def test_gradient_of_a_small_cross_flow(N, nodes):
    """u = O(1), v = O(1e-8): the lifted gradient of v has v's precision."""
    torch, dg = gpu_or_skip()
    n = N + 1
    m = mesh(N, (3, 3, 4), seed=12)
    s = _solver(dg, m, nodes, mu=0.01)
    X = s.node_coords().reshape(m["E"], -1, 3)
    one = np.ones(X.shape[:2])
    U = W.prim_to_cons(one, 1.0 + 0.3 * np.sin(X[..., 1]), 1e-8 * (1.0 + 0.5 * np.sin(X[..., 0])), 0.1 * np.cos(X[..., 2]), 10.0 * one)
    s.rhs(torch.from_numpy(U).cuda())
    torch.cuda.synchronize()
    g = s.debug("grad")
    _, og = O.Mesh(N, m["xyz"], m["period"], quad=True, gauss=nodes == "gauss").rhs(U, oracle_params(s.params), with_grad=True)
    Ja, J = s.debug("metrics")
    v = np.abs(U[..., 2] / U[..., 0])
    inner = _inner(n, nodes)
    for c in range(3):
        local = sum(_lines_max(v * np.abs(Ja[:, :, d, c]), n)[d] for d in range(3)) / np.abs(J)
        bound = (4 if nodes == "gauss" else 2) * 2 * n * n * (n + 12) * EPS * local
        err = np.abs(g[:, :, 1, c] - og[:, :, 1, c])
        assert np.all(err[:, inner] <= bound[:, inner]), (err / bound).max()


@pytest.mark.parametrize("N", [2, 5, 7])
def test_cross_flow_of_a_stretched_mesh(N):
    """A mesh 1e4 times finer in y than in x, with u = O(1) and v = O(1e-4):
    the fluxes along both directions are alike, although the metrics and the
    velocities are not.  (On LGL nodes, whose inner nodes have no surface flux:
    its upwind terms are of the size of the sound speed in y.)"""
    torch, dg = gpu_or_skip()
    n = N + 1
    L = np.array([2 * np.pi, 2 * np.pi * 1e-4, 2 * np.pi])
    m = W.box_mesh(N, (3, 4, 3), length=tuple(L), curved=0.0)
    s = dg.Solver(m, viscous=0)
    X = m["xyz"].reshape(m["E"], -1, 3) * (2 * np.pi / L)
    one = np.ones(X.shape[:2])
    U = W.prim_to_cons(1.0 + 0.1 * np.sin(X[..., 0]), 1.0 + 0.3 * np.sin(X[..., 1]), 1e-4 * (1.0 + 0.5 * np.sin(X[..., 0])),
                       0.1 * np.cos(X[..., 2]), 10.0 * one)
    R = s.rhs(torch.from_numpy(U).cuda()).cpu().numpy()
    ref = O.Mesh(N, m["xyz"], m["period"], quad=True).rhs(U, oracle_params(s.params))
    bound = 4 * n * n * (n + 12) * EPS * _local(s, U, n)
    inner = _inner(n, "lgl")
    err = np.abs(R - ref)
    assert np.all(err[:, inner] <= bound[:, inner]), (err / bound)[:, inner].max(axis=(0, 1))
