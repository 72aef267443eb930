"""GPU: the fixed-point volume kernel's scales where the three directions of an
element, and the elements that share a warp at N = 1, differ most: an aligned
box stretched differently in every direction (two of three metric components
zero per direction), with density and pressure growing by 10^4 across the
mesh.  Within the parity bound of the long-double oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2404_12703_gb300 import workloads as W

from gpu_util import gpu_or_skip, oracle_params, parity_bound, parity_check, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7])
@pytest.mark.parametrize("viscous", [0, 1])
def test_scales_that_differ_by_direction_and_element(N, viscous):
    torch, dg = gpu_or_skip()
    L = (2 * np.pi, 0.3, 40.0)
    m = W.box_mesh(N, (6, 5, 4), length=L, curved=0.0)
    X = m["xyz"].reshape(m["E"], -1, 3) * (2 * np.pi / np.array(L))
    r = 10.0 ** (2 * np.sin(X[..., 0]))
    z = np.zeros(X.shape[:2])
    U = W.prim_to_cons(r, np.sin(X[..., 1]), 0.1 * np.cos(X[..., 2]), z, r * (1.0 + 0.1 * np.sin(X[..., 2])))
    s = dg.Solver(m, mu=0.01 * viscous, viscous=viscous)
    R = s.rhs(torch.from_numpy(U).cuda()).cpu().numpy()
    prm = oracle_params(s.params)
    ref = O.Mesh(N, m["xyz"], m["period"], quad=True).rhs(U, prm)
    o64 = O.Mesh(N, m["xyz"], m["period"]).rhs(U, prm)
    bound, floor = parity_bound(o64, ref)
    parity_check(rel_err(R, ref), bound, floor)
