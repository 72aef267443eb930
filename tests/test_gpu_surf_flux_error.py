"""GPU: rounding error of the FP64 surface flux at low Mach number, where the
pressure is a hundred times the convective momentum flux.

Bound.  The textbook form F = (F_L + F_R - D) / 2, each side's flux formed by
itself, rounds the momentum at the pressure's size some four times (p n of each
side, their sum, the upwind term); the kernel, which adds the pressures last,
rounds it twice.  Its rms error over the faces is therefore no larger than the
FP64 oracle's (the textbook form); 10 % for the sample.  A form that adds the
pressures first and the upwind and viscous terms to their sum is off by 1.3."""
import numpy as np
import pytest

import oracle as O
from paper_2404_12703_gb300 import workloads as W

from gpu_util import gpu_or_skip, mesh, oracle_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 4])
@pytest.mark.parametrize("kw", [dict(mu=0.01), dict(viscous=0), dict(viscous=0, riemann="lf")])
def test_momentum_flux_error_against_the_textbook_form(N, kw):
    torch, dg = gpu_or_skip()
    err = np.zeros(3)
    floor = np.zeros(3)
    for seed in range(6 if N == 1 else 2):
        m = mesh(N, (4, 4, 3), seed=30 + seed)
        X = m["xyz"] + np.random.default_rng(seed).uniform(0, 6, 3)
        U = W.random_perturbation(W.tgv_state(X, Ma=0.1).reshape(m["E"], -1, 5), 1e-2, seed)
        s = dg.Solver(m, **kw)
        s.rhs(torch.from_numpy(U).cuda())
        torch.cuda.synchronize()
        f = s.debug("fstar")
        prm = oracle_params(s.params)
        q = O.Mesh(N, m["xyz"], m["period"], quad=True).rhs(U, prm, with_fstar=True)[1]
        o = O.Mesh(N, m["xyz"], m["period"]).rhs(U, prm, with_fstar=True)[1]
        err += ((f - q)[..., 1:4] ** 2).reshape(-1, 3).sum(0)
        floor += ((o - q)[..., 1:4] ** 2).reshape(-1, 3).sum(0)
        s.close()
    assert np.all(np.sqrt(err) <= 1.1 * np.sqrt(floor)), np.sqrt(err / floor)
