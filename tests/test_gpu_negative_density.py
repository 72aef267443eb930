"""GPU: a negative density on both sides of a face has no Roe average, even
where the energy is negative as well and the enthalpy so is not: the FP64
surface flux is not a number there, as the oracle's (and that of a side with
one such state), so that a step reports it."""
import numpy as np
import pytest

import oracle as O
from paper_2404_12703_gb300 import workloads as W

from gpu_util import gpu_or_skip, mesh, oracle_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(viscous=0), dict(mu=0.01)])
def test_roe_flux_of_negative_densities(kw):
    torch, dg = gpu_or_skip()
    N = 3
    m = mesh(N, (3, 3, 3))
    U = W.tgv_state(m["xyz"], Ma=0.5).reshape(m["E"], -1, 5)
    s = dg.Solver(m, **kw)
    nbr = s.debug("maps")[0]
    e, f = 13, int(nbr[13, 1, 0])
    for x in (e, f):
        U[x, :, 0] *= -1.0
        U[x, :, 4] *= -1.0
    R = s.rhs(torch.from_numpy(U).cuda())
    torch.cuda.synchronize()
    fs = s.debug("fstar")
    ofs = O.Mesh(N, m["xyz"], m["period"]).rhs(U, oracle_params(s.params), with_fstar=True)[1]
    nan, onan = np.isnan(fs).any(axis=-1), np.isnan(ofs).any(axis=-1)
    assert onan.any()
    np.testing.assert_array_equal(nan, onan)
    assert np.isnan(R.cpu().numpy()[[e, f]]).any(axis=(1, 2)).all()
