"""GPU: the launch configuration that is set is the one that is launched.

* The blocks of the element and side kernels as the profiler records them: 2 D
  elements and 128 threads are launched as given on every mesh, the default D
  and 256 are upper limits, and the autotuner times what a step launches.
* Blocks of several elements with a partly filled last one, and elements with
  FP64 sums beside fixed-point ones in a block, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2404_12703_gb300 import workloads as W

from gpu_util import gpu_or_skip, mesh, oracle_params, parity_bound, parity_check, rel_err

pytestmark = pytest.mark.gpu


def _sizes(N):
    n3 = (N + 1) ** 3
    D = 1 if n3 >= 256 else 256 // n3
    return D, 2 * D * n3 <= 1024, 2 * D * n3 <= 512


def _mixed_state(m, c=2.0):
    """A Taylor-Green flow whose density spans 10^c, most of it across some
    elements (whose sums are taken in FP64) and little across the others."""
    X = m["xyz"].reshape(m["E"], -1, 3)
    U = W.tgv_state(X, Ma=0.5).reshape(m["E"], -1, 5)
    r = np.where(X[..., 0] < np.pi, 10.0 ** (c * np.sin(X[..., 0]) * np.sin(X[..., 1]) ** 2 * np.sin(X[..., 2]) ** 2), 1.0)
    q = np.sqrt(r)  # (u / q: the same kinetic energy and pressure)
    return U * np.stack([r, q, q, q, np.ones_like(r)], -1)


def _launched(torch, run):
    """{kernel name: set of (grid x, threads per block)} of the calls in run()."""
    import json
    import os
    import tempfile
    from torch.profiler import ProfilerActivity, profile
    for _ in range(2):  # (the process's first profile may come without records)
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            run()
            torch.cuda.synchronize()
        with tempfile.TemporaryDirectory() as d:
            path = os.path.join(d, "trace.json")
            p.export_chrome_trace(path)
            with open(path) as f:
                events = json.load(f)["traceEvents"]
        out = {}
        for e in events:
            if e.get("cat") == "kernel":
                name = e["name"].split("<")[0].split("::")[-1]
                out.setdefault(name, set()).add((e["args"]["grid"][0], e["args"]["block"][0]))
        if out:
            return out
    pytest.skip("no kernel records (the profiler is not available here)")


@pytest.mark.parametrize("N", [1, 3, 5])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_configured_blocks_are_launched(N, prec):
    torch, dg = gpu_or_skip()
    D, lift2, vol2 = _sizes(N)
    m = mesh(N, (3, 3, 4), seed=41)
    E, n2 = m["E"], (N + 1) ** 2
    s = dg.Solver(m, mu=0.01, precision=dg.FP64 if prec == "fp64" else dg.FP32_BULK)
    s.set_state(W.tgv_state(m["xyz"]).reshape(E, -1, 5))
    dt = 1e-4
    side = "k_surf_flux" if prec == "fp64" else "k_fflux"
    elem = "k_volume_fx" if prec == "fp64" else "k_felem"

    def blocks():
        return _launched(torch, lambda: s.profile_step(1, dt=dt))

    s.set_config()
    small = blocks()
    s.set_config(2 * D if prec == "fp64" and lift2 else 0, 2 * D if vol2 else 0, -1, 128)
    big = blocks()
    sides = 3 * E * n2
    assert {b for _, b in big[side]} == {128} and {g for g, _ in big[side]} == {-(-sides // 128)}
    assert {b for _, b in small[side]} == {32}  # 36 elements leave SMs idle
    if vol2:
        assert {g for g, _ in big[elem]} == {-(-E // (2 * D))}
    if vol2 and lift2 and prec == "fp64":
        assert {g for g, _ in big["k_lift_fx"]} == {-(-E // (2 * D))}
    least = 4 if N == 1 and prec == "fp64" else D if N == 1 or prec == "fp32" and N != 3 else 1
    assert {g for g, _ in small[elem]} == {-(-E // least)}


def test_autotune_times_what_a_step_launches():
    torch, dg = gpu_or_skip()
    m = mesh(3, (3, 3, 4), seed=42)
    for prec in (dg.FP64, dg.FP32_BULK):
        s = dg.Solver(m, mu=0.01, precision=prec)
        s.set_state(W.tgv_state(m["xyz"]).reshape(m["E"], -1, 5))
        elem = "k_volume_fx" if prec == dg.FP64 else "k_felem"
        s.set_config()
        steps = set()
        for ve in (0, 8):
            s.set_config(0, ve, -1, 0)
            steps |= _launched(torch, lambda: s.profile_step(1, dt=1e-4))[elem]
        s.set_config()
        assert _launched(torch, s.autotune)[elem] <= steps


@pytest.mark.parametrize("N,nel", [(1, (3, 4, 5)), (2, (3, 4, 5)), (3, (3, 3, 7)), (4, (3, 3, 7))])
@pytest.mark.parametrize("kw", [dict(mu=0.01), dict(viscous=0, riemann="lf", shock_capturing=1, alpha_force=0.4)])
def test_partial_last_block_of_the_large_form(N, nel, kw):
    """2 D elements per block (8 to 64), which divides neither 60 nor 63."""
    torch, dg = gpu_or_skip()
    D, lift2, vol2 = _sizes(N)
    m = mesh(N, nel)
    assert lift2 and vol2 and m["E"] % (2 * D) != 0
    U = _mixed_state(m)
    s = dg.Solver(m, **kw)
    s.set_config(2 * D, 2 * D, 1, 128)
    s.set_state(U)
    dt = s.time_step()
    s.step(1, dt=dt)
    got = s.get_state()[0]
    prm = oracle_params(s.params)
    ref = O.Mesh(N, m["xyz"], m["period"], quad=True).step(U, prm, 1, dt=dt)[0]
    o64 = O.Mesh(N, m["xyz"], m["period"]).step(U, prm, 1, dt=dt)[0]
    bound, floor = parity_bound(o64, ref)
    parity_check(rel_err(got, ref), bound, floor)
    # the block size changes no arithmetic
    s.set_config()
    s.set_state(U)
    s.step(1, dt=dt)
    np.testing.assert_array_equal(s.get_state()[0], got)


# elements per block 32, 9, 4 and 2 by default on a GPU of up to 152 SMs, the
# last block partly filled
@pytest.mark.parametrize("nodes", ["lgl", "gauss"])
@pytest.mark.parametrize("N,nel", [(1, (22, 22, 21)), (2, (15, 14, 13)), (3, (11, 11, 11)), (4, (9, 9, 9))])
def test_partial_last_block_of_the_default_form(N, nel, nodes):
    torch, dg = gpu_or_skip()
    gauss = nodes == "gauss"
    D = _sizes(N)[0]
    m = mesh(N, nel, seed=43)
    assert m["E"] % D != 0 and -(-m["E"] // D) >= 2 * 152
    s = dg.Solver(m, mu=0.01, **({"nodes": "gauss"} if gauss else {}))
    X = s.node_coords().reshape(m["E"], -1, 3)
    # (interpolated to the faces from two Gauss nodes, more would undershoot zero)
    U = _mixed_state({"xyz": X, "E": m["E"]}, 0.5 if gauss and N == 1 else 2.0)
    R = s.rhs(torch.from_numpy(U).cuda()).cpu().numpy()
    pick = np.zeros(m["E"], bool)
    pick[:2 * D] = pick[-(m["E"] % D) - D:] = True  # the first blocks, the last whole one and the partial one
    pick[np.random.default_rng(N).integers(0, m["E"], 40)] = True
    prm = oracle_params(s.params)
    q = O.Mesh(N, m["xyz"], m["period"], quad=True, metric_mask=pick, gauss=gauss).rhs(U, prm, want=pick)
    o = O.Mesh(N, m["xyz"], m["period"], metric_mask=pick, gauss=gauss).rhs(U, prm, want=pick)
    bound, floor = parity_bound(o[pick], q[pick])
    parity_check(rel_err(R[pick], q[pick]), bound, floor)
