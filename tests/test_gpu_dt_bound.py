"""The two-pass time-step bound (FP32 screen, FP64 on the elements that can
hold the maximum) against the oracle's bound.

The result is the FP64 maximum whatever the screen marks, so every case holds
the FP64 tolerance of the bound, 1e-12 relative: sizes around a tile of the
screen and a block of the FP64 pass, a uniform state (every element is within
the margin), a single element that holds the maximum, values outside the
range of FP32 (the screen marks everything), a state that is not finite.
"""
import numpy as np
import pytest

import dg_inputs
import oracle
from dg_inputs.states import to_kcn

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module")
def dg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_17917_gb300 import build
    build.build()
    import paper_2508_17917_gb300 as m
    return m


def stream():
    import torch
    return torch.cuda.current_stream().cuda_stream


def check(dg, mesh, p, U, vw, precision, **kw):
    P = oracle.Problem(mesh, p, **kw)
    ref, _ = P.dt(U, 0.3, vw)
    s = dg.Solver(mesh, p, precision, stream=stream(), **kw)
    s.set_state(U)
    for _ in range(2):                 # the second call finds the words of the first cleared
        assert abs(s.dt(0.3, vw) / ref - 1.0) <= TOL


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6])
def test_perturbed_states(dg, p, precision):
    for mesh, kw in ((dg_inputs.periodic_square(5), dict(mu=5e-3)),
                     (dg_inputs.ogrid_cylinder(13, 5, 0.5, 4.0, seed=2), dict(mu=0.01, p_inf=17.857142857142858))):
        P = oracle.Problem(mesh, p, **kw)
        U = to_kcn(dg_inputs.free_stream(P.x.shape, rho=1.0, u=1.0, v=0.1, p=kw.get("p_inf", 1.0)))
        check(dg, mesh, p, dg_inputs.perturb(U, seed=p, amp=1e-2), (0.07, -0.03), precision, **kw)


@pytest.mark.parametrize("n,p", [(9, 4), (128, 1), (282, 1)])
def test_uniform_state_marks_every_element(dg, n, p):
    """282: 159,048 elements, more than the FP64 pass looks at in one sweep of its blocks."""
    mesh = dg_inputs.periodic_square(n)
    P = oracle.Problem(mesh, p, mu=1e-3)
    U = to_kcn(dg_inputs.free_stream(P.x.shape, rho=1.0, u=0.4, v=0.1, p=1.0))
    check(dg, mesh, p, U, (0.0, 0.0), "mixed", mu=1e-3)


@pytest.mark.parametrize("where", [0, 700, 2047])
def test_one_element_holds_the_maximum(dg, where):
    mesh = dg_inputs.periodic_square(32)
    P = oracle.Problem(mesh, 3, mu=1e-3)
    U = to_kcn(dg_inputs.free_stream(P.x.shape, rho=1.0, u=0.4, v=0.1, p=1.0))
    U[where, 3] *= 40.0
    check(dg, mesh, 3, U, (0.0, 0.0), "mixed", mu=1e-3)


@pytest.mark.parametrize("rho,u,p", [(1e-30, 1.0, 1e-30), (1.0, 1e12, 1e24), (1e3, 1e-9, 1e-18)])
def test_values_outside_the_screens_range(dg, rho, u, p):
    mesh = dg_inputs.periodic_square(6)
    P = oracle.Problem(mesh, 2, mu=1e-3)
    U = dg_inputs.perturb(to_kcn(dg_inputs.free_stream(P.x.shape, rho=rho, u=u, v=0.3 * u, p=p)), seed=4, amp=1e-3)
    check(dg, mesh, 2, U, (0.0, 0.0), "fp64", mu=1e-3)


@pytest.mark.parametrize("bad", [np.inf, -np.inf])
def test_not_finite_is_reported(dg, bad):
    mesh = dg_inputs.periodic_square(12)
    s = dg.Solver(mesh, 2, "mixed", stream=stream(), mu=1e-3)
    x, y = s.node_coords()
    U = to_kcn(dg_inputs.free_stream(x.shape, rho=1.0, u=0.4, v=0.1, p=1.0))
    good = U.copy()
    U[100, 3, 2] = bad
    s.set_state(U)
    with pytest.raises(dg.DGError) as e:
        s.dt(0.3)
    assert e.value.status == -4
    s.set_state(good)
    P = oracle.Problem(mesh, 2, mu=1e-3)
    assert abs(s.dt(0.3) / P.dt(good, 0.3)[0] - 1.0) <= TOL
