"""The three-phase FP64 stage (every face once, symmetric contractions) where
its tiles can go wrong: element counts around a block's tile, a mesh of one
and of two elements, boundary faces only, and the theta terms there.  Same
tolerances as the FP64 residual everywhere (tests/_parity.py)."""
import numpy as np
import pytest

import dg_inputs
import oracle
from dg_inputs.meshes import Mesh, _connect
from dg_inputs.states import to_kcn

from _parity import RHS_TOL_ALL_FP64, RHS_TOL_FIELD_FP64, all_err, field_err

pytestmark = pytest.mark.gpu
TILE = {1: 64, 2: 42, 3: 25, 4: 16, 5: 11, 6: 9}      # elements per block and pass
KW = dict(mu=0.01, rho_inf=1.0, u_inf=1.0, v_inf=0.2, p_inf=17.857142857142858)


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


def part_of(mesh, count):
    """The first `count` elements; the faces that this exposes are far field,
    the wall faces stay."""
    EToV = mesh.EToV[:count].copy()
    EToE, EToF, owner = _connect(EToV, np.arange(mesh.Nv))
    bc = np.zeros(EToV.shape, dtype=np.int32)
    for (k, f) in owner.values():
        bc[k, f] = mesh.bc[k, f] if mesh.bc[k, f] else 2
    return Mesh(mesh.vx, mesh.vy, EToV, EToE.astype(np.int32), EToF.astype(np.int32), bc, None, "part")


@pytest.mark.parametrize("theta", [0.0, 1.0, -0.5])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6])
def test_rhs_tile_edges(dg, p, theta):
    kw = dict(KW, theta=theta, C1=0.05)
    whole = dg_inputs.ogrid_cylinder(13, 6, 0.5, 4.0, seed=3)
    t = TILE[p]
    for count in sorted({1, 2, t - 1, t, t + 1, 2 * t + 1}):
        mesh = part_of(whole, min(count, whole.K))
        P = oracle.Problem(mesh, p, **kw)
        U = to_kcn(dg_inputs.free_stream(P.x.shape, rho=1.0, u=1.0, v=0.2, p=kw["p_inf"]))
        U = dg_inputs.perturb(U, seed=count, amp=1e-2)
        vw = (0.0, 0.03)
        s = dg.Solver(mesh, p, "fp64", stream=stream(), **kw)
        s.set_state(U)
        got, ref = s.rhs(0.0, vw), P.rhs(U, vw=vw)
        assert all_err(got, ref) <= RHS_TOL_ALL_FP64, count
        assert np.all(field_err(got, ref) <= RHS_TOL_FIELD_FP64), count


def test_phase_words_are_left_clean(dg):
    """Two contexts in turn, residuals and steps mixed: no launch leaves its
    barrier in a state that the next one reads."""
    mesh = dg_inputs.periodic_square(9)
    P = oracle.Problem(mesh, 3, mu=1e-3)
    U = dg_inputs.perturb(to_kcn(dg_inputs.isentropic_vortex(P.x, P.y)), seed=1, amp=1e-3)
    a, b = (dg.Solver(mesh, 3, "fp64", stream=stream(), mu=1e-3) for _ in range(2))
    for s in (a, b):
        s.set_state(U)
    ref = a.rhs()
    for s in (a, b, a):
        assert np.array_equal(s.rhs(), ref)
    a.steps(0.0, 1e-4, 3)
    for _ in range(3):
        b.step(0.0, 1e-4)
        b.rhs()
    assert np.array_equal(a.get_state(), b.get_state())
    dg.dg_barrier_status(a.ctx)
