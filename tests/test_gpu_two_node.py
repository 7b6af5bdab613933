"""The two-node tile shape of the mixed stage kernel (variant 2) where its
tiles can go wrong: element counts around a group's tile and around a block's,
a mesh of one and of two elements, wall and far-field faces, residuals and
updates, five launches a step and one; and both sides of the sizes from which
the hand-off kernel takes p = 3 and 5.  Residuals as everywhere on the mixed
path (tests/_parity.py); the increment of a step is a sum of dt R, so its
error per field is held to the residual's own bound, MIXED_SENS times the
FP32 sensitivity, and to INC_TOL where that is the larger one."""
import numpy as np
import pytest

import dg_inputs
import oracle
from dg_inputs.meshes import Mesh, _connect
from dg_inputs.states import to_kcn

from _parity import INC_TOL, MIXED_SENS, check_rhs, fp32_sensitivity, inc_err

pytestmark = pytest.mark.gpu
TILE = {1: (16, 64), 2: (10, 40), 3: (6, 24), 4: (4, 16), 5: (11, 11), 6: (9, 9)}    # elements per group, per block
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


def part_of(mesh, count):
    """The first `count` elements; the faces that this exposes are far field,
    the wall faces stay."""
    EToV = mesh.EToV[:count].copy()
    EToE, EToF, owner = _connect(EToV, np.arange(mesh.Nv))
    bc = np.zeros(EToV.shape, dtype=np.int32)
    for (k, f) in owner.values():
        bc[k, f] = mesh.bc[k, f] if mesh.bc[k, f] else 2
    return Mesh(mesh.vx, mesh.vy, EToV, EToE.astype(np.int32), EToF.astype(np.int32), bc, None, "part")


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6])
def test_tile_edges(dg, p):
    import torch
    stream = torch.cuda.current_stream().cuda_stream
    whole = dg_inputs.ogrid_cylinder(13, 6, 0.5, 4.0, seed=3)
    group, block = TILE[p]
    counts = {1, 2, group - 1, group, group + 1, block - 1, block, block + 1, 2 * block + 1}
    for count in sorted(c for c in counts if 0 < c <= whole.K):
        mesh = part_of(whole, count)
        P = oracle.Problem(mesh, p, **KW)
        U = to_kcn(dg_inputs.free_stream(P.x.shape, rho=1.0, u=1.0, v=0.2, p=KW["p_inf"]))
        U = dg_inputs.perturb(U, seed=count, amp=1e-2)
        vw = (0.0, 0.03)
        s = dg.Solver(mesh, p, "mixed", stream=stream, **KW)
        s.set_variant(2)
        s.set_state(U)
        check_rhs(P, U, s.rhs(0.0, vw), "mixed", 0.0, vw)
        dt = P.dt(U, 0.1)[0]
        ref = P.run(U, 0.0, dt, 2, vw)
        bound = max(INC_TOL["mixed"], MIXED_SENS * fp32_sensitivity(P, U, 0.0, vw).max())
        for fused in (False, True):
            s.set_fused(fused)
            s.set_state(U)
            s.steps(0.0, dt, 2, vw)
            assert np.all(inc_err(P, s.get_state(), ref, U) <= bound), (count, fused)
            dg.dg_barrier_status(s.ctx)


@pytest.mark.parametrize("p, count", [(3, 24999), (3, 25001), (5, 14999), (5, 15001)])
def test_both_kernels(dg, p, count):
    import torch
    mesh = part_of(dg_inputs.ogrid_cylinder(128, 98, 0.5, 8.0, seed=3), count)
    P = oracle.Problem(mesh, p, **KW)
    U = to_kcn(dg_inputs.free_stream(P.x.shape, rho=1.0, u=1.0, v=0.2, p=KW["p_inf"]))
    U = dg_inputs.perturb(U, seed=p, amp=1e-2)
    vw = (0.0, 0.03)
    s = dg.Solver(mesh, p, "mixed", stream=torch.cuda.current_stream().cuda_stream, **KW)
    s.set_variant(2)
    s.set_state(U)
    check_rhs(P, U, s.rhs(0.0, vw), "mixed", 0.0, vw)
    dt = P.dt(U, 0.1)[0]
    ref = P.run(U, 0.0, dt, 1, vw)
    s.steps(0.0, dt, 1, vw)
    assert np.all(inc_err(P, s.get_state(), ref, U) <= INC_TOL["mixed"])
