"""Both kernels of the two-node shape at the edges of their tiles, per field.

* Single meshes with element counts that leave a remainder of one, none and
  one short of a group's and of a block's tile, at the degrees with a second
  kernel (stages that stand alone) from the size on from which the hand-off
  kernel is taken, and one element fewer; five launches a step and one.  Which
  of the two ran is asked with a wait limit of 0: only the hand-off kernel
  waits.
* Batches whose cases have element counts around the tiles, so that tiles hold
  elements of two cases with their own viscosity, mesh velocity and step.

The increment of a step is a sum of dt R, so its error is held, per field, to
the residual's own bound (MIXED_SENS times the FP32 sensitivity of that field)
or to INC_TOL where that is larger.
"""
import os
import re

import numpy as np
import pytest

import dg_inputs
import oracle
from dg_inputs.meshes import Mesh, _connect
from dg_inputs.states import to_kcn

from _parity import INC_TOL, MIXED_SENS, check_rhs, fp32_sensitivity, inc_err

pytestmark = pytest.mark.gpu
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_17917_gb300", "csrc")
FAR = dict(rho_inf=1.0, u_inf=1.0, v_inf=0.2, p_inf=17.857142857142858)


@pytest.fixture(scope="module")
def dg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_17917_gb300 import build
    build.build()
    import paper_2508_17917_gb300 as m
    return m


def first_handoff(p):
    text = open(os.path.join(CSRC, "stage_mixed.cu")).read()
    m = re.search(rf"p == {p} && K < (\d+)", text)
    return int(m.group(1)) if m else 1


def tiles(p):
    """Elements of a group's tile and of a block's (Sym64, Layout2)."""
    nodes, axis = (p + 1) * (p + 2) // 2, p // 2 + 1
    pairs = (nodes - axis) // 2
    threads = pairs + (axis + 1) // 2
    group = (32 if p <= 4 else 128) // threads
    return group, group * (4 if p <= 4 else 1)


def part_of(mesh, count):
    """The first `count` elements; the faces that this exposes are far field,
    the wall faces stay."""
    EToV = mesh.EToV[:count].copy()
    EToE, EToF, owner = _connect(EToV, np.arange(mesh.Nv))
    bc = np.zeros(EToV.shape, dtype=np.int32)
    for (k, f) in owner.values():
        bc[k, f] = mesh.bc[k, f] if mesh.bc[k, f] else 2
    return Mesh(mesh.vx, mesh.vy, EToV, EToE.astype(np.int32), EToF.astype(np.int32), bc, None, "part")


def bound(P, U, vw=(0.0, 0.0)):
    return np.maximum(INC_TOL["mixed"], MIXED_SENS * fp32_sensitivity(P, U, 0.0, vw))


def free_stream(P, seed):
    U = to_kcn(dg_inputs.free_stream(P.x.shape, rho=1.0, u=1.0, v=0.2, p=FAR["p_inf"]))
    return dg_inputs.perturb(U, seed=seed, amp=1e-2)


def hands_off(dg, s, U):
    s.set_state(U)
    dg.dg_set_barrier_limit(s.ctx, 0)
    try:
        s.steps(0.0, 1e-9, 1)
        s.get_state()
        return False
    except dg.DGError as e:
        assert e.status == -5
        return True
    finally:
        dg.dg_set_barrier_limit(s.ctx, 1 << 24)


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6])
def test_single_mesh(dg, p):
    import torch
    stream = torch.cuda.current_stream().cuda_stream
    first, (group, block) = first_handoff(p), tiles(p)
    whole = dg_inputs.ogrid_cylinder(*((128, 100, 0.5, 8.0) if first > 1 else (13, 10, 0.5, 4.0)), seed=3)
    at = -(-first // block) * block
    vw, kw = (0.0, 0.03), dict(mu=0.01, **FAR)
    counts = {first - 1, first, at, at + 1, at + group - 1, at + group + 1, at + block - 1, 2 if first == 1 else first}
    for count in sorted(c for c in counts if c > 0):
        mesh = part_of(whole, count)
        P = oracle.Problem(mesh, p, **kw)
        U = free_stream(P, seed=count)
        s = dg.Solver(mesh, p, "mixed", stream=stream, **kw)
        s.set_variant(2)
        if count < first or count > 1000:            # one block passes its own barrier at once
            assert hands_off(dg, s, U) == (count >= first)
        s.set_state(U)
        check_rhs(P, U, s.rhs(0.0, vw), "mixed", 0.0, vw)
        dt = P.dt(U, 0.1)[0]
        ref, tol = P.run(U, 0.0, dt, 1, vw), bound(P, U, vw)
        for fused in (False, True):
            s.set_fused(fused)
            s.set_state(U)
            s.steps(0.0, dt, 1, vw)
            assert np.all(inc_err(P, s.get_state(), ref, U) <= tol), (count, fused)
            dg.dg_barrier_status(s.ctx)


@pytest.mark.parametrize("fused", [0, 1])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6])
def test_batch(dg, p, fused):
    whole = dg_inputs.ogrid_cylinder(13, 6, 0.5, 4.0, seed=3)
    group, block = tiles(p)
    counts = [1, group - 1, group + 1, block - 1, block + 1, 2, 2 * block + 1, group]
    counts = [min(max(c, 1), whole.K) for c in counts]
    cases = [dict(mesh=part_of(whole, c), p=p, mu=0.005 * (1 + i), M_r=1.0, C_r=0.1, K_r=2.0, mass=8.0,
                  y0=0.02 * (i - 3), ydot0=0.1 * (i - 3)) for i, c in enumerate(counts)]
    b = dg.BatchSolver(cases, **FAR)
    b.set_variant(2)
    b.set_fused(fused)
    P = [oracle.Problem(c["mesh"], p, mu=c["mu"], **FAR) for c in cases]
    U = [free_stream(q, seed=i) for i, q in enumerate(P)]
    for i, u in enumerate(U):
        b.set_state(i, u)
    dts = [q.dt(u, 0.1 + 0.01 * i)[0] for i, (q, u) in enumerate(zip(P, U))]
    b.set_fixed_dt(dts)
    b.run(0.3, 1, use_graph=False)
    for i, (c, q, u, dt) in enumerate(zip(cases, P, U, dts)):
        assert b.variant(i) == 2
        F = q.wall_forces(u)
        _, vb = oracle.newmark_step((c["M_r"], c["C_r"], c["K_r"]), F[1] / c["mass"], dt,
                                    np.array([c["y0"], c["ydot0"], 0.0]))
        ref = q.lsrk_step(u, 0.0, dt, (0.0, vb))
        assert np.all(inc_err(q, b.get_state(i), ref, u) <= bound(q, u, (0.0, vb))), i
