"""Calls whose faster kernel finds no place: no memory for the arrays that it
keeps between its phases or stages, or a stream with a part of the device's
multiprocessors, which refuses its grid as a cooperative launch.  They run
with the kernel that needs neither, within the parity bounds of the other
kernels; nothing is refused.
"""
import ctypes as C

import numpy as np
import pytest

import dg_inputs
from dg_inputs.states import to_kcn

from _parity import RHS_TOL_ALL_FP64, STATE_TOL, all_err

pytestmark = pytest.mark.gpu
MB = 1 << 20


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


def vortex(s):
    x, y = s.node_coords()
    return to_kcn(dg_inputs.isentropic_vortex(x, y))


def free_bytes():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.fixture
def part_of_the_device(dg):
    """A stream of a green context with a part of the multiprocessors."""
    import torch
    torch.zeros(1, device="cuda")
    cu = C.CDLL("libcuda.so.1")

    def ok(r):
        if r != 0:
            pytest.skip(f"no green context here (error {r})")

    whole, part, rest = (C.create_string_buffer(4096) for _ in range(3))
    n, desc, ctx, st = C.c_uint(1), C.c_void_p(), C.c_void_p(), C.c_void_p()
    ok(cu.cuDeviceGetDevResource(0, whole, 1))
    ok(cu.cuDevSmResourceSplitByCount(part, C.byref(n), whole, rest, 0, 32))
    ok(cu.cuDevResourceGenerateDesc(C.byref(desc), part, 1))
    ok(cu.cuGreenCtxCreate(C.byref(ctx), desc, 0, 1))
    ok(cu.cuGreenCtxStreamCreate(C.byref(st), ctx, 1, 0))
    yield st.value
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(st)
    cu.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("p,theta", [(2, 0.0), (4, 0.0), (4, 1.0)])
def test_fp64_on_a_part_of_the_device(dg, part_of_the_device, p, theta):
    mesh = dg_inputs.periodic_square(64)                # more tiles than the part holds blocks
    kw = dict(mu=1e-3, theta=theta, C1=0.05)
    ref = dg.Solver(mesh, p, "fp64", stream=stream(), **kw)
    s = dg.Solver(mesh, p, "fp64", stream=part_of_the_device, **kw)
    U = vortex(ref)
    for q in (ref, s):
        q.set_state(U)
    assert all_err(s.rhs(), ref.rhs()) <= RHS_TOL_ALL_FP64
    for q in (ref, s):
        q.steps(0.0, 1e-5, 2)
    assert all_err(s.get_state(), ref.get_state()) <= STATE_TOL["fp64"]
    dg.dg_barrier_status(s.ctx)


def test_over_integration_keeps_no_phase_arrays(dg):
    mesh = dg_inputs.periodic_square(200)               # 80,000 elements: 115 MB between the phases at p = 4
    free0 = free_bytes()
    s = dg.Solver(mesh, 4, "fp64", stream=stream(), mu=1e-3)
    U = vortex(s)
    s.set_state(U)
    s.rhs()
    phases = free_bytes()
    s.set_overint(True)
    assert free_bytes() - phases >= 100 * MB
    s.rhs()
    s.set_overint(False)
    ref = s.rhs()
    assert abs(free_bytes() - phases) <= 4 * MB
    t = dg.Solver(mesh, 4, "fp64", stream=stream(), mu=1e-3)
    t.set_state(U)
    assert np.array_equal(t.rhs(), ref)
    assert free0 > phases


@pytest.mark.parametrize("p,theta", [(4, 0.0), (2, 1.0)])
def test_fp64_without_memory_between_the_phases(dg, p, theta):
    """All but what the state needs, and half of what the phases need besides,
    is taken."""
    import torch
    mesh = dg_inputs.periodic_square(400)               # 320,000 elements
    kw = dict(mu=1e-3, theta=theta, C1=0.05)
    torch.cuda.empty_cache()
    free0 = free_bytes()
    ref = dg.Solver(mesh, p, "fp64", stream=stream(), **kw)
    U = vortex(ref)
    ref.set_state(U)
    want = ref.rhs()
    dt = ref.dt(0.3)
    used = free0 - free_bytes()
    Np, nfn = (p + 1) * (p + 2) // 2, 3 * (p + 1)
    phases = mesh.K * (64 * Np + 32 * nfn + (64 * nfn if theta else 0))
    assert used > phases
    del ref
    hold = torch.empty(free_bytes() - (used - phases // 2), dtype=torch.uint8, device="cuda")
    try:
        s = dg.Solver(mesh, p, "fp64", stream=stream(), **kw)
        s.set_state(U)
        assert all_err(s.rhs(), want) <= RHS_TOL_ALL_FP64
        assert s.dt(0.3) == dt
        s.steps(0.0, dt, 1)
        assert np.all(np.isfinite(s.get_state()))
    finally:
        del hold
        torch.cuda.empty_cache()
