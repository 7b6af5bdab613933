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
import oracle
from dg_inputs.states import to_kcn

from _parity import INC_TOL, RHS_TOL_ALL_FP64, STATE_TOL, all_err, check_rhs, inc_err

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


@pytest.fixture
def take_all_but(dg):
    """take_all_but(n) leaves about n bytes of the device's memory."""
    import torch
    cu = C.CDLL("libcuda.so.1")
    held = []

    def alloc(size, most):
        got = 0
        p = C.c_uint64()
        while got + size <= most and cu.cuMemAlloc_v2(C.byref(p), C.c_size_t(size)) == 0:
            held.append((p.value, size))
            got += size
        return got

    def take(n):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        for size in (1024 * MB, 64 * MB, 2 * MB):
            alloc(size, 1 << 40)
        freed = 0
        while freed < n:
            p, size = held.pop()
            assert cu.cuMemFree_v2(C.c_uint64(p)) == 0
            freed += size
        alloc(2 * MB, freed - n)

    yield take
    torch.cuda.synchronize()
    for p, _ in held:
        cu.cuMemFree_v2(C.c_uint64(p))


@pytest.mark.parametrize("p,theta", [(4, 0.0), (2, 1.0)])
def test_fp64_without_memory_between_the_phases(dg, part_of_the_device, take_all_but, p, theta):
    """All but what the state needs, and half of what the phases need besides,
    is taken.  Same kernel, and so the same bits, as on a part of the device."""
    mesh = dg_inputs.periodic_square(400)               # 320,000 elements
    kw = dict(mu=1e-3, theta=theta, C1=0.05)
    alone = dg.Solver(mesh, p, "fp64", stream=part_of_the_device, **kw)
    U = vortex(alone)
    alone.set_state(U)
    want = alone.rhs()
    dt = alone.dt(0.3)
    alone.steps(0.0, dt, 1)
    after = alone.get_state()
    del alone
    Np, nfn = (p + 1) * (p + 2) // 2, 3 * (p + 1)
    state = mesh.K * (4 * 32 * Np + 128 + 16 + 4)       # two states, register, residual; element records
    phases = mesh.K * (64 * Np + 32 * nfn + (64 * nfn if theta else 0))
    take_all_but(state + phases // 2)
    s = dg.Solver(mesh, p, "fp64", stream=stream(), **kw)
    s.set_state(U)
    assert np.array_equal(s.rhs(), want)
    assert s.dt(0.3) == dt
    s.steps(0.0, dt, 1)
    assert np.array_equal(s.get_state(), after)


@pytest.mark.parametrize("p,variant", [(1, 2), (2, 2), (4, 2), (6, 2), (4, 0), (6, 0)])
def test_mixed_on_a_part_of_the_device(dg, part_of_the_device, p, variant):
    mesh = dg_inputs.periodic_square(64)
    P = oracle.Problem(mesh, p, mu=1e-3)
    s = dg.Solver(mesh, p, "mixed", stream=part_of_the_device, mu=1e-3)
    s.set_variant(variant)
    U = dg_inputs.perturb(to_kcn(dg_inputs.isentropic_vortex(P.x, P.y)), seed=3, amp=1e-3)
    s.set_state(U)
    check_rhs(P, U, s.rhs(), "mixed")
    dt = P.dt(U, 0.3)[0]
    s.steps(0.0, dt, 2)
    got = s.get_state()
    assert np.all(inc_err(P, got, P.run(U, 0.0, dt, 2), U) <= INC_TOL["mixed"])
    s.set_state(U)
    s.steps(0.0, dt, 2)
    assert np.array_equal(s.get_state(), got)


@pytest.mark.parametrize("p", [2, 4])
def test_two_nodes_without_memory_between_the_stages(dg, part_of_the_device, take_all_but, p):
    """As for the FP64 phases; five launches a step and one."""
    mesh = dg_inputs.periodic_square(400)
    alone = dg.Solver(mesh, p, "mixed", stream=part_of_the_device, mu=1e-3)
    U = vortex(alone)
    alone.set_variant(2)
    alone.set_state(U)
    want = alone.rhs()
    alone.steps(0.0, 1e-5, 2)
    after = alone.get_state()
    del alone
    Np = (p + 1) * (p + 2) // 2
    state = mesh.K * (4 * 32 * Np + 2 * 16 * Np + 2 * 4 * ((Np + 3) & ~3) + 192 + 16 + 4)
    stages = mesh.K * 16 * (Np + 6 * (p + 1))
    take_all_but(state + stages // 2)
    s = dg.Solver(mesh, p, "mixed", stream=stream(), mu=1e-3)
    s.set_variant(2)
    s.set_state(U)
    assert np.array_equal(s.rhs(), want)
    s.steps(0.0, 1e-5, 2)
    assert np.array_equal(s.get_state(), after)
    s.set_fused(True)
    s.set_state(U)
    s.steps(0.0, 1e-5, 2)
    assert np.abs(s.get_state() - after).max() <= 1e-9 * np.abs(after).max()


def test_the_two_node_arrays_go_when_another_shape_is_taken(dg):
    mesh = dg_inputs.periodic_square(200)               # 80,000 elements: 58 MB between the stages at p = 4
    s = dg.Solver(mesh, 4, "mixed", stream=stream(), mu=1e-3)
    s.set_state(vortex(s))
    for v in (1, 2, 3):                                 # every kernel is loaded
        s.set_variant(v)
        s.steps(0.0, 1e-6, 1)
    without = free_bytes()
    s.set_variant(2)
    assert without - free_bytes() >= 50 * MB
    s.set_variant(1)
    assert abs(without - free_bytes()) <= 4 * MB
    s.set_variant(0)
    s.steps(0.0, 1e-6, 1)
    if s.variant != 2:
        assert abs(without - free_bytes()) <= 4 * MB


def test_batch_without_memory_between_the_stages(dg, take_all_but):
    """A group takes the one-node shape instead of the two-node shape."""
    kw = dict(rho_inf=1.0, u_inf=1.0, v_inf=0.0, p_inf=17.857142857142858)
    case = dict(mesh=dg_inputs.ogrid_cylinder(400, 100, 0.5, 20.0, seed=1), p=4, mu=0.01, y0=0.0, ydot0=0.0, M_r=1.0,
                C_r=0.1, K_r=2.0, mass=8.0)             # 80,000 elements: 58 MB between the stages
    got = []
    for variant in (1, 2):
        b = dg.BatchSolver([case], **kw)
        b.set_variant(variant)
        x, y = b.node_coords(0)
        b.set_state(0, to_kcn(dg_inputs.free_stream(x.shape, rho=1.0, u=1.0, v=0.0, p=kw["p_inf"])))
        if variant == 2:
            take_all_but(24 * MB)
        b.run(0.3, 2, use_graph=False)
        assert b.variant(0) == 1
        got.append(b.get_state(0))
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("precision,fused", [("fp64", False), ("mixed", False), ("mixed", True)])
def test_arrays_in_a_callers_graph_stay(dg, precision, fused):
    """Steps captured into a graph of the caller's hold the addresses of the
    arrays between phases or stages: another shape, over-integration or the
    tuner does not give them back, and the graph replays the same steps."""
    import torch
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        s = dg.Solver(dg_inputs.periodic_square(200), 4, precision, stream=st.cuda_stream, mu=1e-3)
        if precision == "mixed":
            s.set_variant(2)
            s.set_fused(fused)
        U = vortex(s)
        s.set_state(U)
        s.steps(0.0, 1e-5, 2)
        want = s.get_state()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            s.steps(0.0, 1e-5, 2)
        held = free_bytes()
        if precision == "fp64":
            s.set_overint(True)
        else:
            s.set_fused(False)
            s.set_variant(3)
            s.set_variant(0)
            s.set_state(U)
            s.steps(0.0, 1e-5, 2)
        assert held - free_bytes() >= -MB
        s.set_state(U)
        g.replay()
        st.synchronize()
        assert np.array_equal(s.get_state(), want)
        del g
