"""The bounded waits of the FP64 stage's phases and of the two-node kernel run
out when the caller's limit is 0: the launch ends early, the next call that
synchronises reports DG_ETIMEOUT, the flag is cleared, and with the limit
restored and the state set again the context gives the reference bit for bit.
The mesh has more tiles than one block takes, so the first blocks at a barrier
find it closed.  (No wait can run longer than the limit: nothing hangs.)
"""
import numpy as np
import pytest

import dg_inputs
from dg_inputs.states import to_kcn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_17917_gb300 import build
    build.build()
    import paper_2508_17917_gb300 as m
    return m


def solver(dg, p, precision, variant, fused):
    import torch
    s = dg.Solver(dg_inputs.periodic_square(64), p, precision, stream=torch.cuda.current_stream().cuda_stream, mu=1e-3)
    if variant:
        s.set_variant(variant)
    s.set_fused(fused)
    x, y = s.node_coords()
    return s, dg_inputs.perturb(to_kcn(dg_inputs.isentropic_vortex(x, y)), seed=3, amp=1e-3)


# the two-node kernel: a warp's tiles (p = 2, 4) and a block's (6)
@pytest.mark.parametrize("p,precision,variant,fused", [
    (2, "fp64", 0, False), (4, "fp64", 0, False), (2, "mixed", 2, False), (4, "mixed", 2, False),
    (2, "mixed", 2, True), (4, "mixed", 2, True), (6, "mixed", 2, False), (6, "mixed", 2, True)])
def test_waits_that_run_out_are_reported(dg, p, precision, variant, fused):
    s, U0 = solver(dg, p, precision, variant, fused)
    s.set_state(U0)
    residual = s.rhs()
    s.steps(0.0, 1e-5, 2)
    want = s.get_state()

    def call_step():
        s.steps(0.0, 1e-5, 2)
        s.get_state()

    def call_barrier_status():
        s.steps(0.0, 1e-5, 1)
        dg.dg_barrier_status(s.ctx)

    for call in (call_step, call_barrier_status) + (() if fused else (lambda: s.rhs(),)):
        s.set_state(U0)
        dg.dg_set_barrier_limit(s.ctx, 0)
        with pytest.raises(dg.DGError) as e:
            call()
        assert e.value.status == -5
        dg.dg_barrier_status(s.ctx)                   # the flag was cleared
        dg.dg_set_barrier_limit(s.ctx, 1 << 24)
        s.set_state(U0)
        assert np.array_equal(s.rhs(), residual)
        s.steps(0.0, 1e-5, 2)
        assert np.array_equal(s.get_state(), want)
