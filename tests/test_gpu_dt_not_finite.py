"""States without a time-step bound: dg_compute_dt reports them.

Lambda_K is a maximum of terms, and a maximum taken with fmax drops a NaN: a
blown-up state would come back with the bound of its other nodes.  Each case
puts one value that has no Lambda_K at one node of one element, on a face or
in the interior, and expects DG_ENONFINITE, then the oracle's bound for the
state without it.
"""
import numpy as np
import pytest

import dg_inputs
import oracle
from dg_inputs.states import to_kcn

pytestmark = pytest.mark.gpu
TOL = 1e-12
P = 4
VERTEX, INTERIOR = 0, 6        # node rows 0..4, 5..8, ...: (0, 0) and (1, 1) of p = 4


@pytest.fixture(scope="module")
def dg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_17917_gb300 import build
    build.build()
    import paper_2508_17917_gb300 as m
    return m


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("node", [VERTEX, INTERIOR])
@pytest.mark.parametrize("field,value", [(0, np.nan), (1, np.nan), (2, np.nan), (3, np.nan), (0, np.inf),
                                         (2, -np.inf), (0, 0.0), (3, -1.0)])
def test_reported(dg, precision, node, field, value):
    import torch
    mesh = dg_inputs.periodic_square(12)
    s = dg.Solver(mesh, P, precision, stream=torch.cuda.current_stream().cuda_stream, mu=1e-3)
    x, y = s.node_coords()
    good = to_kcn(dg_inputs.free_stream(x.shape, rho=1.0, u=0.4, v=0.1, p=1.0))
    U = good.copy()
    U[100, field, node] = value                # (3, -1.0): a negative pressure
    s.set_state(U)
    for vw in (None, (0.2, -0.1)):             # a moving mesh has a wave speed where the flow has none
        with pytest.raises(dg.DGError) as e:
            s.dt(0.3, vw)
        assert e.value.status == -4
    s.set_state(good)
    ref = oracle.Problem(mesh, P, mu=1e-3).dt(good, 0.3)[0]
    assert abs(s.dt(0.3) / ref - 1.0) <= TOL
