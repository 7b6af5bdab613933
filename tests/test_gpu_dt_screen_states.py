"""The two-pass time-step bound at states that the FP32 screen finds hard:
gamma / Pr above 2 and speeds far from 1, where the penalty norm cancels, and
velocities that differ from element to element so that many come close to the
maximum.  The result is the FP64 maximum whatever the screen marks, so it
holds the FP64 tolerance against the oracle, 1e-12 relative."""
import numpy as np
import pytest

import dg_inputs
import oracle

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


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("Pr", [0.72, 0.6, 0.28])
@pytest.mark.parametrize("speed", [1e-3, 1.0, 2500.0, 8000.0])
@pytest.mark.parametrize("ratio", [2e-3, 0.02, 1.0, 17.0])
def test_hard_states(dg, precision, Pr, speed, ratio):
    """ratio: pressure over rho v^2; 2e-3 is a Mach number of 19."""
    import torch
    mesh = dg_inputs.periodic_square(24)
    kw = dict(mu=1e-3, Pr=Pr)
    P = oracle.Problem(mesh, 2, **kw)
    rng = np.random.default_rng(7)
    K, Np = P.x.shape
    th = rng.uniform(0, 2 * np.pi, (K, 1)) + 0.01 * rng.normal(size=(K, Np))
    v = speed * (1 + 0.02 * rng.normal(size=(K, 1))) * (1 + 1e-4 * rng.normal(size=(K, Np)))
    rho = 1 + 1e-3 * rng.normal(size=(K, Np))
    p = ratio * speed ** 2 * (1 + 1e-3 * rng.normal(size=(K, Np)))
    U = np.stack([rho, rho * v * np.cos(th), rho * v * np.sin(th), p / 0.4 + 0.5 * rho * v * v], axis=1)
    s = dg.Solver(mesh, 2, precision, stream=torch.cuda.current_stream().cuda_stream, **kw)
    s.set_state(U)
    for vw in ((0.0, 0.0), (0.3 * speed, -0.9 * speed)):
        ref = P.dt(U, 0.3, vw)[0]
        assert abs(s.dt(0.3, vw) / ref - 1.0) <= TOL
