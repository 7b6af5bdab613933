"""Rounding of the FP64 broken gradient against exact arithmetic: the error
with the symmetric contraction is no larger than that of the plain rows of the
library's operators, fused multiply-adds in row order as a kernel with a
thread per node forms them, over the fields and both directions.

Exact: the derivatives of the polynomial through the library's nodes, from a
monomial basis in extended precision (about 1e-19), and products in extended
precision; the element maps in FP64 are inputs of both sides.
"""
import numpy as np
import pytest

import dg_inputs
from dg_inputs.states import to_kcn

pytestmark = pytest.mark.gpu
ld = np.longdouble


@pytest.fixture(scope="module")
def dg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_17917_gb300 import build
    build.build()
    import paper_2508_17917_gb300 as m
    return m


def inverse(V):
    n = len(V)
    A = np.concatenate([V, np.eye(n, dtype=ld)], 1)
    for c in range(n):
        p = c + int(np.argmax(np.abs(A[c:, c])))
        A[[c, p]] = A[[p, c]]
        A[c] /= A[c, c]
        for r in range(n):
            if r != c:
                A[r] -= A[r, c] * A[c]
    return A[:, n:]


def exact_operators(r, s, p):
    r, s = ld(r), ld(s)
    powers = [(i, j) for i in range(p + 1) for j in range(p + 1 - i)]
    inv = inverse(np.stack([r ** i * s ** j for i, j in powers], 1))
    dr = np.stack([i * r ** max(i - 1, 0) * s ** j for i, j in powers], 1)
    ds = np.stack([r ** i * (j * s ** max(j - 1, 0)) for i, j in powers], 1)
    return dr @ inv, ds @ inv


def rows(A, u):
    """A u with one rounding per term."""
    out = np.zeros(u.shape)
    for j in range(A.shape[1]):
        out = (ld(A[:, j]) * ld(u[..., j:j + 1]) + ld(out)).astype(np.float64)
    return out


@pytest.mark.parametrize("p", [3, 4, 5, 6])         # the degrees that take it
def test_no_less_accurate_than_the_plain_rows(dg, p):
    import torch
    mesh = dg_inputs.periodic_square(32)
    s = dg.Solver(mesh, p, "fp64", stream=torch.cuda.current_stream().cuda_stream, mu=1e-3)
    x, y = s.node_coords()
    U = to_kcn(dg_inputs.isentropic_vortex(x, y))
    s.set_state(U)
    got = s.broken_gradient(0)
    o = dg.dg_reference_operators(p)
    vx, vy = mesh.vx[mesh.EToV], mesh.vy[mesh.EToV]
    xr, xs, yr, ys = (0.5 * (v[:, i] - v[:, 0]) for v in (vx, vy) for i in (1, 2))
    J = xr * ys - xs * yr
    rx, ry, sx, sy = ((v / J)[:, None, None] for v in (ys, -xs, -yr, xr))
    Er, Es = exact_operators(o["r"], o["s"], p)
    er, es = ld(U) @ Er.T, ld(U) @ Es.T
    pr, ps = rows(o["Dr"], U), rows(o["Ds"], U)
    ratio = []
    for g, a, b in ((got[0], rx, sx), (got[1], ry, sy)):
        exact = ld(a) * er + ld(b) * es
        plain = (ld(a) * ld(pr) + ld(b * ps)).astype(np.float64)
        err, ref = (np.sqrt(np.mean((np.asarray(v - exact, dtype=np.float64)) ** 2, axis=(0, 2))) for v in (g, plain))
        ratio += list(err / ref)
    assert np.sqrt(np.mean(np.square(ratio))) <= 1.0, ratio
