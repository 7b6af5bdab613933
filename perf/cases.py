"""The work that a user of this library has it do, as cases that can be timed.

Every case goes through the public Python calls (`Solver`, `BatchSolver`,
`Mlp` and the `dg_*` functions of the binding) with what a user's program has
in hand: a context with its mesh and a state on the device, a batch of cases,
a network with its training set.  A pass of a time-stepping case advances the
state it finds, as a run does, and reads it back whole, in FP64; motions and
loads are logged in FP32 (the mixed path's stated accuracy of loads is 1e-4).

`exact` states the same results in plain torch FP64 (the nodal
interior-penalty DG residual in strong form, the five-stage 2N-storage
Runge-Kutta scheme, the time-step bound, the wall forces and the Newmark step
of the coupled loop; the network without its bfloat16 roundings).
"""
import functools
import math

import numpy as np
import torch

import paper_2508_17917_gb300 as dg

GAMMA, PRANDTL = 1.4, 0.72
MACH = 0.2                                    # of the cylinder flows
P_INF = 1.0 / (GAMMA * MACH * MACH)
WIDTH, DEPTH, N_IN, N_OUT = 128, 3, 67, 2     # the load surrogate's network
CFL = 0.1
DEV = "cuda" if torch.cuda.is_available() else "cpu"

# One step on 512 x 512 split quads at p = 4: nothing costs more
MOST_DOF_STEPS = 4 * 524288 * 15


def listed():
    return [
        # the smallest solver run: the 512-triangle vortex that a user starts
        # with, two steps between two looks at the state (launches count)
        dict(name="vortex_p2_k512", kind="vortex", precision="mixed", p=2, n=16, theta=0.0, steps=2, host=False),
        # the benchmark's vortex at its own size, mixed precision
        dict(name="vortex_p4_k32768", kind="vortex", precision="mixed", p=4, n=128, theta=0.0, steps=5, host=False),
        # a mesh whose state is far larger than the L2 cache
        dict(name="vortex_p4_k524288", kind="vortex", precision="mixed", p=4, n=512, theta=0.0, steps=1, host=False),
        # the same benchmark mesh on the plain FP64 path
        dict(name="vortex_p4_k32768_fp64", kind="vortex", precision="fp64", p=4, n=128, theta=0.0, steps=1,
             host=False),
        # the weakly coupled loop on the fixed 40,800-triangle cylinder mesh:
        # time-step bound, Newmark step, Runge-Kutta step, wall forces
        dict(name="cylinder_p4_coupled", kind="coupled", p=4, n_theta=120, n_r=170, steps=4),
        # symmetric interior penalty on an O-grid with odd counts
        dict(name="sip_p3_ogrid", kind="cylinder", precision="mixed", p=3, n_theta=91, n_r=61, theta=1.0, steps=5,
             host=False),
        # the highest degree on the 80,000-triangle cylinder mesh
        dict(name="cylinder_p6_k80000", kind="cylinder", precision="mixed", p=6, n_theta=200, n_r=200, theta=0.0,
             steps=1, host=False),
        # a reduced-velocity sweep: cases of 10k to 20k triangles and degrees
        # 3 to 6, advanced together with everything on the device
        dict(name="viv_batch", kind="batch", cases=12, k_min=10000, k_max=20000, p_min=3, p_max=6, steps=2,
             fixed=False),
        # the screening sweep over physical time: twelve 768-triangle cases at
        # a fixed step, run between two samples
        dict(name="viv_screen", kind="batch", cases=12, k_min=768, k_max=768, p_min=3, p_max=3, steps=8, fixed=True),
        # the broken gradient of a state (vorticity and stress output), the
        # call's default arithmetic
        dict(name="gradient_p4_k131072", kind="gradient", p=4, n=256, impl=0),
        # training of the load surrogate on a full batch of windows
        dict(name="mlp_train_b4096", kind="mlp_train", rows=4096, steps=20),
        # its prediction for the twelve cases of a screen
        dict(name="mlp_predict_b12", kind="mlp_predict", rows=12),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["vortex", "vortex", "cylinder", "cylinder", "coupled", "batch", "gradient", "mlp_train",
                       "mlp_predict"])
    p = rng.randint(1, 6)
    nodes = (p + 1) * (p + 2) // 2
    if kind in ("vortex", "cylinder"):
        precision = rng.choice(["mixed", "mixed", "fp64"])
        # an FP64 pass costs about 30 times a mixed one
        most = MOST_DOF_STEPS // (30 if precision == "fp64" else 1)
        c = dict(kind=kind, precision=precision, p=p, theta=rng.choice([0.0, 0.0, 1.0]), host=rng.random() < 0.25)
        if kind == "vortex":
            c["n"] = _log_int(rng, 8, min(512, math.isqrt(most // (8 * nodes))))
            k = 2 * c["n"] ** 2
        else:
            c["n_theta"] = _log_int(rng, 24, 200)
            c["n_r"] = _log_int(rng, 8, max(9, min(200, most // (8 * nodes * c["n_theta"]))))
            k = 2 * c["n_theta"] * c["n_r"]
        c["steps"] = max(1, min(rng.randint(1, 5 if k > 4000 else 2), most // (4 * nodes * k)))
        return c
    if kind == "coupled":
        return dict(kind=kind, p=p, n_theta=_log_int(rng, 24, 160), n_r=_log_int(rng, 8, 170), steps=rng.randint(1, 5))
    if kind == "batch":
        small = rng.random() < 0.5
        k_min = _log_int(rng, 300, 1200) if small else _log_int(rng, 1200, 12000)
        lo = rng.randint(1, 6)
        return dict(kind=kind, cases=rng.randint(4, 16), k_min=k_min, k_max=int(k_min * rng.uniform(1.0, 2.0)),
                    p_min=lo, p_max=rng.randint(lo, 6), steps=rng.randint(4, 12) if small else rng.randint(1, 3),
                    fixed=small)
    if kind == "gradient":
        impl = rng.randint(0, 1)
        return dict(kind=kind, p=p, n=_log_int(rng, 8, math.isqrt(MOST_DOF_STEPS // (8 * nodes))), impl=impl)
    if kind == "mlp_train":
        return dict(kind=kind, rows=_log_int(rng, 256, 8192), steps=rng.randint(8, 40))
    return dict(kind=kind, rows=_log_int(rng, 1, 8192))


# ---- meshes -----------------------------------------------------------------

class Mesh:
    """What `Solver` and `BatchSolver` take as a mesh."""

    def __init__(self, vx, vy, tri, canon):
        x, y = vx[tri], vy[tri]
        area = (x[:, 1] - x[:, 0]) * (y[:, 2] - y[:, 0]) - (x[:, 2] - x[:, 0]) * (y[:, 1] - y[:, 0])
        tri = np.where((area < 0)[:, None], tri[:, [0, 2, 1]], tri)
        self.vx, self.vy, self.EToV = vx, vy, np.ascontiguousarray(tri, dtype=np.int32)
        self.K = len(tri)
        a, b = canon[tri].astype(np.int64).ravel(), canon[np.roll(tri, -1, axis=1)].astype(np.int64).ravel()
        order = np.lexsort((np.maximum(a, b), np.minimum(a, b)))
        lo, hi = np.minimum(a, b)[order], np.maximum(a, b)[order]
        first = np.nonzero((lo[1:] == lo[:-1]) & (hi[1:] == hi[:-1]))[0]
        other = np.arange(3 * self.K)
        other[order[first]], other[order[first + 1]] = order[first + 1], order[first]
        self.EToE = (other // 3).astype(np.int32).reshape(-1, 3)
        self.EToF = (other % 3).astype(np.int32).reshape(-1, 3)
        self.bc = np.zeros((self.K, 3), dtype=np.int32)
        self.alone = (other == np.arange(3 * self.K)).reshape(-1, 3)


@functools.lru_cache(maxsize=2)
def _square(n, side=10.0):
    """Periodic square of n x n quads split along their diagonals."""
    at = np.arange(n + 1) * (side / n)
    vx, vy = np.tile(at, n + 1), np.repeat(at, n + 1)
    i, j = np.tile(np.arange(n), n), np.repeat(np.arange(n), n)
    a, b, c, d = (j * (n + 1) + i, j * (n + 1) + i + 1, (j + 1) * (n + 1) + i + 1, (j + 1) * (n + 1) + i)
    tri = np.stack([np.stack([a, b, c], 1), np.stack([a, c, d], 1)], 1).reshape(-1, 3)
    v = np.arange(vx.size)
    return Mesh(vx, vy, tri, (v % (n + 1)) % n + ((v // (n + 1)) % n) * n)


@functools.lru_cache(maxsize=32)
def _ogrid(n_theta, n_r, seed, r0=0.5, r1=30.0):
    """O-grid around a cylinder, radially stretched, with seeded diagonals."""
    h = 2.0 * math.pi * r0 / n_theta
    if h * n_r >= r1 - r0:
        radii = np.linspace(r0, r1, n_r + 1)
    else:
        lo, hi = 1.0 + 1e-12, 64.0
        for _ in range(200):
            q = 0.5 * (lo + hi)
            lo, hi = (lo, q) if h * (q ** n_r - 1.0) / (q - 1.0) > r1 - r0 else (q, hi)
        radii = r0 + h * (q ** np.arange(n_r + 1) - 1.0) / (q - 1.0)
    th = 2.0 * math.pi * np.arange(n_theta) / n_theta
    vx, vy = np.outer(radii, np.cos(th)).ravel(), np.outer(radii, np.sin(th)).ravel()
    k, i = np.repeat(np.arange(n_r), n_theta), np.tile(np.arange(n_theta), n_r)
    a, b = k * n_theta + i, k * n_theta + (i + 1) % n_theta
    c, d = b + n_theta, a + n_theta
    f = np.random.default_rng(seed).integers(0, 2, k.size).astype(bool)[:, None]
    t1 = np.where(f, np.stack([a, b, c], 1), np.stack([a, b, d], 1))
    t2 = np.where(f, np.stack([a, c, d], 1), np.stack([b, c, d], 1))
    m = Mesh(vx, vy, np.stack([t1, t2], 1).reshape(-1, 3), np.arange(vx.size))
    ring = m.EToV // n_theta
    wall = m.alone & (ring == 0) & (np.roll(ring, -1, axis=1) == 0)
    m.bc[wall], m.bc[m.alone & ~wall] = 1, 2
    return m


def _mesh(c):
    return _square(c["n"]) if "n" in c else _ogrid(c["n_theta"], c["n_r"], 0)


# ---- states -----------------------------------------------------------------

def _noise(shape, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + 17)
    return 2.0 * torch.rand(shape, generator=g, device=DEV, dtype=torch.float64) - 1.0


def _vortex(x, y, seed):
    """The isentropic vortex on [0, 10]^2, centre moved and values perturbed by the seed."""
    at = 4.0 + 2.0 * torch.rand(2, generator=torch.Generator().manual_seed(int(seed) + 5), dtype=torch.float64)
    dx, dy = x - float(at[0]), y - float(at[1])
    dx, dy = dx - 10.0 * torch.round(dx / 10.0), dy - 10.0 * torch.round(dy / 10.0)
    r2, beta = dx * dx + dy * dy, 5.0
    t = 1.0 - (GAMMA - 1.0) * beta ** 2 * torch.exp(1.0 - r2) / (8.0 * GAMMA * math.pi ** 2)
    f = beta / (2.0 * math.pi) * torch.exp(0.5 * (1.0 - r2))
    u, v = 0.3 * math.sqrt(GAMMA) - f * dy, f * dx
    rho = t ** (1.0 / (GAMMA - 1.0))
    U = torch.stack([rho, rho * u, rho * v, rho * t / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)], 1)
    return U * (1.0 + 1e-3 * _noise(U.shape, seed))


def _stream(x, y, seed):
    """The free stream past the cylinder, slowed to rest at its wall, perturbed by the seed."""
    u = torch.tanh(4.0 * (torch.hypot(x, y) - 0.5))
    one, none = torch.ones_like(u), torch.zeros_like(u)
    U = torch.stack([one, u, none, P_INF / (GAMMA - 1.0) + 0.5 * u * u], 1)
    return U * (1.0 + 1e-3 * _noise(U.shape, seed))


def _physics(c):
    """(parameters of the flow, start state, CFL number) of a case."""
    if "n" in c:
        return dict(mu=1e-3, C1=0.05 if c.get("theta") else 0.01, p_inf=1.0), _vortex, CFL
    return dict(mu=0.01, C1=0.05 if c.get("theta") else 0.01, p_inf=P_INF), _stream, CFL


def _viv(c):
    """Meshes, degrees and oscillators of a sweep."""
    out = []
    for i in range(c["cases"]):
        f = i / max(1, c["cases"] - 1)
        k = c["k_min"] + f * (c["k_max"] - c["k_min"])
        n_theta = 32 if k < 1000 else (64, 80, 96, 112, 128)[i % 5]
        p = c["p_min"] + i % (c["p_max"] - c["p_min"] + 1)
        fn = 1.0 / (3.0 + 5.0 * f)                               # U* from 3 to 8
        out.append(dict(n_theta=n_theta, n_r=max(2, int(round(k / (2 * n_theta)))), seed=i, p=p,
                        mu=1.0 / (100.0 + 50.0 * f), r1=8.0 if c["fixed"] else 30.0,
                        M_r=1.0, C_r=4.0 * math.pi * fn * 1e-3,
                        K_r=1.1 * (2.0 * math.pi * fn) ** 2, mass=10.0 * math.pi / 4.0, y0=0.05, ydot0=0.0,
                        # well inside the largest stable step
                        dt=1e-5 * (3.0 / p) ** 4 * (32.0 / n_theta) ** 2))
    return out


# ---- the calls ----------------------------------------------------------------

def _device_xy(xy):
    return (torch.from_numpy(xy[0]).to(DEV), torch.from_numpy(xy[1]).to(DEV))


def _mlp_data(c, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + 29)
    X = torch.randn((c["rows"], N_IN), generator=g, device=DEV)
    T = torch.tanh(X[:, :N_OUT] + 0.5 * X[:, N_OUT:2 * N_OUT]) + 0.1 * torch.randn((c["rows"], N_OUT), generator=g,
                                                                              device=DEV)
    return X, T, _mlp_start(seed)


def _mlp_start(seed):
    """Weights of a network in training: uniform as at creation, small biases."""
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + 31)
    parts = []
    for n, m in zip([N_IN] + DEPTH * [WIDTH], DEPTH * [WIDTH] + [N_OUT]):
        a = math.sqrt(6.0 / (n + m))
        parts += [a * (2.0 * torch.rand(n * m, generator=g, device=DEV) - 1.0),
                  0.01 * torch.randn(m, generator=g, device=DEV)]
    return torch.cat(parts)


def prepare(c, seed):
    kind = c["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind in ("mlp_train", "mlp_predict"):
        X, T, P = _mlp_data(c, seed)
        net = dg.Mlp(N_IN, WIDTH, DEPTH, N_OUT, max_batch=8192, seed=1)
        net.set_params(P)
        return dict(case=c, net=net, X=X, T=T, loss=torch.zeros(max(1, c.get("steps", 1)), device=DEV))
    if kind == "batch":
        viv = _viv(c)
        b = dg.BatchSolver([dict(mesh=_ogrid(v["n_theta"], v["n_r"], v["seed"], r1=v["r1"]),
                                 **{k: v[k] for k in ("p", "mu", "M_r", "C_r", "K_r", "mass", "y0", "ydot0")})
                            for v in viv], p_inf=P_INF)
        out = []
        for i in range(b.ncases):
            U = _stream(*_device_xy(b.node_coords(i)), seed + 100 * i)
            torch.cuda.current_stream().synchronize()
            b.set_state(i, U)
            out.append(torch.empty_like(U))
        if c["fixed"]:
            b.set_fixed_dt([v["dt"] for v in viv])
        return dict(case=c, b=b, out=out)
    phys, state, cfl = _physics(c)
    s = dg.Solver(_mesh(c), c["p"], c.get("precision", "mixed"), stream=stream, theta=c.get("theta", 0.0), **phys)
    U = state(*_device_xy(s.node_coords()), seed)
    s.set_state(U)
    got = dict(case=c, s=s, out=torch.empty_like(U))
    if kind == "gradient":
        got["gx"], got["gy"] = torch.empty_like(U), torch.empty_like(U)
    elif kind == "coupled":
        got.update(rigid=np.array([0.05, 0.0, 0.0]), vb=0.0, t=0.0, F=s.wall_forces())
    else:
        got["dt"] = s.dt(cfl)
        if c["host"]:
            got["host"] = U.cpu().pin_memory()
            got["out"] = torch.empty(U.shape, dtype=U.dtype, pin_memory=True)
    return got


_SPRING = (1.0, 4.0 * math.pi * 0.2 * 1e-3, 1.1 * (0.4 * math.pi) ** 2)
_MASS = 10.0 * math.pi / 4.0


def run(st):
    c = st["case"]
    kind = c["kind"]
    if kind == "mlp_predict":
        return st["net"].forward(st["X"])
    if kind == "mlp_train":
        loss = st["net"].train(st["X"], st["T"], c["steps"], 1e-3, out=st["loss"])
        return dict(loss=loss, params=st["net"].get_params())
    if kind == "batch":
        b = st["b"]
        b.run(CFL, c["steps"])
        for i, U in enumerate(st["out"]):
            dg.dg_batch_get_state(b.b, i, U)
        return dict(states=st["out"], rigid=b.rigid().astype(np.float32))
    s = st["s"]
    if kind == "gradient":
        dg.dg_broken_gradient(s.ctx, st["gx"], st["gy"], c["impl"])
        return st["gx"], st["gy"]
    if kind == "coupled":
        log = []
        for _ in range(c["steps"]):
            dt = s.dt(CFL, (0.0, st["vb"]))
            st["rigid"], st["vb"] = dg.dg_rigid_step(_SPRING, st["F"][1] / _MASS, dt, st["rigid"])
            s.step(st["t"], dt, (0.0, st["vb"]))
            st["t"] += dt
            st["F"] = s.wall_forces()
            log.append([st["t"], dt, *st["rigid"], st["vb"], *st["F"]])
        return dict(state=s.get_state(st["out"]), motion=np.array(log, dtype=np.float32))
    if c["host"]:
        s.set_state(st["host"])
    s.steps(0.0, st["dt"], c["steps"])
    return s.get_state(st["out"])


# ---- what a pass cannot do without -----------------------------------------------

def _stage_work(K, p):
    """Bytes and operations of one Runge-Kutta stage: every stage needs all of
    its neighbours' results of the stage before, so state and register (FP64)
    are read and written once per stage, with 80 bytes of geometry and
    connectivity per element; contractions, nodal fluxes, face fluxes, update."""
    n, f = (p + 1) * (p + 2) // 2, 3 * (p + 1)
    return 4 * K * n * 32 + 80 * K, K * (32 * n * n + 8 * n * f + 136 * n + 250 * f)


def work(c):
    kind = c["kind"]
    if kind in ("mlp_train", "mlp_predict"):
        weights = N_IN * WIDTH + (DEPTH - 1) * WIDTH * WIDTH + WIDTH * N_OUT
        if kind == "mlp_predict":
            return dict(bytes=4 * (weights + c["rows"] * (N_IN + N_OUT)), flops=2 * c["rows"] * weights)
        # each step: rows and targets read, weights and two moments read and written
        return dict(bytes=c["steps"] * 4 * (6 * weights + c["rows"] * (N_IN + N_OUT)),
                    flops=c["steps"] * 6 * c["rows"] * weights)
    if kind == "batch":
        each = [_stage_work(2 * v["n_theta"] * v["n_r"], v["p"]) for v in _viv(c)]
        return dict(bytes=5 * c["steps"] * sum(b for b, _ in each), flops=5 * c["steps"] * sum(f for _, f in each))
    p = c["p"]
    n = (p + 1) * (p + 2) // 2
    K = 2 * c["n"] ** 2 if "n" in c else 2 * c["n_theta"] * c["n_r"]
    if kind == "gradient":
        return dict(bytes=K * (4 * n * 24 + 32), flops=K * 4 * n * (4 * n + 6))
    b, f = _stage_work(K, p)
    return dict(bytes=5 * c["steps"] * b, flops=5 * c["steps"] * f)


# ---- the same in plain FP64 -------------------------------------------------------

def _jacobi(x, a, b, n):
    """Orthonormal Jacobi polynomial of degree n at x."""
    g0 = 2.0 ** (a + b + 1) / (a + b + 1) * math.gamma(a + 1) * math.gamma(b + 1) / math.gamma(a + b + 1)
    P = [np.full_like(x, 1.0 / math.sqrt(g0))]
    if n == 0:
        return P[0]
    g1 = (a + 1) * (b + 1) / (a + b + 3) * g0
    P.append(((a + b + 2) * x / 2 + (a - b) / 2) / math.sqrt(g1))
    old = 2.0 / (2 + a + b) * math.sqrt((a + 1) * (b + 1) / (a + b + 3))
    for i in range(1, n):
        h = 2 * i + a + b
        new = 2.0 / (h + 2) * math.sqrt((i + 1) * (i + 1 + a + b) * (i + 1 + a) * (i + 1 + b) / (h + 1) / (h + 3))
        mid = -(a * a - b * b) / h / (h + 2)
        P.append(((x - mid) * P[i] - old * P[i - 1]) / new)
        old = new
    return P[n]


def _jacobi_d(x, a, b, n):
    return np.zeros_like(x) if n == 0 else math.sqrt(n * (n + a + b + 1)) * _jacobi(x, a + 1, b + 1, n - 1)


class _Reference:
    """Nodes and operators of degree p on the triangle (-1,-1), (1,-1), (-1,1)."""

    def __init__(self, p):
        alpha = (0.0, 0.0, 1.4152, 0.1001, 0.2751, 0.9800)[p - 1]
        L1 = np.array([n / p for n in range(p + 1) for m in range(p + 1 - n)])
        L3 = np.array([m / p for n in range(p + 1) for m in range(p + 1 - n)])
        L2 = 1.0 - L1 - L3
        even = np.linspace(-1.0, 1.0, p + 1)
        inner = np.polynomial.legendre.Legendre.basis(p).deriv().roots()
        shift = np.concatenate([[-1.0], np.sort(inner.real), [1.0]]) - even
        x, y = L3 - L2, (2.0 * L1 - L2 - L3) / math.sqrt(3.0)
        for u, v, w, angle in ((L2, L3, L1, 0.0), (L3, L1, L2, 2 * math.pi / 3), (L1, L2, L3, 4 * math.pi / 3)):
            t = v - u
            warp = sum(shift[i] * np.prod([(t - even[j]) / (even[i] - even[j]) for j in range(p + 1) if j != i], axis=0)
                       for i in range(p + 1))
            inside = np.abs(t) < 1.0 - 1e-10
            warp = np.where(inside, warp / np.where(inside, 1.0 - t * t, 1.0), 0.0)
            move = 4.0 * u * v * warp * (1.0 + (alpha * w) ** 2)
            x, y = x + math.cos(angle) * move, y + math.sin(angle) * move
        B1, B2 = (math.sqrt(3.0) * y + 1.0) / 3.0, (2.0 - 3.0 * x - math.sqrt(3.0) * y) / 6.0
        B3 = 1.0 - B1 - B2
        r, s = B3 - B2 - B1, B1 - B2 - B3
        top = np.abs(1.0 - s) < 1e-12
        a = np.where(top, -1.0, 2.0 * (1.0 + r) / np.where(top, 1.0, 1.0 - s) - 1.0)
        V, Vr, Vs = [], [], []
        for i in range(p + 1):
            for j in range(p + 1 - i):
                fa, da = _jacobi(a, 0, 0, i), _jacobi_d(a, 0, 0, i)
                gb, db = _jacobi(s, 2 * i + 1, 0, j), _jacobi_d(s, 2 * i + 1, 0, j)
                half = 0.5 * (1.0 - s)
                low = half ** (i - 1) if i > 0 else np.ones_like(s)
                scale = 2.0 ** (i + 0.5)
                V.append(scale * fa * gb * half ** i)
                dr = da * gb * low
                ds = da * gb * 0.5 * (1.0 + a) * low + fa * (db * half ** i - (0.5 * i * gb * low if i else 0.0))
                Vr.append(scale * dr)
                Vs.append(scale * ds)
        V, Vr, Vs = (np.stack(v, 1) for v in (V, Vr, Vs))
        inv = np.linalg.inv(V)
        M = inv.T @ inv
        Dr, Ds = Vr @ inv, Vs @ inv
        faces = []
        for on, along in ((s + 1, r), (r + s, s), (r + 1, -s)):
            at = np.nonzero(np.abs(on) < 1e-7)[0]
            faces.append(at[np.argsort(along[at])])
        lift = np.zeros((len(r), 3 * (p + 1)))
        edge = np.sort(r[faces[0]])
        V1 = np.stack([_jacobi(edge, 0, 0, j) for j in range(p + 1)], 1)
        M1 = np.linalg.inv(V1 @ V1.T)
        for f in range(3):
            lift[faces[f], f * (p + 1):(f + 1) * (p + 1)] = M1
        put = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(DEV)  # noqa: E731
        self.p, self.r, self.s, self.Dr, self.Ds = p, put(r), put(s), put(Dr), put(Ds)
        self.LIFT, self.wface = put(np.linalg.solve(M, lift)), put(M1.sum(1))
        self.Wr, self.Ws = put(np.linalg.solve(M, Dr.T @ M)), put(np.linalg.solve(M, Ds.T @ M))
        self.fmask = torch.from_numpy(np.stack(faces)).to(DEV)


_A = (0.0, -567301805773 / 1357537059087, -2404267990393 / 2016746695238, -3550918686646 / 2091501179385,
      -1275806237668 / 842570457699)
_B = (1432997174477 / 9575080441755, 5161836677717 / 13612068292357, 1720146321549 / 2090206949498,
      3134564353537 / 4481467310338, 2277821191437 / 14882151754819)


class _Exact:
    """The discretisation on one mesh, in FP64, fields [K, 4, nodes]."""

    def __init__(self, mesh, p, mu, p_inf, C1=0.01, theta=0.0):
        self.ref = R = _Reference(p)
        self.p, self.mu, self.theta, self.sig = p, mu, theta, 3.0 * C1 * (1.0 + theta) ** 2
        put = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(DEV)  # noqa: E731
        vx, vy = put(mesh.vx)[put(mesh.EToV).long()], put(mesh.vy)[put(mesh.EToV).long()]
        self.x, self.y = (0.5 * (-(R.r + R.s) * v[:, :1] + (1 + R.r) * v[:, 1:2] + (1 + R.s) * v[:, 2:])
                          for v in (vx, vy))
        xr, xs, yr, ys = (0.5 * (v[:, i] - v[:, 0]) for v in (vx, vy) for i in (1, 2))
        self.J = J = xr * ys - xs * yr
        self.rx, self.ry, self.sx, self.sy = ((v / J)[:, None, None] for v in (ys, -xs, -yr, xr))
        ex, ey = torch.roll(vx, -1, 1) - vx, torch.roll(vy, -1, 1) - vy
        size = torch.hypot(ex, ey)
        self.n1, self.n2 = (ey / size)[:, None, :, None], (-ex / size)[:, None, :, None]
        self.sJ, self.fs = 0.5 * size, 0.5 * size / J[:, None]
        self.nb, self.nf, self.bc = (put(v).long() for v in (mesh.EToE, mesh.EToF, mesh.bc))
        self.vm = R.fmask                                            # [3, Nfp]
        self.vp = R.fmask[self.nf].flip(-1)                          # [K, 3, Nfp]
        self.wall, self.far = (self.bc == 1)[:, None, :, None], (self.bc == 2)[:, None, :, None]
        e = p_inf / (GAMMA - 1.0) + 0.5
        self.uinf = torch.tensor([1.0, 1.0, 0.0, e], dtype=torch.float64, device=DEV)[None, :, None, None]

    @staticmethod
    def pressure(U):
        return (GAMMA - 1.0) * (U[:, 3] - 0.5 * (U[:, 1] ** 2 + U[:, 2] ** 2) / U[:, 0])

    def grad(self, U):
        ur, us = U @ self.ref.Dr.T, U @ self.ref.Ds.T
        return self.rx * ur + self.sx * us, self.ry * ur + self.sy * us

    def viscous(self, U, gx, gy, adiabatic=None):
        """G(U) grad U; `adiabatic`: where the heat flux is left out."""
        r, v1, v2, e = U[:, 0], U[:, 1] / U[:, 0], U[:, 2] / U[:, 0], U[:, 3] / U[:, 0]
        ax, ay, bx, by = ((g[:, i] - v * g[:, 0]) / r for i, v in ((1, v1), (2, v2)) for g in (gx, gy))
        qx, qy = ((g[:, 3] - e * g[:, 0]) / r - v1 * a - v2 * b for g, a, b in ((gx, ax, bx), (gy, ay, by)))
        k = self.mu * GAMMA / PRANDTL
        k = k if adiabatic is None else k * (~adiabatic).double()
        xx, yy, xy = self.mu * (4 * ax - 2 * by) / 3, self.mu * (4 * by - 2 * ax) / 3, self.mu * (ay + bx)
        o = torch.zeros_like(xx)
        return (torch.stack([o, xx, xy, v1 * xx + v2 * xy + k * qx], 1),
                torch.stack([o, xy, yy, v1 * xy + v2 * yy + k * qy], 1))

    def advective(self, U, vw):
        P = self.pressure(U)
        v1, v2, o = U[:, 1] / U[:, 0], U[:, 2] / U[:, 0], torch.zeros_like(P)
        return (U * (v1 - vw[0])[:, None] + torch.stack([o, P, o, P * v1], 1),
                U * (v2 - vw[1])[:, None] + torch.stack([o, o, P, P * v2], 1))

    def norm(self, U):
        """Spectral norm of n1^2 G11 + n1 n2 (G12 + G21) + n2^2 G22 at face nodes."""
        cols = []
        for k in range(4):
            unit = torch.zeros_like(U)
            unit[:, k] = 1.0
            Fx, Fy = self.viscous(U, self.n1 * unit, self.n2 * unit)
            cols.append(self.n1 * Fx + self.n2 * Fy)
        N = torch.stack(cols, -1).movedim(1, -2)                     # [K, 3, Nfp, row, column]
        A = N.transpose(-1, -2) @ N
        P = A / (A.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None] + 1e-300)
        for _ in range(36):                                          # squared up to the leading projector
            P = P @ P
            P = P / P.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None]
        return torch.sqrt((A * P).sum((-1, -2)))

    def traces(self, U, vw):
        """Own and outer traces [K, 4, 3, Nfp], the outer one a ghost on boundaries."""
        up = U[:, :, self.vm]
        um = U[self.nb[:, :, None], :, self.vp].permute(0, 3, 1, 2)
        w = torch.stack([up[:, 0], up[:, 0] * vw[0], up[:, 0] * vw[1],
                         self.pressure(up) / (GAMMA - 1.0) + 0.5 * up[:, 0] * (vw[0] ** 2 + vw[1] ** 2)], 1)
        return up, torch.where(self.wall, w, torch.where(self.far, self.uinf, um))

    def penalty(self, up, um):
        g = torch.maximum(self.norm(up), self.norm(um)).amax(-1)
        c = 0.5 * (self.p + 1) * (self.p + 2)
        fs = torch.where(self.bc == 0, torch.maximum(self.fs, self.fs[self.nb, self.nf]), self.fs)
        return self.sig * g * c * fs                                 # [K, 3]

    def roe(self, up, um, vw):
        n1, n2 = self.n1[:, 0], self.n2[:, 0]
        pp, pm = self.pressure(up), self.pressure(um)
        a, b = torch.sqrt(up[:, 0]), torch.sqrt(um[:, 0])
        mean = lambda p, m: (a * p + b * m) / (a + b)  # noqa: E731
        v1, v2 = mean(up[:, 1] / up[:, 0], um[:, 1] / um[:, 0]), mean(up[:, 2] / up[:, 0], um[:, 2] / um[:, 0])
        H = mean((up[:, 3] + pp) / up[:, 0], (um[:, 3] + pm) / um[:, 0])
        q = 0.5 * (v1 * v1 + v2 * v2)
        c = torch.sqrt((GAMMA - 1.0) * (H - q))
        vn, vt, rt = v1 * n1 + v2 * n2, v2 * n1 - v1 * n2, a * b
        d1, d2 = up[:, 1] / up[:, 0] - um[:, 1] / um[:, 0], up[:, 2] / up[:, 0] - um[:, 2] / um[:, 0]
        dn, dt, dp, dr = d1 * n1 + d2 * n2, d2 * n1 - d1 * n2, pp - pm, up[:, 0] - um[:, 0]
        w = vn - vw[0] * n1 - vw[1] * n2
        k1 = torch.abs(w - c) * 0.5 * (dp - rt * c * dn) / c ** 2
        k4 = torch.abs(w + c) * 0.5 * (dp + rt * c * dn) / c ** 2
        k2, k3 = torch.abs(w) * (dr - dp / c ** 2), torch.abs(w) * rt * dt
        return torch.stack([k1 + k2 + k4, k1 * (v1 - c * n1) + k2 * v1 - k3 * n2 + k4 * (v1 + c * n1),
                            k1 * (v2 - c * n2) + k2 * v2 + k3 * n1 + k4 * (v2 + c * n2),
                            k1 * (H - c * vn) + k2 * q + k3 * vt + k4 * (H + c * vn)], 1)

    def rhs(self, U, vw):
        R, n1, n2 = self.ref, self.n1, self.n2
        gx, gy = self.grad(U)
        (cx, cy), (vx, vy) = self.advective(U, vw), self.viscous(U, gx, gy)
        Fx, Fy = cx - vx, cy - vy
        out = -((self.rx * Fx + self.ry * Fy) @ R.Dr.T + (self.sx * Fx + self.sy * Fy) @ R.Ds.T)
        up, um = self.traces(U, vw)
        at = lambda g: g[self.nb[:, :, None], :, self.vp].permute(0, 3, 1, 2)  # noqa: E731
        gxp, gyp = gx[:, :, self.vm], gy[:, :, self.vm]
        edge = self.wall | self.far
        gxm, gym = torch.where(edge, gxp, at(gx)), torch.where(edge, gyp, at(gy))
        normal = lambda F: n1 * F[0] + n2 * F[1]  # noqa: E731
        cp, cm = normal(self.advective(up, vw)), normal(self.advective(um, vw))
        dp = normal(self.viscous(up, gxp, gyp))
        far_d = dp                                                   # the far field takes G(U+) grad U+
        wall_d = normal(self.viscous(um, gxm, gym, adiabatic=self.wall[:, 0]))
        in_d = 0.5 * (dp + wall_d)
        d = torch.where(self.wall, wall_d, torch.where(self.far, far_d, in_d))
        c = torch.where(self.wall, cm, 0.5 * (cp + cm) + 0.5 * self.roe(up, um, vw))
        jump = up - um
        H = c - d + self.penalty(up, um)[:, None, :, None] * jump
        flat = lambda v: (self.fs[:, None, :, None] * v).reshape(v.shape[0], 4, -1) @ R.LIFT.T  # noqa: E731
        out += flat(cp - dp - H)
        if self.theta:
            base = torch.where(self.wall, um, up)
            w = self.theta * (0.5 + 0.5 * edge.double())
            t = []
            for o in (0, 1):
                rows = []
                for k in range(4):
                    unit, none = torch.zeros_like(up), torch.zeros_like(up)
                    unit[:, k] = 1.0
                    F = normal(self.viscous(base, unit if o == 0 else none, none if o == 0 else unit))
                    rows.append((jump * F).sum(1))
                t.append(flat(w * torch.stack(rows, 1)))
            out += (self.rx * t[0] + self.ry * t[1]) @ R.Wr.T + (self.sx * t[0] + self.sy * t[1]) @ R.Ws.T
        return out

    def step(self, U, dt, vw=(0.0, 0.0)):
        K1 = torch.zeros_like(U)
        for a, b in zip(_A, _B):
            K1 = a * K1 + dt * self.rhs(U, vw)
            U = U + b * K1
        return U

    def dt(self, U, cfl, vw=(0.0, 0.0)):
        up, um = self.traces(U, vw)
        low = torch.minimum(up[:, 0], um[:, 0]).amin((-1, -2))
        G = max(4.0 / 3.0, GAMMA / PRANDTL) * self.mu / low
        c = torch.sqrt(GAMMA * self.pressure(U) / U[:, 0])
        beta = torch.hypot(torch.abs(U[:, 1] / U[:, 0] - vw[0]) + c, torch.abs(U[:, 2] / U[:, 0] - vw[1]) + c).amax(-1)
        rho = 2.0 * 2.0 * self.J / (2.0 * self.sJ).sum(1)
        ci = 0.5 * (self.p + 1) * (self.p + 2) * self.fs.amax(1)
        lam = 1.5 * self.p ** 4 / rho ** 2 * G + 3.0 * ci * (3.0 * self.penalty(up, um).amax(1) + beta)
        return cfl / float(lam.max())

    def forces(self, U):
        gx, gy = self.grad(U)
        Fx, Fy = self.viscous(U, gx, gy)
        P, vm = self.pressure(U)[:, self.vm], self.vm
        n1, n2 = self.n1[:, 0], self.n2[:, 0]
        tx = P * n1 - (Fx[:, 1][:, vm] * n1 + Fy[:, 1][:, vm] * n2)
        ty = P * n2 - (Fx[:, 2][:, vm] * n1 + Fy[:, 2][:, vm] * n2)
        w = (self.sJ[:, :, None] * self.ref.wface) * (self.bc == 1)[:, :, None]
        x, y = self.x[:, vm], self.y[:, vm]
        return [float((w * v).sum()) for v in (tx, ty, x * ty - y * tx)]


def _newmark(spring, F, dt, state):
    M, C, K = spring
    y, v, a = state
    ys, vs = y + dt * v + 0.25 * dt * dt * a, v + 0.5 * dt * a
    a = (F - C * vs - K * ys) / (M + 0.5 * dt * C + 0.25 * dt * dt * K)
    new = (ys + 0.25 * dt * dt * a, vs + 0.5 * dt * a, a)
    return new, (new[0] - y) / dt


def _exact_mlp(c, seed):
    X, T, P = _mlp_data(c, seed)
    X, T, P = X.double(), T.double(), P.double()

    def net(q):
        h, at = X, 0
        for k, (n, m) in enumerate(zip([N_IN] + DEPTH * [WIDTH], DEPTH * [WIDTH] + [N_OUT])):
            z = h @ q[at:at + n * m].reshape(m, n).T + q[at + n * m:at + n * m + m]
            h, at = (torch.nn.functional.gelu(z) if k < DEPTH else z), at + n * m + m
        return h

    if c["kind"] == "mlp_predict":
        return net(P)
    m, v, losses = torch.zeros_like(P), torch.zeros_like(P), []
    for k in range(1, c["steps"] + 1):
        q = P.clone().requires_grad_(True)
        loss = ((net(q) - T) ** 2).mean()
        g, = torch.autograd.grad(loss, q)
        losses.append(loss.detach())
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        P = P - 1e-3 * (m / (1 - 0.9 ** k)) / (torch.sqrt(v / (1 - 0.999 ** k)) + 1e-8)
    return dict(loss=torch.stack(losses), params=P)


def exact(c, seed):
    kind = c["kind"]
    if kind in ("mlp_train", "mlp_predict"):
        return _exact_mlp(c, seed)
    if kind == "batch":
        states, rigid = [], []
        for i, v in enumerate(_viv(c)):
            E = _Exact(_ogrid(v["n_theta"], v["n_r"], v["seed"], r1=v["r1"]), v["p"], v["mu"], P_INF)
            U = _stream(E.x, E.y, seed + 100 * i)
            q, vb, t, F = (v["y0"], v["ydot0"], 0.0), 0.0, 0.0, E.forces(U)
            for _ in range(c["steps"]):
                dt = v["dt"] if c["fixed"] else E.dt(U, CFL, (0.0, vb))
                q, vb = _newmark((v["M_r"], v["C_r"], v["K_r"]), F[1] / v["mass"], dt, q)
                U, t = E.step(U, dt, (0.0, vb)), t + dt
                F = E.forces(U)
            states.append(U)
            rigid.append([t, dt, *q, vb, *F, 0.0])
        return dict(states=states, rigid=np.array(rigid))
    phys, state, cfl = _physics(c)
    E = _Exact(_mesh(c), c["p"], phys["mu"], phys["p_inf"], phys["C1"], c.get("theta", 0.0))
    U = state(E.x, E.y, seed)
    if kind == "gradient":
        return E.grad(U)
    if kind == "coupled":
        q, vb, t, F, log = (0.05, 0.0, 0.0), 0.0, 0.0, E.forces(U), []
        for _ in range(c["steps"]):
            dt = E.dt(U, CFL, (0.0, vb))
            q, vb = _newmark(_SPRING, F[1] / _MASS, dt, q)
            U, t = E.step(U, dt, (0.0, vb)), t + dt
            F = E.forces(U)
            log.append([t, dt, *q, vb, *F])
        return dict(state=U, motion=np.array(log))
    dt = E.dt(U, cfl)
    for _ in range(c["steps"]):
        U = E.step(U, dt)
    return U
