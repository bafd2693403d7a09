"""What this framework is timed on: its public calls at the sizes they are used with.

Every case is one call (or one short sequence of calls) of ``paper_1307_7867_gb300.heat3d``,
the ABI's binding: the spatial operator, one multigrid solve, one SDC sweep of resident items,
serial SDC, two-level MLSDC and PFASST over their steps, and the serving loop.  Grids are the
2^k - 1 ones that multigrid takes; stencils, node counts, step lengths, tolerances and the
interpolation of the coarse correction are those of the repository's benchmark and tests.

Inputs: sums of eight sine modes with normal amplitudes (what the tests, the serving stream and
the paper's initial value are made of; MLSDC and PFASST start from low modes, as the paper does),
for solves with a rough part on top, as the collocation
right-hand sides of a sweep have.
"""
import math

import numpy as np
import torch

from paper_1307_7867_gb300 import heat3d as H
from paper_1307_7867_gb300 import inputs

PI = math.pi
NU = 0.1


def listed():
    return [
        # the operator alone on a small grid: two copies and one stencil, all latency
        dict(name="operator_31_wide", kind="operator", N=31, order=4),
        # the operator at the paper's fine size, compact stencil (the paper's own)
        dict(name="operator_255_compact", kind="operator", N=255, order=19),
        # one implicit solve of the smallest production size (31^3, 7 points)
        dict(name="solve_31_fp64", kind="solve", N=31, order=2, precision=0, c=6.25e-3, graphs=0),
        # a 63^3 solve in mixed precision, the coarse levels of 127^3 hierarchies
        dict(name="solve_63_mixed", kind="solve", N=63, order=4, precision=1, c=2e-3, graphs=1),
        # a solve at the headline size, every field FP64
        dict(name="solve_255_wide_fp64", kind="solve", N=255, order=4, precision=0, c=5e-4, graphs=1),
        # one sweep of four resident items (a small serving batch), compact stencil
        dict(name="sweep_127_compact_x4", kind="sweep", N=127, order=19, M=5, precision=0, items=4,
             dt=1 / 32, graphs=1),
        # serial SDC of small problems: 31^3, 7 points, 3 nodes, dt = 1/8, 4 sweeps, FP64
        dict(name="sdc_31_fp64", kind="sdc", N=31, order=2, M=3, precision=0, dt=1 / 8, steps=2,
             sweeps=4, graphs=1),
        # the benchmark's MLSDC step (255^3 wide over 127^3, dt = 1/64, to 1e-10), FP64, with the
        # 8-point interpolation of the coarse correction
        dict(name="mlsdc_255_fp64", kind="mlsdc", N=255, order=4, M=5, precision=0, dt=1 / 64,
             slices=1, interp=8, rel=0.0, kmax=2, graphs=1),
        # the same step in mixed precision with trilinear interpolation and the adaptive solver
        # tolerance: many iterations of few V-cycles
        dict(name="mlsdc_255_mixed_trilinear", kind="mlsdc", N=255, order=4, M=5, precision=1,
             dt=1 / 64, slices=1, interp=2, rel=0.02, kmax=2, graphs=1),
        # one sweep at the largest fine grid of the benchmark, 511^3, mixed precision
        dict(name="sweep_511_mixed", kind="sweep", N=511, order=4, M=5, precision=1, items=1, dt=1 / 32,
             graphs=1),
        # PFASST: four time slices in one batch, the paper's compact fine stencil, mixed
        dict(name="pfasst_4x127_mixed", kind="mlsdc", N=127, order=19, M=5, precision=1, dt=1 / 16,
             slices=4, interp=8, rel=0.0, kmax=2, graphs=1),
        # the serving loop: twelve requests of three sizes at once, results on the host
        dict(name="serve_12", kind="serve", requests=12, Nmax=127, precision=1, dt=1 / 32, steps=4),
    ]


def draw(rng):
    """One more case: any kind at any size, stencil, precision and option of its range."""
    kind = rng.choice(["operator", "solve", "solve", "sweep", "sdc", "mlsdc", "mlsdc", "pfasst"])
    prec = rng.randrange(2)
    dt = 2.0 ** rng.uniform(-6, -4.5)
    if kind == "operator":
        # one of the sizes over the whole range, batches being one item here
        return dict(kind="operator", N=2 ** rng.randint(2, 9) - 1, order=rng.choice([2, 4, 19]),
                    nu=round(rng.uniform(0.05, 0.2), 4))
    if kind == "solve":
        return dict(kind="solve", N=2 ** rng.randint(4, 9) - 1, order=rng.choice([2, 4, 19]),
                    precision=prec, c=10.0 ** rng.uniform(-3.5, -2), graphs=rng.randrange(2))
    if kind == "sweep":
        N = 2 ** rng.randint(4, 8) - 1
        return dict(kind="sweep", N=N, order=rng.choice([2, 4, 19]), M=rng.randint(2, 5), precision=prec,
                    items=rng.randint(1, 2 if N > 127 else 5), dt=dt, graphs=rng.randrange(2))
    if kind == "sdc":
        return dict(kind="sdc", N=2 ** rng.randint(4, 7) - 1, order=rng.choice([2, 4]), M=rng.randint(2, 5),
                    precision=prec, dt=dt, steps=rng.randint(1, 3), sweeps=rng.randint(3, 5), graphs=1)
    order = rng.choice([4, 19])
    if kind == "mlsdc":
        N = 2 ** rng.randint(5, 8) - 1
        return dict(kind="mlsdc", N=N, order=order, M=5, precision=prec, dt=dt, slices=1,
                    interp=8 if N > 127 else rng.choice([4, 6, 8]), rel=rng.choice([0.0, 0.02]), kmax=rng.randint(1, 3), graphs=1)
    N = 2 ** rng.randint(5, 7) - 1
    return dict(kind="mlsdc", N=N, order=order, M=5, precision=prec, dt=dt,
                slices=rng.randint(2, 3 if N > 63 else 6), interp=8, rel=0.0, kmax=rng.randint(1, 2), graphs=1)


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------


def _modes(rng, n=8, kmax=8):
    return [(tuple(int(k) for k in rng.integers(1, kmax + 1, size=3)), float(rng.standard_normal()))
            for _ in range(n)]


def _field(N, modes):
    x = torch.arange(1, N + 1, dtype=torch.float64, device="cuda") / (N + 1)
    u = torch.zeros(N, N, N, dtype=torch.float64, device="cuda")
    for (k1, k2, k3), a in modes:
        u += (a * torch.sin(k3 * PI * x))[:, None, None] * torch.sin(k2 * PI * x)[None, :, None] * \
            torch.sin(k1 * PI * x)[None, None, :]
    return u


def _smooth(case, seed, item=0):
    return _field(case["N"], _modes(np.random.default_rng([seed, item]), kmax=case.get("kmax", 8)))


def _rhs_and_start(case, seed):
    """Right-hand side (modes plus a rough part) and warm start (the modes damped) of a solve."""
    u = _smooth(case, seed)
    g = torch.Generator(device="cuda").manual_seed(seed)
    rough = torch.rand(u.shape, generator=g, dtype=torch.float64, device="cuda") - 0.5
    return u + 0.05 * rough, 0.9 * u


def _requests(case, seed):
    """The serving stream's requests at one horizon: sizes in turn, nu and modes drawn."""
    sizes = [n for n in (31, 63, 127, 255) if n <= case["Nmax"]]
    out = []
    for i in range(case["requests"]):
        rng = np.random.default_rng([seed, i])
        modes = [(*k, a) for k, a in _modes(rng)]
        out.append(inputs.Request(i, 0.0, sizes[i % len(sizes)], float(rng.uniform(0.05, 0.2)),
                                  case["steps"] * case["dt"], case["dt"], modes))
    return out


# ---------------------------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------------------------


def _config(case):
    k = case["kind"]
    common = dict(nu=case.get("nu", NU), mg_tol=1e-10 if k in ("operator", "solve", "sdc") else 1e-11,
                  precision=case.get("precision", 0), use_graphs=case.get("graphs", 0),
                  inner=0 if case.get("precision") else 1)
    if k in ("operator", "solve"):
        return H.make_config((case["N"], case["order"], 2), None, **common)
    if k == "sweep":
        return H.make_config((case["N"], case["order"], case["M"]), None, dt=case["dt"],
                             batch=case["items"], **common)
    if k == "sdc":
        return H.make_config((case["N"], case["order"], case["M"]), None, dt=case["dt"],
                             T=case["steps"] * case["dt"], sweeps_fine=case["sweeps"], tol_sdc=-1.0, **common)
    return H.make_config((case["N"], case["order"], case["M"]), ((case["N"] - 1) // 2, 2, 3), dt=case["dt"],
                         T=case["slices"] * case["dt"], slices=case["slices"], batch=case["slices"],
                         sweeps_fine=2, sweeps_coarse=1, iters=50, tol_sdc=1e-10, interp=case["interp"],
                         mg_rel=case["rel"], **common)


def prepare(case, seed):
    s = {"case": case}
    k = case["kind"]
    if k == "serve":
        s["requests"] = _requests(case, seed)
        s["pool"] = torch.empty(6 << 30, dtype=torch.uint8, device="cuda")
        s["server"] = H.Server(s["pool"], max_active=4, sweeps=4, precision=case["precision"], mg_tol=1e-10,
                               inner=0)
        torch.cuda.synchronize()
        # the server keeps its groups (one per grid size) from the first request on
        first = {r.N: r for r in s["requests"]}.values()
        for t in [s["server"].submit(r) for r in first]:
            s["server"].wait(t)
        return s
    if k == "solve":
        s["rhs"], s["u0"] = _rhs_and_start(case, seed)
        s["u"] = torch.empty_like(s["u0"])
    elif k == "sweep":
        s["u0"] = [_smooth(case, seed, b) for b in range(case["items"])]
        s["out"] = [[torch.empty_like(u) for _ in range(case["M"] - 1)] for u in s["u0"]]
    else:
        s["u0"] = _smooth(case, seed)
        s["out"] = torch.empty_like(s["u0"])
    stream = torch.cuda.Stream() if case.get("graphs") else None
    torch.cuda.synchronize()
    s["ctx"] = H.Context(_config(case), stream=stream)
    return s


def run(s):
    case = s["case"]
    k = case["kind"]
    if k == "operator":
        H.heat3d_apply_laplacian(s["ctx"], 0, s["u0"], s["out"])
        return s["out"]
    if k == "solve":
        with torch.cuda.stream(s["ctx"].stream):
            s["u"].copy_(s["u0"])
        H.mg_vcycle(s["ctx"], 0, case["c"], s["rhs"], s["u"], 50, 1e-10)
        return s["u"]
    if k == "sweep":
        for b, u in enumerate(s["u0"]):
            H.heat3d_set_state(s["ctx"], 0, b, 0.25 * b, u)
        H.sdc_sweep(s["ctx"], 0, 0, case["items"])
        for b, nodes in enumerate(s["out"]):
            for m, o in enumerate(nodes):
                H.heat3d_get_node(s["ctx"], 0, b, m + 1, o)
        return s["out"]
    if k == "serve":
        tickets = [s["server"].submit(r) for r in s["requests"]]
        return [s["server"].wait(t)[0] for t in tickets]
    H.pfasst_run(s["ctx"], s["u0"], s["out"])
    return s["out"]


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------


def work(case):
    """Inputs read and results written once; operations of the stencil, and for solves of six
    V(2,1) cycles (a tenth per cycle brings a residual of order one to the tolerance's order)
    with one residual each, of which a point takes about six stencils over all levels."""
    k = case["kind"]
    if k == "serve":
        sizes = [r.N ** 3 for r in _requests(case, 0)]
        pts, solves = sum(sizes), case["steps"] * 4 * 2
        return {"bytes": 8.0 * pts, "flops": pts * solves * 3.0 * 6 * 9}
    pts = case["N"] ** 3
    fl = {2: 9.0, 4: 16.0, 19: 22.0}[case["order"]]
    if k == "operator":
        return {"bytes": 16.0 * pts, "flops": fl * pts}
    cycle = 6 * fl * pts
    if k == "solve":
        return {"bytes": 24.0 * pts, "flops": 6 * cycle}
    M = case["M"]
    if k == "sweep":
        return {"bytes": 8.0 * M * pts * case["items"],
                "flops": case["items"] * ((M - 1) * 5 * cycle + pts * 2.0 * M * (M - 1))}
    steps, sweeps = (case["steps"], case["sweeps"]) if k == "sdc" else (case["slices"], 4)
    return {"bytes": 16.0 * pts, "flops": steps * sweeps * ((M - 1) * 3 * cycle + pts * 2.0 * M * (M - 1))}


# ---------------------------------------------------------------------------------------------
# the results in 64 bits: every operator here is diagonal in the sine basis
# ---------------------------------------------------------------------------------------------


def _sines(N):
    i = torch.arange(1, N + 1, dtype=torch.float64, device="cuda")
    # reduce j k modulo the period before the sine, for accuracy at high modes
    return torch.sin(PI * torch.remainder(torch.outer(i, i), 2 * (N + 1)) / (N + 1))


def _transform(u, S):
    u = torch.matmul(u, S)
    u = torch.matmul(S, u)
    return torch.matmul(S, u.reshape(u.shape[0], -1)).reshape(u.shape)


def _to_modes(u):
    return _transform(u, _sines(u.shape[0])) * (2.0 / (u.shape[0] + 1)) ** 3


def _from_modes(a):
    return _transform(a, _sines(a.shape[0]))


def _symbols(N, order):
    """Eigenvalues of the Laplacian (compact: L and the weighting matrix W) on the sine modes."""
    h = 1.0 / (N + 1)
    c = torch.cos(PI * h * torch.arange(1, N + 1, dtype=torch.float64, device="cuda"))
    a, b, d = c[:, None, None], c[None, :, None], c[None, None, :]
    one = torch.ones(N, N, N, dtype=torch.float64, device="cuda")
    if order == 2:
        return (2.0 * (a + b + d) - 6.0) / h ** 2, one
    if order == 4:
        w = (32.0 * c - 2.0 * (2.0 * c * c - 1.0) - 30.0) / (12.0 * h * h)
        return w[:, None, None] + w[None, :, None] + w[None, None, :], one
    lap = (-24.0 + 4.0 * (a + b + d) + 4.0 * (a * b + a * d + b * d)) / (6.0 * h * h)
    return lap, (6.0 + 2.0 * (a + b + d)) / 12.0


def _collocation(M):
    """Gauss-Lobatto nodes on [0, 1] and Q[m][j] = int_0^{tau_m} l_j."""
    P = np.polynomial.legendre.Legendre.basis(M - 1)
    tau = (np.concatenate([[-1.0], np.sort(np.real(P.deriv().roots())) if M > 2 else [], [1.0]]) + 1) / 2
    Q = np.zeros((M, M))
    for j in range(M):
        p = np.poly1d([1.0])
        for i in range(M):
            if i != j:
                p = p * np.poly1d([1.0, -tau[i]]) / (tau[j] - tau[i])
        q = p.integ()
        Q[:, j] = q(tau) - q(0.0)
    return tau, Q


def _forcing(t, nu):
    """Eq. 3 as printed, the amplitude of the first sine mode."""
    return -(math.sin(t) - nu * PI * PI * math.cos(t))


def _sdc(a0, lam, W, t0, dt, M, sweeps, nu=NU, forced=True):
    """SDC sweeps from the spread initial value, mode by mode: the values at the nodes."""
    tau, Q = _collocation(M)
    S = Q[1:] - Q[:-1]
    U = [a0.clone() for _ in range(M)]
    for _ in range(sweeps):
        F = [lam * u for u in U]
        for m in range(M - 1):
            dtm = dt * (tau[m + 1] - tau[m])
            r = W * U[m] - dtm * F[m + 1]
            for j in range(M):
                r = r + dt * S[m, j] * F[j]
            if forced:
                g = sum(dt * S[m, j] * _forcing(t0 + dt * tau[j], nu) for j in range(M))
                r[0, 0, 0] += g * W[0, 0, 0]
            U[m + 1] = r / (W - dtm * lam)
    return U


def _converged(a0, lam, W, t0, dt, M, nu=NU):
    """The collocation solution at the end of one step: (W - dt Q lam) U = W U_0 + dt Q W f."""
    tau, Q = _collocation(M)
    n = M - 1
    A = [[(W if i == j else 0.0) - dt * Q[i + 1, j + 1] * lam for j in range(n)] for i in range(n)]
    r = [W * a0 + dt * Q[i + 1, 0] * lam * a0 for i in range(n)]
    for i in range(n):
        g = sum(dt * Q[i + 1, j] * _forcing(t0 + dt * tau[j], nu) for j in range(M))
        r[i][0, 0, 0] += g * W[0, 0, 0]
    for i in range(n):  # elimination; the diagonal dominates for lam <= 0
        for k in range(i + 1, n):
            f = A[k][i] / A[i][i]
            for j in range(i + 1, n):
                A[k][j] = A[k][j] - f * A[i][j]
            r[k] = r[k] - f * r[i]
    x = [None] * n
    for i in reversed(range(n)):
        v = r[i]
        for j in range(i + 1, n):
            v = v - A[i][j] * x[j]
        x[i] = v / A[i][i]
    return x[-1]


def exact(case, seed):
    k = case["kind"]
    if k == "serve":
        out = []
        for r in _requests(case, seed):
            lap, W = _symbols(r.N, 2)
            a = _to_modes(_field(r.N, [((k1, k2, k3), amp) for k1, k2, k3, amp in r.modes]))
            for _ in range(case["steps"]):
                a = _sdc(a, r.nu * lap, W, 0.0, r.dt, 3, 4, forced=False)[-1]
            out.append(_from_modes(a).cpu().numpy())
        return out
    lap, W = _symbols(case["N"], case["order"])
    if k == "operator":
        return _from_modes(case.get("nu", NU) * lap * _to_modes(_smooth(case, seed)))
    if k == "solve":
        rhs, _ = _rhs_and_start(case, seed)
        return _from_modes(_to_modes(rhs) / (W - case["c"] * lap))
    lam = NU * lap
    if k == "sweep":
        return [[_from_modes(v) for v in _sdc(_to_modes(_smooth(case, seed, b)), lam, W, 0.25 * b, case["dt"],
                                              case["M"], 1)[1:]] for b in range(case["items"])]
    a = _to_modes(_smooth(case, seed))
    for n in range(case["steps"] if k == "sdc" else case["slices"]):
        if k == "sdc":
            a = _sdc(a, lam, W, n * case["dt"], case["dt"], case["M"], case["sweeps"])[-1]
        else:
            a = _converged(a, lam, W, n * case["dt"], case["dt"], case["M"])
    return _from_modes(a)
