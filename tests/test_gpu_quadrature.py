"""GPU test of the fixed-point quadrature kernel (k_integrals): the collocation
residual of random node fields against the same sums in plain torch FP64.

Tolerance: the residual is max |U_0 + sum_j (dt Q[m][j] F_j + ...) - U_m|; both
sides round each of at most seven terms, so 16 x 2^-53 times the largest term
bounds the difference (the sums of the two sides are each off by less than
eight roundings)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1307_7867_gb300 import build, heat3d
    build.build()
    heat3d.load()
    return heat3d


def collocation(M):
    P = np.polynomial.legendre.Legendre.basis(M - 1)
    inner = np.sort(np.real(P.deriv().roots())) if M > 2 else []
    tau = (np.concatenate([[-1.0], inner, [1.0]]) + 1) / 2
    Q = np.zeros((M, M))
    for j in range(M):
        p = np.poly1d([1.0])
        for i in range(M):
            if i != j:
                p = p * np.poly1d([1.0, -tau[i]]) / (tau[j] - tau[i])
        q = p.integ()
        Q[:, j] = q(tau) - q(0.0)
    return tau, Q


@pytest.mark.parametrize("M", [2, 3, 4, 5])
@pytest.mark.parametrize("N,forcing,scale", [(31, 1, 1.0), (63, 0, 1e-9), (127, 1, 1.0), (255, 0, 1.0),
                                             (31, 0, 1e200), (31, 0, 1e-200)])
def test_residual_matches_plain_fp64(H, M, N, forcing, scale):
    dt, t0, nu = 1 / 16, 0.3, 0.1
    ctx = H.Context(H.make_config((N, 2, M), None, dt=dt, nu=nu, forcing=forcing))
    rng = torch.Generator(device="cuda").manual_seed(5)
    u = [scale * (torch.rand(N, N, N, generator=rng, dtype=torch.float64, device="cuda") - 0.5) for _ in range(M)]
    u[0][: N // 2] = 0.0  # points where every node is zero in u_0
    H.heat3d_set_state(ctx, 0, 0, t0, u[0])
    for m in range(1, M):
        H.heat3d_set_node(ctx, 0, 0, m, u[m])
    got = H.heat3d_sdc_residual(ctx, 0, 0)
    F = []
    for v in u:
        F.append(torch.empty_like(v))
        H.heat3d_apply_laplacian(ctx, 0, v, F[-1])
    tau, Q = collocation(M)
    x = torch.arange(1, N + 1, dtype=torch.float64, device="cuda") / (N + 1)
    s = torch.sin(np.pi * x)
    phi = s[:, None, None] * s[None, :, None] * s[None, None, :]
    g = [-(np.sin(t0 + dt * t) - nu * np.pi ** 2 * np.cos(t0 + dt * t)) if forcing else 0.0 for t in tau]
    want, term = 0.0, float(u[0].abs().max())
    for m in range(1, M):
        r = u[0] - u[m] + phi * float(sum(dt * Q[m, j] * g[j] for j in range(M)))
        for j in range(M):
            r = r + dt * Q[m, j] * F[j]
            term = max(term, float((dt * Q[m, j] * F[j]).abs().max()))
        want = max(want, float(r.abs().max()))
    assert abs(got - want) <= 16 * 2.0 ** -53 * 7 * term


def test_nan_in_a_node_is_reported(H):
    ctx = H.Context(H.make_config((31, 2, 3), None, dt=1 / 16))
    u = torch.rand(31, 31, 31, dtype=torch.float64, device="cuda")
    H.heat3d_set_state(ctx, 0, 0, 0.0, u)
    u[3, 4, 5] = float("nan")
    H.heat3d_set_node(ctx, 0, 0, 1, u)
    with pytest.raises(H.Heat3DError) as e:
        H.heat3d_sdc_residual(ctx, 0, 0)
    assert e.value.code == H.ENAN
