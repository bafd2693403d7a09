"""GPU tests of the fixed-point sums on values near the bottom of FP64's range:
operator, solve, sweep and collocation residual.

The operator is compared with a plain torch FP64 stencil: with W the sum of the
stencil's weights (12, 192, 48) and m the largest |u| of the five planes around,
24 roundings of W m cover both sides (19 operations of FP64; the fixed-point
sums are off by at most 1.3 W m 2^-53), and results below the normal range are
rounded to multiples of 2^-1074.

Solve, sweep and residual are linear without forcing, and a power of two scales
every FP64 number exactly: a run on scaled inputs must give the scaled result.
The two runs may take different routes (fixed point or FP64), so they differ by
their roundings: some 1e3 operations on numbers up to the condition number
(below 1e3 here) times the largest, 1e6 x 2^-53 = 1e-10 of it, and 2^-1074 at
each operation on values below the normal range, here amplified by less than
2^20 (nu dt / h^2 and the sums).
"""
import numpy as np
import pytest

from paper_1307_7867_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NU = 0.1


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1307_7867_gb300 import build, heat3d
    build.build()
    heat3d.load()
    return heat3d


def plain(u, order):
    """nu L u in torch FP64 with the boundary rule of the stencils."""
    n, h2 = u.shape[0], 1.0 / (u.shape[0] + 1) ** 2
    p = torch.zeros(n + 4, n + 4, n + 4, dtype=u.dtype, device=u.device)
    p[2:-2, 2:-2, 2:-2] = u
    if order == 4:
        for ax in range(3):
            q = p.movedim(ax, 0)
            q[0], q[-1] = -q[2].clone(), -q[-3].clone()

    def at(dz, dy, dx):
        return p[2 + dz:2 + dz + n, 2 + dy:2 + dy + n, 2 + dx:2 + dx + n]

    f = sum(at(*d) for d in ((1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)))
    c = at(0, 0, 0)
    if order == 2:
        return NU / h2 * (f - 6 * c)
    if order == 4:
        s = sum(at(*d) for d in ((2, 0, 0), (-2, 0, 0), (0, 2, 0), (0, -2, 0), (0, 0, 2), (0, 0, -2)))
        return NU / (12 * h2) * (16 * f - s - 90 * c)
    e = sum(at(a, b, 0) + at(a, 0, b) + at(0, a, b) for a in (1, -1) for b in (1, -1))
    return NU / (6 * h2) * (2 * f + e - 24 * c)


def weights(order, n):
    """nu times the sum of the stencil's weights."""
    return NU * (n + 1) ** 2 * {2: 12.0, 4: 192.0 / 12, 19: 48.0 / 6}[order]


def field(name, n):
    x = inputs.grid(n)
    if name == "gauss":  # a hot spot whose tail runs through the whole range of FP64
        g = np.exp(-(x - 0.4) ** 2 / (2 * 0.015 ** 2))
        return g[:, None, None] * g[None, :, None] * g[None, None, :]
    if name == "beside":  # a plane of 1e-290 and one of 1e-312 beside planes of order one
        u = inputs.random_field(n, 3)
        u[20] *= 1e-290
        u[40] *= 1e-312
        return u
    return float(name) * inputs.random_field(n, 4)


@pytest.mark.parametrize("order,n", [(2, 127), (4, 127), (19, 63), (19, 127)])
@pytest.mark.parametrize("name", ["1e-285", "1e-290", "1e-300", "1e-305", "1e-312", "gauss", "beside"])
def test_operator(H, order, n, name):
    ctx = H.Context(H.make_config((n, order, 2), None, nu=NU))
    u = torch.from_numpy(field(name, n)).cuda()
    out = torch.full_like(u, float("nan"))
    H.heat3d_apply_laplacian(ctx, 0, u, out)
    ref = plain(u, order)
    top = u.abs().amax(dim=(1, 2))
    near = torch.nn.functional.max_pool1d(top[None, None], 5, 1, 2)[0, 0]
    tol = weights(order, n) * (24 * 2.0 ** -53 * near + 24 * 2.0 ** -1074)
    assert bool(((out - ref).abs().amax(dim=(1, 2)) <= tol).all())


def close(a, b, scale):
    """a is `scale` times b up to the roundings named above."""
    top = float(b.abs().max())
    return float((a - b * scale).abs().max()) <= 1e-10 * top * scale + 2.0 ** -1054


@pytest.mark.parametrize("power", [-945, -963, -997])
@pytest.mark.parametrize("order,n", [(2, 127), (4, 127), (19, 63)])
def test_solve(H, order, n, power):
    ctx = H.Context(H.make_config((n, order, 2), None))
    rhs = torch.from_numpy(inputs.random_field(n, 9)).cuda()
    one, two = torch.zeros_like(rhs), torch.zeros_like(rhs)
    H.mg_vcycle(ctx, 0, 5e-4, rhs, one, 3, -1.0)
    H.mg_vcycle(ctx, 0, 5e-4, rhs * 2.0 ** power, two, 3, -1.0)
    assert float(one.abs().max()) > 0.01
    assert close(two, one, 2.0 ** power)


@pytest.mark.parametrize("power", [-945, -963, -997, -1014, -1030])
@pytest.mark.parametrize("order,n,M", [(2, 31, 3), (2, 31, 5), (4, 127, 3), (19, 63, 5)])
def test_sweep_and_residual(H, order, n, M, power):
    u = torch.from_numpy(inputs.smooth_random_field(n, 5)).cuda()
    res, node = [], []
    for s in (1.0, 2.0 ** power):
        ctx = H.Context(H.make_config((n, order, M), None, dt=1 / 32, nu=NU, forcing=H.FORCING_NONE, mg_tol=-1.0,
                                      max_cycles=3))
        H.heat3d_set_state(ctx, 0, 0, 0.0, u * s)
        H.sdc_sweep(ctx, 0, 0, 1)
        res.append(torch.tensor(H.heat3d_sdc_residual(ctx, 0, 0), dtype=torch.float64))
        node.append(torch.empty_like(u))
        H.heat3d_get_node(ctx, 0, 0, M - 1, node[-1])
    assert float(node[0].abs().max()) > 1e-3 and float(res[0]) > 1e-8
    assert close(node[1], node[0], 2.0 ** power)
    # the residual is a difference of numbers of the field's size
    assert abs(float(res[1]) - float(res[0]) * 2.0 ** power) <= \
        1e-10 * float(u.abs().max()) * 2.0 ** power + 2.0 ** -1054
