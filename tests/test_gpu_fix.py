"""GPU tests of the fixed-point FP64 stencils (csrc/stencil_fix.cuh), the
kernel of every FP64 stencil on grids with N >= 127: against a plain torch
FP64 stencil on the fields where the format can go wrong (single points at
tile edges, planes of very different size, zeros, values that only FP64 takes,
Inf and NaN), and batches against single items bit for bit.

Tolerance of the first: both sides round.  FP64 sums of the stencil are off by
at most about 13 roundings of the largest partial sum (weights' sum 192 times
the largest neighbour); the fixed-point sums by a few units of 2^-58 of the
largest value of the planes involved times 16.  With m the largest |u| of the
five planes around, 200 x 16 x 2^-53 m covers both by a factor of two.
"""
import numpy as np
import pytest

from paper_1307_7867_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

N = 127
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


def field(name):
    rng = np.random.default_rng(11)
    if name == "points":  # single points at corners and around tile edges
        u = np.zeros((N, N, N))
        for k in (0, 1, 5, 63, N - 2, N - 1):
            for j in (0, 1, 15, 16, 31, 63, N - 2, N - 1):
                for i in (0, 1, 62, 63, 64, 65, N - 2, N - 1):
                    u[k, j, i] = rng.standard_normal()
        return u
    if name == "planes":  # the planes' sizes differ by up to 2^60
        return inputs.random_field(N, 3) * (2.0 ** rng.integers(-60, 1, N))[:, None, None]
    if name == "zeros":
        u = inputs.random_field(N, 4)
        u[:, :64, :] = 0.0
        u[40:60] = 0.0
        return u
    if name == "huge":
        return 1e200 * inputs.random_field(N, 5)
    if name == "tiny":
        u = 1e-200 * inputs.random_field(N, 5)
        u[64:] *= 1e180  # next to values that the format takes
        return u
    assert name == "random"
    return inputs.random_field(N, 6)


@pytest.mark.parametrize("order", [2, 4, 19])
@pytest.mark.parametrize("name", ["random", "points", "planes", "zeros", "huge", "tiny"])
def test_operator_matches_plain_fp64(H, order, name):
    ctx = H.Context(H.make_config((N, order, 2), None, nu=NU))
    u = torch.from_numpy(field(name)).cuda()
    out = torch.full_like(u, float("nan"))
    H.heat3d_apply_laplacian(ctx, 0, u, out)
    ref = plain(u, order)
    top = u.abs().amax(dim=(1, 2))
    near = torch.nn.functional.max_pool1d(top[None, None], 5, 1, 2)[0, 0]
    scale = NU * (N + 1) ** 2 / {2: 1, 4: 12, 19: 6}[order]
    tol = scale * 200 * 16 * 2.0 ** -53 * near
    assert bool(((out - ref).abs().amax(dim=(1, 2)) <= tol).all())
    if name in ("points", "zeros"):  # exact zeros stay exact zeros
        assert bool((out[ref == 0] == 0).all())


@pytest.mark.parametrize("order", [2, 4, 19])
def test_inf_and_nan_reach_the_same_points(H, order):
    ctx = H.Context(H.make_config((N, order, 2), None, nu=NU))
    u = torch.from_numpy(inputs.random_field(N, 8)).cuda()
    u[20, 30, 64] = float("inf")
    u[90, 127 // 2, 3] = float("nan")
    u[N - 1, 0, 0] = float("-inf")
    out = torch.empty_like(u)
    H.heat3d_apply_laplacian(ctx, 0, u, out)
    ref = plain(u, order)
    assert torch.equal(torch.isnan(out), torch.isnan(ref))
    assert torch.equal(torch.isinf(out), torch.isinf(ref))
    assert torch.equal(out[torch.isinf(ref)], ref[torch.isinf(ref)])


@pytest.mark.parametrize("order", [4, 19])
def test_items_of_a_batch_equal_single_items(H, order):
    """A block's run of planes may end one tile or item and begin the next."""
    items, M = 5, 3
    big = H.Context(H.make_config((N, order, M), None, dt=1 / 32, batch=items))
    one = H.Context(H.make_config((N, order, M), None, dt=1 / 32))
    u = [torch.from_numpy(inputs.smooth_random_field(N, 20 + b)).cuda() for b in range(items)]
    for b in range(items):
        H.heat3d_set_state(big, 0, b, 0.1 * b, u[b])
    H.sdc_sweep(big, 0, 0, items)
    a, c = torch.empty_like(u[0]), torch.empty_like(u[0])
    for b in range(items):
        H.heat3d_set_state(one, 0, 0, 0.1 * b, u[b])
        H.sdc_sweep(one, 0, 0, 1)
        H.heat3d_get_node(big, 0, b, M - 1, a)
        H.heat3d_get_node(one, 0, 0, M - 1, c)
        assert torch.equal(a, c)


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("c", [0.0, 1e-70])
def test_solve_with_coefficients_beyond_the_format(H, order, c):
    """c = 0 (zero coefficients) and a c whose coefficients FP64 alone takes."""
    ctx = H.Context(H.make_config((N, order, 2), None))
    rhs = torch.from_numpy(inputs.random_field(N, 9)).cuda()
    u = torch.zeros_like(rhs)
    H.mg_vcycle(ctx, 0, c, rhs, u, 50, 1e-12)
    assert float((u - rhs).abs().max()) <= 1e-12
