"""GPU test of the dense <-> pitched copies and of the spreading of one field to
all nodes, on both sides of the line (127) between one and eight planes a
thread: bitwise round trips."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N", [1, 3, 15, 63, 127, 255])
@pytest.mark.parametrize("items", [1, 3])
def test_round_trips_are_exact(N, items):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1307_7867_gb300 import build, heat3d as H
    build.build()
    M = 3
    ctx = H.Context(H.make_config((N, 2, M), None, batch=items, autotune=0))
    g = torch.Generator(device="cuda").manual_seed(N)
    u = [torch.rand(N, N, N, generator=g, dtype=torch.float64, device="cuda") for _ in range(items)]
    v = torch.rand(N, N, N, generator=g, dtype=torch.float64, device="cuda")
    for b in range(items):
        H.heat3d_set_state(ctx, 0, b, 0.0, u[b])
    H.heat3d_set_node(ctx, 0, items - 1, 1, v)
    out = torch.empty_like(v)
    for b in range(items):
        for m in range(M):
            out.fill_(-1.0)
            H.heat3d_get_node(ctx, 0, b, m, out)
            assert torch.equal(out, v if (b, m) == (items - 1, 1) else u[b])
