"""E of the grid-resident sweeps (hp_project's history) at its edges."""
import pytest

from test_gpu_resident_strips import dev  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
hp = pytest.importorskip("paper_2109_09363_gb300")


@pytest.mark.parametrize("shape", [(2, 128, 128), (1, 512, 512), (2, 200, 700)])
def test_an_overflowing_sum_is_infinite(dev, shape):  # noqa: F811
    """|div| of 2e38 in every cell of one grid: finite, but not its sum over a warp."""
    B, ny, nx = shape
    u = torch.zeros((B, ny, nx + 1), device=dev)
    v = torch.zeros((B, ny + 1, nx), device=dev)
    fl = torch.zeros(shape, dtype=torch.uint8, device=dev)
    u[B - 1] = 1e38 * (1 - 2 * (torch.arange(nx + 1, device=dev) % 2))
    ctx = hp.Context(*shape)
    for kw in (dict(threshold=1e-3, max_iters=50), dict(fixed_iters=5)):
        out = hp.hp_project(ctx, u.clone(), v.clone(), fl, hp.ProjectParams(**kw), hist_len=8)
        assert torch.isposinf(out["e_hist"][B - 1, 0])
        assert out["iters"][B - 1] == 0
