"""E of the grid-resident sweeps (hp_project's history) at its edges."""
import pytest

from test_gpu_resident_strips import dev  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
hp = pytest.importorskip("paper_2109_09363_gb300")


@pytest.mark.parametrize("shape", [(19, 512, 512), (3, 1024, 1024), (1, 2048, 2048)])
def test_chains_of_additions_are_short(dev, shape):  # noqa: F811
    """E_0 = mean |div| of a 1 in row 0 and of t = 0.95 * 2^-24 everywhere else:
    every t added to a sum that holds the 1 by itself is lost.  In chains of
    eight values, then sums of these in pairs over at most 1,024 cells (eight
    additions that the 1 goes through, each rounding by 2^-24 at most), the
    error stays below 7 t + 8 * 2^-24 = 8.8e-7; a chain of 32 values loses 31 t =
    1.76e-6 by itself.  Bar 1e-6 of E >= 1 / cells."""
    div = torch.full(shape, 0.95 * 2.0 ** -24, device=dev)
    div[:, 0, 5] = 1.0
    fl = torch.zeros(shape, dtype=torch.uint8, device=dev)
    ctx = hp.Context(*shape)
    _, e = hp.hp_jacobi_sweeps(ctx, torch.zeros(shape, device=dev), div, fl, 2, with_e=True)
    ref = div.double().mean(dim=(1, 2))
    assert (((e[:, 0] - ref) * shape[1] * shape[2]).abs() <= 1e-6).all()


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
