"""The grid-resident sweep kernel against the blocked kernel where its split of
a grid can go wrong: one strip and many, a last strip of one row, rows of any
length in every width class, columns with copied cells (grids wider than 512),
more grids than fit at once, stops around a checkpoint, at and before the cap,
a guess without alignment, values so large that a fixed count has to watch E.
Both kernels use the same cell update in the same order: every bit must agree."""
import numpy as np
import pytest

from paper_2109_09363_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
hp = pytest.importorskip("paper_2109_09363_gb300")


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_09363_gb300 import build
    build.build()
    return torch.device("cuda:0")


def case(B, ny, nx, dev, kinds=3):
    us, vs, fs = [], [], []
    for b in range(B):
        if b < kinds:
            u, v = W.vortex_velocity(ny, nx, 40 + b, n_vortices=6, width=(2.0, 10.0))
            f = W.random_obstacles(ny, nx, 60 + b, rect_side=(3, 20), disc_radius=(2, 10))
        us.append(u), vs.append(v), fs.append(f)
    f32 = lambda a: torch.from_numpy(np.stack(a).astype(np.float32)).to(dev)  # noqa: E731
    return f32(us), f32(vs), torch.from_numpy(np.stack(fs)).to(dev)


def both(u, v, fl, phi0=None, **kw):
    out = []
    for kernel in (2, 0):
        ctx = hp.Context(*fl.shape)
        a, b = u.clone(), v.clone()
        o = hp.hp_project(ctx, a, b, fl, hp.ProjectParams(sweep_kernel=kernel, **kw), phi0=phi0)
        ctx.check()
        out.append(dict(o, u=a, v=b))
    for k in out[0]:
        x, y = out[0][k], out[1][k]
        same = (x == y) | ((x != x) & (y != y)) if x.is_floating_point() else x == y
        assert bool(same.all()), (k, kw)
    return out[1]


@pytest.mark.parametrize("shape", [
    (1, 1, 1), (2, 33, 128), (1, 129, 127), (200, 20, 100), (2, 257, 200), (1, 129, 256),
    (3, 65, 257), (1, 512, 512), (10, 200, 511), (1, 300, 513), (2, 129, 752), (1, 130, 2047)])
def test_strips_match_blocked_kernel(dev, shape):
    u, v, fl = case(*shape, dev)
    for kw in (dict(fixed_iters=1), dict(fixed_iters=41), dict(threshold=0.0, max_iters=0),
               dict(threshold=0.0, max_iters=63), dict(threshold=0.0, max_iters=97),
               dict(threshold=2e-3, max_iters=400),
               dict(threshold=2e-3, max_iters=400, open_top=1, inflow=(0, shape[2] // 2))):
        both(u, v, fl, **kw)


def test_guess_without_alignment_and_stops_around_checkpoints(dev):
    shape = (2, 96, 300)
    u, v, fl = case(*shape, dev)
    n = int(np.prod(shape))
    phi0 = (0.05 * torch.randn(n + 1, generator=torch.Generator().manual_seed(1))).to(dev)[1:]
    phi0 = phi0.view(shape)
    assert phi0.data_ptr() % 16 != 0
    ctx = hp.Context(*shape)
    hist = hp.hp_project(ctx, u.clone(), v.clone(), fl, hp.ProjectParams(0.0, 300), phi0=phi0,
                         hist_len=301)["e_hist"][0].cpu().numpy()
    for k in (0, 1, 31, 32, 33, 63, 64, 255, 256, 257):
        # between E_{k-1} and E_k (the first falls monotonically from a rough guess)
        thr = float(hist[k]) * 1.000001
        out = both(u, v, fl, phi0=phi0, threshold=thr, max_iters=300)
        assert out["iters"][0] <= k


def test_fixed_count_stops_a_grid_that_is_not_finite(dev):
    u, v, fl = case(3, 96, 96, dev)
    u[1, 40, 40] = float("inf")
    fl[1, 40, 38:43] = 0
    out = both(u, v, fl, fixed_iters=20)
    assert out["iters"].tolist() == [20, 0, 20]
