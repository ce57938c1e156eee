"""Stops of the grid-resident sweeps at the edges of their decisions and
checkpoints: the rounds that are waited for and the first that is not, the
sweeps next to a checkpoint, replays of none and of all sweeps since one; one
CTA per grid and several, one wave of grids and two, strips with columns, a cap
between two checkpoints.  Against the blocked kernel, every bit."""
import pytest

from test_gpu_resident_strips import both, case, dev  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
hp = pytest.importorskip("paper_2109_09363_gb300")


@pytest.mark.parametrize("shape", [(1, 128, 128), (200, 64, 128), (64, 256, 256), (10, 600, 600),
                                   (4, 1024, 1024)])
def test_stops_match_blocked_kernel(dev, shape):  # noqa: F811
    u, v, fl = case(*shape, dev)
    ctx = hp.Context(*shape)
    hist = hp.hp_project(ctx, u.clone(), v.clone(), fl,
                         hp.ProjectParams(0.0, 300, sweep_kernel=2), hist_len=301)["e_hist"]
    e = hist.max(dim=0).values.cpu().tolist()
    for k in (1, 3, 4, 7, 8, 11, 12, 15, 16, 17, 31, 32, 48, 63, 64, 65, 97, 255, 256, 257):
        both(u, v, fl, threshold=0.5 * (e[k - 1] + e[k]), max_iters=300)
    for cap in (15, 16, 17, 33, 64):
        both(u, v, fl, threshold=0.0, max_iters=cap)
