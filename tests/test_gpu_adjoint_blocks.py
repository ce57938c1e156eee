"""Blocks of adjoint sweeps (hp_project_adjoint) at the edges of their regions:
a region holds 64 x 64 cells, 48 x 48 of them its own after eight sweeps, and
a grid that it holds as a whole takes all sweeps in one block.  Against the
FP64 adjoint; bar: 1e-5 of the largest gradient entry, as for the other sizes
(a sweep averages, so that k sweeps of five FP32 roundings each stay below
5 k * 2^-24 of it: 7.5e-6 at k = 25)."""
import numpy as np
import pytest

import oracle
from oracle import adjoint as AD
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
    oracle.build()
    return torch.device("cuda:0")


@pytest.mark.parametrize("shape,k", [((1, 1, 1), 3), ((2, 64, 64), 17), ((1, 65, 64), 8),
                                     ((1, 64, 65), 9), ((2, 48, 97), 1), ((1, 145, 49), 16),
                                     ((1, 96, 193), 8), ((1, 7, 130), 25), ((1, 130, 3), 15)])
def test_blocks_match_oracle(dev, shape, k):
    B, ny, nx = shape
    rng = np.random.default_rng(ny * 1000 + nx + k)
    fl = np.zeros(shape, np.uint8)
    if min(ny, nx) > 8:
        fl = np.stack([W.random_obstacles(max(ny, nx), max(ny, nx), 5 + b, rect_side=(3, 20),
                                          disc_radius=(2, 9))[:ny, :nx] for b in range(B)])
    gu, gv, gp = (rng.standard_normal(s).astype(np.float32)
                  for s in ((B, ny, nx + 1), (B, ny + 1, nx), shape))
    d = [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in (gu, gv, gp, fl)]
    ctx = hp.Context(B, ny, nx)
    got = hp.hp_project_adjoint(ctx, *d, k)
    exp = AD.project_fixed_adjoint(*(a.astype(np.float64) for a in (gu, gv, gp)), fl, k)
    for g, e in zip(got, exp):
        assert np.abs(g.cpu().numpy() - e).max() <= 1e-5 * max(np.abs(e).max(), 1e-30)
