"""hp_resident_grids answers for the kernel that hp_project launches (a launch
of the resident kernel that is split over SMs is told apart by its waits, made
to run out), and both kernels against the FP64 oracle at 2048^2, where the
blocked one runs on request only."""
import numpy as np
import pytest

import oracle
from paper_2109_09363_gb300 import workloads as W
from test_gpu_resident_strips import case, dev  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
hp = pytest.importorskip("paper_2109_09363_gb300")


# (the counts tell 4, 8 or 16 rows a thread apart: an instance that the device
# does not run as it is meant to would show as another count)
@pytest.mark.parametrize("shape,grids", [((1, 128, 128), 38), ((70, 128, 128), 76),
                                         ((1, 256, 256), 19), ((38, 256, 256), 38),
                                         ((1, 512, 512), 4), ((16, 512, 512), 9), ((2, 100, 600), 25),
                                         ((1, 2048, 2048), 1), ((1, 2600, 2600), 0),
                                         ((1, 20000, 64), 0)])
def test_query_is_the_launch(dev, shape, grids):  # noqa: F811
    ctx = hp.Context(*shape)
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    got = hp.hp_resident_grids(ctx, *shape)
    assert got == grids if sms == 152 else (got > 0) == (grids > 0)
    u, v, fl = case(*shape, dev, kinds=1)
    ctx.set_wait_limit(1)
    out = hp.hp_project(ctx, u, v, fl, hp.ProjectParams(threshold=1e-4, max_iters=40))
    assert ((out["iters"] < 0) == (got > 0)).all()


@pytest.mark.parametrize("kernel", [0, 2])
def test_2048_against_oracle(dev, kernel):  # noqa: F811
    n, sweeps, tol = 2048, 40, 1e-5  # as for the other large grids
    u, v = W.vortex_velocity(n, n, 17)
    fl = W.random_obstacles(n, n, 18)[None]
    u, v = u[None].astype(np.float32), v[None].astype(np.float32)
    d = [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in (u, v, fl)]
    ctx = hp.Context(1, n, n)
    hp.hp_project(ctx, *d, hp.ProjectParams(fixed_iters=sweeps, sweep_kernel=kernel))
    ctx.check()
    oracle.build()
    oracle.set_threads(0)
    ref = oracle.project(u.astype(np.float64), v.astype(np.float64), fl, 0.0, 0,
                         fixed_iters=sweeps)
    umax = max(np.abs(ref["u"]).max(), np.abs(ref["v"]).max())
    assert np.abs(d[0].cpu().numpy() - ref["u"]).max() <= tol * umax
    assert np.abs(d[1].cpu().numpy() - ref["v"]).max() <= tol * umax
