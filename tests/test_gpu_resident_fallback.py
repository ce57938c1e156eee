"""What the grid-resident sweeps cannot serve goes to the blocked kernel instead
of failing: a context limited to fewer SMs than a shape needs.  With just as many
as its tallest strips need (128 and 256 rows of strips of 16 rows a thread, eight
of them at 512 columns, 40 at 1024^2) the shape is resident, which also checks
that every one of those instances has the registers its split assumes."""
import pytest

from test_gpu_resident_strips import case, dev  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
hp = pytest.importorskip("paper_2109_09363_gb300")


@pytest.mark.parametrize("shape,sms", [((2, 128, 128), 1), ((2, 256, 256), 2), ((2, 512, 512), 8),
                                       ((2, 1024, 1024), 40)])
def test_shapes_that_do_not_fit(dev, shape, sms):  # noqa: F811
    u, v, fl = case(*shape, dev)
    ctx = hp.Context(*shape)
    prm = dict(threshold=1e-3, max_iters=60)

    def project(**kw):
        a, b = u.clone(), v.clone()
        o = hp.hp_project(ctx, a, b, fl, hp.ProjectParams(**prm, **kw))
        ctx.check()
        return dict(o, u=a, v=b)

    ref = project(sweep_kernel=2)
    for limit, grids in ((sms, 1), (sms - 1, 0) if sms > 1 else (sms, 1), (2 * sms, None), (0, None)):
        ctx.set_resident_sms(limit)
        got = hp.hp_resident_grids(ctx, *shape)
        assert got > 0 if grids is None else got == grids
        for kernel in (0, 4):
            out = project(sweep_kernel=kernel)
            for k in ref:
                assert torch.equal(ref[k], out[k]), (limit, k)
